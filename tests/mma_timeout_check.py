"""Subprocess body of tests/test_gpu_batched_status.py: with HATT_MMA_WAITS=0 every wait for
tensor-core products gives up at once (the products themselves end: the kernels wait for them
before they leave). Runs batched plans whose pairs are all on streams, in FP64 and with FP32
sketch products, then recompressions in FP64 and TF32, and reads the statuses; then a small pair,
which has no such products, against the oracle: the context stays usable. Prints one JSON line."""
import json
import os
import sys

import numpy as np
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
from oracle import hatt as ohatt  # noqa: E402
from oracle import tt as ott  # noqa: E402
from paper_2410_04385_gb300 import binding as B  # noqa: E402
from paper_2410_04385_gb300 import workloads as wl  # noqa: E402


def gpu(cores):
    return [torch.from_numpy(np.ascontiguousarray(c)).cuda() for c in cores]


def pair(n, r, d, precision):
    ranks = [1] + [r] * (d - 1) + [1]
    return (gpu(wl.gaussian_tt([n] * d, ranks, 3)), gpu(wl.gaussian_tt([n] * d, ranks, 4)),
            dict(sketch_rank=2 * r, max_rank=2 * r, oversample=0, seed=5, precision=precision))


def main():
    B.load()
    out = {}
    B.device_status()                                 # clear
    for name, precision in (("fp64", B.TT_FP64), ("fp32", B.TT_MIXED_FP32)):
        for d in (3, 5):
            eng = B.BatchedRecompressor([pair(32, 30, d, precision), pair(24, 26, d, precision)], autotune=False)
            for rep in ("first", "again"):
                eng.run()
                out["%s d%d %s" % (name, d, rep)] = eng.status()
    out["device_after_batches"] = B.device_status()
    for name, precision in (("fp64", B.TT_FP64), ("tf32", B.TT_MIXED_TF32)):
        Y, Z, o = pair(32, 30, 5, precision)
        h = B.HadamardRecompressor(Y, Z, sketch_rank=60, seed=2, precision=precision)
        h.run()
        torch.cuda.synchronize()
        out["device_after_" + name] = B.device_status()
    y, z = wl.gaussian_tt([6] * 4, [1, 3, 3, 3, 1], 7), wl.gaussian_tt([6] * 4, [1, 2, 3, 2, 1], 8)
    h = B.HadamardRecompressor(gpu(y), gpu(z), sketch_rank=9, seed=2)
    h.run()
    torch.cuda.synchronize()
    x = [c.cpu().numpy() for c in h.result()]
    a = ohatt.hadamard_recompress(y, z, sketch_rank=9, seed=2)
    out["small_rel"] = ott.tt_diff_norm(x, a) / ott.tt_norm(a)
    out["device_after_small"] = B.device_status()
    print(json.dumps(out))


if __name__ == "__main__":
    main()
