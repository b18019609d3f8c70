"""Rounding a sum returns the cores it has always returned, signs included.

The weighted sum of four rank-24 tensors on a 64^8 grid, rounded to rank 24: from the third
bond on the discarded energies lie below FP32, and the signs of the kept directions follow the
last bits of every product, QR and refinement before them. round_cores_d8.npz holds samples
(mode index 5, the first four right indices) of the cores that the DFMA products, the
one-column QR and the one-chain refinement give, recorded with untimed tilings. Two of its four
inputs come with negated directions in cores 1 and 2 when any of these sums runs in another
order, a relative difference of 0.36 and more. Runs in a process of its own (a shape's tiling
is fixed for the life of a process).

Bound: 1e-9, far above what the bits can differ by (these are the same operations) and far
below a sign."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SEEDS = (2, 4, 9, 30)


def terms(seed, d=8, n=64, r=24):
    rng = np.random.RandomState(seed)
    ranks = [1] + [r] * (d - 1) + [1]
    return [[(2.0 * rng.random_sample((ranks[k], n, ranks[k + 1])) - 1.0) * np.sqrt(3.0 / (n * ranks[k + 1]))
             for k in range(d)] for _ in range(4)]


def main():
    from paper_2410_04385_gb300 import binding
    binding.load()
    binding.gemm_autotune(False)
    gold = np.load(os.path.join(ROOT, "tests", "golden", "round_cores_d8.npz"))
    worst = {}
    for seed in SEEDS:
        w = binding.tt_lincomb([[torch.from_numpy(c).cuda() for c in t] for t in terms(seed)],
                               [1.0, 0.03, -0.02, 0.01])
        rnd = binding.Rounder(w, max_rank=24, tol=1e-8, fixed_ranks=1)
        rnd.run()
        for form in ("eager", "graph"):
            if form == "graph":
                g = torch.cuda.CUDAGraph()
                for c in rnd.result():
                    c.zero_()
                torch.cuda.synchronize()
                s = torch.cuda.Stream()
                with torch.cuda.graph(g, stream=s):
                    rnd.run(stream=s)
                g.replay()
            torch.cuda.synchronize()
            rel = []
            for k, core in enumerate(rnd.result()):
                want = gold["%d/%d" % (seed, k)]
                got = core[:, 5, :want.shape[1]].cpu().numpy()
                rel.append(float(np.linalg.norm(got - want) / np.linalg.norm(want)))
            worst["%s %d" % (form, seed)] = max(rel)
    print(json.dumps(worst))


def test_cores_are_the_recorded_ones():
    from paper_2410_04385_gb300 import binding, build
    if not os.path.exists(binding.LIB_PATH):
        build.build()
    p = subprocess.run([sys.executable, "-m", "tests.test_gpu_round_signs"], capture_output=True, text=True,
                       timeout=600, cwd=ROOT)
    assert p.returncode == 0, p.stderr[-3000:]
    worst = json.loads(p.stdout.strip().splitlines()[-1])
    assert len(worst) == 2 * len(SEEDS) and max(worst.values()) <= 1e-9, worst


if __name__ == "__main__":
    main()
