"""Pairs of the batched plan that run on the plan's own streams: against the
task engine and the oracle, bitwise repeatable, in a CUDA graph, mixed with
pairs that stay in the engine, with the status of a non-finite input, and two
plans from two threads at once.

Tolerance: the FP64 parity bar of the suite (relative 1e-12)."""
import json
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import hatt as ohatt
from oracle import tt as ott
from paper_2410_04385_gb300 import workloads as wl

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def pairs(big, small, precision=0):
    """`big` pairs above the engine's size (ragged ranks, odd modes), `small` tiny ones between them."""
    rng = np.random.default_rng(17)
    out = []
    for j in range(max(big, small)):
        for d, n, lo, hi, on in ((5, 21, 9, 22, j < big), (4, 7, 2, 5, j < small)):
            if on:
                ry = [1] + [int(v) for v in rng.integers(lo, hi, size=d - 1)] + [1]
                rz = [1] + [int(v) for v in rng.integers(lo, hi, size=d - 1)] + [1]
                ell = 2 * max(max(ry), max(rz))
                out.append((wl.gaussian_tt([n] * d, ry, int(rng.integers(1 << 30))),
                            wl.gaussian_tt([n] * d, rz, int(rng.integers(1 << 30))),
                            dict(sketch_rank=ell, max_rank=ell, oversample=0, seed=40 + j, precision=precision)))
    return out


def gpu(ps):
    return [([torch.from_numpy(c).cuda() for c in Y], [torch.from_numpy(c).cuda() for c in Z], o) for Y, Z, o in ps]


def host(eng):
    torch.cuda.synchronize()
    return [[c.cpu().numpy().copy() for c in eng.result(j)] for j in range(eng.count)]


def worst(X, ps):
    w = 0.0
    for x, (Y, Z, o) in zip(X, ps):
        Xo = ohatt.hadamard_recompress(Y, Z, **{k: v for k, v in o.items() if k != "precision"})
        w = max(w, ott.tt_diff_norm(x, Xo) / ott.tt_norm(Xo))
    return w


@pytest.fixture(scope="module")
def B():
    from paper_2410_04385_gb300 import binding, build
    if not os.path.exists(binding.LIB_PATH):
        build.build()
    binding.load()
    return binding


@pytest.mark.parametrize("big, small", [(1, 0), (3, 0), (2, 3), (18, 0)])
def test_streams_match_the_oracle_and_repeat(B, big, small):
    ps = pairs(big, small)
    eng = B.BatchedRecompressor(gpu(ps))
    assert (eng.info()["stages"] > 0) == (small > 0)     # the tiny ones alone stay in the engine
    eng.run()
    first = host(eng)
    assert eng.status() == 0 and worst(first, ps) <= 1e-12
    eng.run()
    assert all(np.array_equal(a, b) for x, y in zip(first, host(eng)) for a, b in zip(x, y))
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    for bufs in eng.out_bufs:
        for c in bufs:
            c.zero_()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        eng.run(stream=s)
    g.replay()
    assert all(np.array_equal(a, b) for x, y in zip(first, host(eng)) for a, b in zip(x, y))


def test_fp32_sketches_within_the_mixed_bound(B):
    ps = pairs(3, 0, precision=B.TT_MIXED_FP32)
    eng = B.BatchedRecompressor(gpu(ps))
    eng.run()
    for x, (Y, Z, o) in zip(host(eng), ps):
        o = {k: v for k, v in o.items() if k != "precision"}
        X64 = ohatt.hadamard_recompress(Y, Z, **o)
        X32 = ohatt.hadamard_recompress(Y, Z, fmt="fp32", **o)
        A = ott.hadamard_pkp(Y, Z)
        bound = 10 * max(ott.tt_rel_error(X64, A), ott.tt_rel_error(X32, A), 1e-12)
        assert ott.tt_rel_error(x, A) <= bound


def test_every_pair_either_way():
    script = ("import json, sys; sys.path.insert(0, %r)\n"
              "from tests import test_gpu_batched_streams as T\nfrom paper_2410_04385_gb300 import binding as B\n"
              "ps = T.pairs(3, 3); eng = B.BatchedRecompressor(T.gpu(ps)); eng.run(); X = T.host(eng)\n"
              "print(json.dumps([T.worst(X, ps), eng.status(), eng.info()['stages']]))" % ROOT)
    for form in ("engine", "lanes"):
        p = subprocess.run([sys.executable, "-c", script], capture_output=True, text=True, timeout=600, cwd=ROOT,
                           env=dict(os.environ, HATT_BATCH_FORM=form))
        assert p.returncode == 0, p.stderr[-2000:]
        rel, status, stages = json.loads(p.stdout.strip().splitlines()[-1])
        assert rel <= 1e-12 and status == 0 and (stages > 0) == (form == "engine")


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_input_sets_the_plan_status(B, bad):
    ps = pairs(2, 0)
    ps[1][0][2][0, 3, 1] = bad
    eng = B.BatchedRecompressor(gpu(ps))
    eng.run()
    X = host(eng)
    assert eng.status() == B.TT_ERR_NONFINITE
    assert B.device_status() == B.TT_OK                  # the plan's own word, as for the engine's pairs
    assert worst(X[:1], ps[:1]) <= 1e-12


def test_two_plans_from_two_threads(B):
    sets = [pairs(2, 0), pairs(3, 1)]
    engs = [B.BatchedRecompressor(gpu(ps)) for ps in sets]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in engs]

    def work(i):
        for _ in range(5):
            engs[i].run(stream=streams[i])

    ts = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for eng, ps in zip(engs, sets):
        assert worst(host(eng), ps) <= 1e-12 and eng.status() == 0
