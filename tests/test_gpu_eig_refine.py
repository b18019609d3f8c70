"""Rank cuts at the sizes where the eigenvector refinement changes form (one block
per column from 8 to 96, K groups of 8 down to 2), single call (whole GPU) and
stream lanes (cluster), against the oracle.

The kept subspace of a bond is resolved to about c u s1^2 / (s_r^2 - s_{r+1}^2)
against an SVD; Gaussian pairs of these sizes have s1^2 / gap below 1e4, c <= 128,
two truncated bonds: 2 x 128 x 1.1e-16 x 1e4 < 3e-10."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import hatt as ohatt
from oracle import tt as ott
from paper_2410_04385_gb300 import workloads as wl

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("c", [2, 7, 8, 9, 16, 31, 32, 33, 42, 51, 64, 65, 85, 86, 95, 96, 97])
def test_rank_cut_matches_the_oracle(c):
    from paper_2410_04385_gb300 import binding, build
    if not os.path.exists(binding.LIB_PATH):
        build.build()
    r = max(2, int(np.ceil(np.sqrt(c))) + 1)
    n = [max(4, c), 5, max(4, c)]
    Y = wl.gaussian_tt(n, [1, r, r, 1], 70 + c)
    Z = wl.gaussian_tt(n, [1, r, r, 1], 71 + c)
    opts = dict(sketch_rank=c, max_rank=max(1, (3 * c) // 4), seed=c)
    Yg, Zg = [torch.from_numpy(x).cuda() for x in Y], [torch.from_numpy(x).cuda() for x in Z]
    Xo = ohatt.hadamard_recompress(Y, Z, **opts)
    lanes = binding.BatchRecompressor([(Yg, Zg, opts)], lanes=1)
    lanes.run()
    single = binding.tt_hadamard_recompress(Yg, Zg, **opts)
    assert all(torch.equal(a, b) for a, b in zip(single, lanes.result(0)))   # both forms, bit for bit
    for X in (single, lanes.result(0)):
        X = [x.cpu().numpy() for x in X]
        assert ott.ranks(X) == ott.ranks(Xo)
        assert ott.tt_diff_norm(X, Xo) <= 3e-10 * ott.tt_norm(Xo)
    assert binding.device_error() == 0
