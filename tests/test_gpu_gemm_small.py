"""Small FP64 products (k_gemm_small.cu) where tiles, the threads' K groups and
the four sums of a thread end, with every stride the recompression uses.

Bound: an element's error is at most gamma_K (|A| |B|) for any order of the K
multiply-adds; alpha and beta add three roundings."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import hatt as ohatt
from oracle import tt as ott
from paper_2410_04385_gb300 import workloads as wl

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def B():
    from paper_2410_04385_gb300 import binding, build
    if not os.path.exists(binding.LIB_PATH):
        build.build()
    binding.load()
    return binding


@pytest.mark.parametrize("nb, M, N, K", [
    (1, 1, 1, 1), (1, 1, 1, 6000), (3, 1, 257, 3), (2, 257, 1, 4), (1, 5, 5, 50), (50, 50, 5, 50), (1, 7, 11, 13),
    (65535, 1, 1, 2), (1, 16, 16, 15), (1, 17, 16, 64), (1, 33, 31, 65), (5, 100, 3, 255), (1, 2, 3000, 127),
    (1, 3000, 2, 128), (1, 34, 34, 2176), (9, 60, 60, 61), (1, 1000, 1000, 1), (1, 300, 310, 32)])
@pytest.mark.parametrize("alpha", [1.0, -0.375])
def test_product_within_the_fp64_bound(B, nb, M, N, K, alpha):
    rng = np.random.default_rng(M + 3 * N + 7 * K)
    A = rng.standard_normal((nb, M, K))
    Bm = rng.standard_normal((nb, K, N))
    C = B.gemm(torch.from_numpy(A).cuda(), torch.from_numpy(Bm).cuda(), alpha=alpha).cpu().numpy()
    ref = alpha * np.matmul(A.astype(np.longdouble), Bm.astype(np.longdouble))
    u = 2.0 ** -53
    bound = (K + 3) * u / (1 - (K + 3) * u) * abs(alpha) * (np.abs(A) @ np.abs(Bm))
    assert np.all(np.abs(C - ref) <= bound)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_entries_stay_in_their_row(B, bad):
    A, Bm = np.ones((1, 9, 21)), np.ones((1, 21, 10))
    A[0, 4, 20] = bad
    C = B.gemm(torch.from_numpy(A).cuda(), torch.from_numpy(Bm).cuda()).cpu().numpy()
    assert not np.isfinite(C[0, 4]).any() and np.all(np.delete(C[0], 4, 0) == 21.0)


@pytest.mark.parametrize("n, ry, rz, ell", [(3, 2, 3, 4), (7, 4, 5, 9), (8, 5, 2, 12), (10, 9, 3, 5)])
@pytest.mark.parametrize("variant", [1, 2])
def test_strided_contractions_match_the_oracle(B, n, ry, rz, ell, variant):
    Y = wl.gaussian_tt([n] * 5, [1] + [ry] * 4 + [1], 5)
    Z = wl.gaussian_tt([n] * 5, [1] + [rz] * 4 + [1], 6)
    opts = dict(sketch_rank=ell, seed=3, variant=variant, ep=1e-12 if variant == 2 else 0.0)
    X = B.tt_hadamard_recompress([torch.from_numpy(x).cuda() for x in Y], [torch.from_numpy(x).cuda() for x in Z],
                                 **opts)
    X = [x.cpu().numpy() for x in X]
    Xo = ohatt.hadamard_recompress(Y, Z, sketch_rank=ell, seed=3)
    A = ott.hadamard_pkp(Y, Z)
    assert ott.tt_rel_error(X, A) <= ott.tt_rel_error(Xo, A) + 1e-12
