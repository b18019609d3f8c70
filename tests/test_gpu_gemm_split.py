"""FP64 products on the tensor cores from exact digits (k_gemm_split.cu),
through tt_gemm, at the sizes where tiles (128 x 32), K chunks (32) and K
splits end, against exact products.

Bounds, derived before the first run. Digits keep each entry to 2^-62 of its
row's (column's) largest after the scaling, dropped digit products weigh less
than 8 2^-64 per term, and each chunk's sum and each addition over chunks
rounds by 2^-53 of a value below |A||B| in the Gaussian cases: the error of
an element is below gamma_K (|A| |B|) with u = 2^-53 (the bound of an FP64
chain), K >= 4. With |a|, |b| <= 1 and every digit at its extreme the sum of
each chunk is one correctly rounded FP64 number, so equal entries give
K x y to (chunks + 1) roundings."""
import json
import os
import subprocess
import sys
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def B():
    from paper_2410_04385_gb300 import binding, build
    if not os.path.exists(binding.LIB_PATH):
        build.build()
    binding.load()
    return binding


def product(B, A, Bm, alpha=1.0):
    C = B.gemm(torch.from_numpy(A).cuda(), torch.from_numpy(Bm).cuda(), alpha=alpha)
    torch.cuda.synchronize()
    assert B.device_error() == 0
    return C.cpu().numpy()


@pytest.mark.parametrize("nb, M, N, K", [
    (40, 127, 31, 33), (40, 128, 32, 32), (30, 129, 33, 31), (300, 20, 20, 50), (7, 1, 4099, 150),
    (7, 4099, 1, 150), (1, 97, 65, 4099), (2, 1025, 50, 63), (900, 5, 257, 4), (3, 300, 90, 96)])
@pytest.mark.parametrize("grade", [0.0, 6.0])
def test_product_within_the_fp64_bound(B, nb, M, N, K, grade):
    rng = np.random.default_rng(M + 3 * N + 7 * K)
    A = rng.standard_normal((nb, M, K)) * np.exp(rng.uniform(-20, 20, (nb, M, 1)))
    Bm = rng.standard_normal((nb, K, N)) * np.exp(rng.uniform(-20, 20, (nb, 1, N)))
    D = np.exp(rng.uniform(-grade, grade, (nb, 1, K)))       # a gauge of the inner index
    A, Bm = A * D, Bm / np.swapaxes(D, 1, 2)
    C = product(B, A, Bm, alpha=0.75)
    ref = 0.75 * np.matmul(A.astype(np.longdouble), Bm.astype(np.longdouble)) if M * N * K * nb < 3e7 \
        else 0.75 * (A @ Bm)
    scale = 0.75 * (np.abs(A) @ np.abs(Bm))
    u = 2.0 ** -53
    assert np.all(np.abs(C - ref) <= 2 * K * u / (1 - K * u) * scale)


def test_inner_scaling_by_powers_of_two_changes_nothing(B):
    rng = np.random.default_rng(5)
    A, Bm = rng.standard_normal((4, 300, 90)), rng.standard_normal((4, 90, 70))
    p = 2.0 ** (2 * rng.integers(-200, 200, (4, 1, 90)))
    assert np.array_equal(product(B, A, Bm), product(B, A * p, Bm / np.swapaxes(p, 1, 2)))


# significands whose digits are all +127, all near -128, and 0x55 / 0xAA patterns
@pytest.mark.parametrize("m", [0x1FBFBFBFBFBFBF, 0x1FC04040404040, 0x15555555555555, 0x1AAAAAAAAAAAAA])
@pytest.mark.parametrize("sign", [1, -1])
def test_extreme_digits_sum_exactly(B, m, sign):
    K, M, N = 512, 130, 70
    x = float(m) * 2.0 ** -53
    y = sign * x
    C = product(B, np.full((1, M, K), x), np.full((1, K, N), y))
    want = K * Fraction(x) * Fraction(y)
    chunks = -(-K // 32)
    assert all(abs(Fraction(float(v)) - want) <= (chunks + 1) * abs(want) / 2 ** 53 for v in np.unique(C))


def test_range_ends_and_nonfinite_entries(B):
    rng = np.random.default_rng(9)
    A, Bm = rng.standard_normal((200, 64)), rng.standard_normal((64, 400))
    A[0] *= 1e-310                                           # subnormal rows
    A[1] = 0.0
    A[2] *= 1e300
    Bm[:, 0] *= 1e-300
    Bm[:, 1] *= 1e30
    C = product(B, A, Bm)
    with np.errstate(over="ignore", invalid="ignore"):
        ref, scale = A @ Bm, np.abs(A) @ np.abs(Bm)
    fine = np.isfinite(scale)
    assert np.all(np.abs(C - ref)[fine] <= 1e-13 * scale[fine] + 64 * 5e-324)
    assert np.all(C[1] == 0.0)
    assert np.all(~np.isfinite(C[2, 1]) | (np.abs(ref[2, 1]) < np.inf))
    A2, B2 = A.copy(), Bm.copy()
    A2[7, 3], A2[8, 60], B2[5, 9] = np.nan, np.inf, -np.inf
    C2 = product(B, A2, B2)
    bad = np.zeros(C2.shape, bool)
    bad[7] = bad[8] = True
    bad[:, 9] = True
    assert not np.isfinite(C2[bad]).any()
    ok = ~bad & fine
    assert np.all(np.abs(C2 - ref)[ok] <= 1e-13 * scale[ok] + 64 * 5e-324)


def test_workloads_with_every_product_on_the_dfma_kernel():
    """The other side of the dispatch, on the same workloads as the default's check in
    test_gpu_gemm_forms.py, within the same parity bar of the oracle."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, os.path.join(root, "tests", "gemm_forms_check.py")], capture_output=True,
                       text=True, env=dict(os.environ, HATT_GEMM_FORM="dfma"), timeout=900, cwd=root)
    assert p.returncode == 0, p.stderr[-3000:]
    r = json.loads(p.stdout.strip().splitlines()[-1])
    assert r["d20_ranks_equal"] and r["trunc_ranks_equal"] and r["round_ranks_equal"]
    assert max(r["d20_rel"], r["trunc_rel"], r["round_rel_to_input"], r["uneven_rel_max"]) <= 1e-12
    assert r["device_error"] == 0
