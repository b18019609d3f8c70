"""FP64 products whose large entries meet zeros or small entries of the other operand: an output
there is a sum of terms far below its row's and its column's largest, which the digits of
k_gemm_split.cu alone do not hold.

Bound, derived before the first run: that of an FP64 chain for every element, gamma_K (|A| |B|)
with u = 2^-53, doubled for alpha and the reference, as in test_gpu_gemm_split.py. An output
either has a term of at least 2^-6.2 of the product of its scales, where 36 digit products leave at
most 2^-59.2 of that product per term, or is summed in FP64.

The difference of a tensor and its own left-orthogonal form is zero; every step on it rounds by
u per term of at most 1600, over 20 cores: 1e-12 of the tensor's norm."""
import os

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


def blocks(rng, nb, M, N, K, p):
    """Rows [R, 2^-p S] against the block diagonal of two factors, the border between the blocks
    off every multiple of 32."""
    kb, jb = K // 2 + 5, N // 2 + 1
    A, Bm = rng.standard_normal((nb, M, K)), rng.standard_normal((nb, K, N))
    A[:, :, kb:] *= 2.0 ** -p
    Bm[:, :kb, jb:] = 0.0
    Bm[:, kb:, :jb] = 0.0
    return A, Bm


def alternating(rng, nb, M, N, K, p):
    """Rows alternating (1, e, 1, e, ..) and (e, 1, ..) against columns (e, 1, ..) and (1, e, ..)."""
    e = 2.0 ** -p
    i, k, j = np.arange(M)[:, None], np.arange(K), np.arange(N)
    A = np.where((i + k) % 2 == 0, 1.0, e) * rng.uniform(1, 2, (nb, M, K))
    Bm = np.where((k[:, None] + j) % 2 == 1, 1.0, e) * rng.uniform(1, 2, (nb, K, N))
    return A, Bm


def scattered(rng, nb, M, N, K, p):
    """Entries of unrelated size, some of them zero."""
    A = rng.standard_normal((nb, M, K)) * 2.0 ** rng.uniform(-p, 0, (nb, M, K))
    Bm = rng.standard_normal((nb, K, N)) * 2.0 ** rng.uniform(-p, 0, (nb, K, N))
    A[rng.random(A.shape) < 0.2] = 0.0
    Bm[rng.random(Bm.shape) < 0.2] = 0.0
    return A, Bm


def spiked(rng, nb, M, N, K, p):
    """A few large entries per row, at other places than the columns'."""
    A, Bm = rng.standard_normal((nb, M, K)), rng.standard_normal((nb, K, N))
    A[:, :, 3::41] *= 2.0 ** p
    Bm[:, 7::37, :] *= 2.0 ** p
    Bm[:, 3::41, :] = 0.0
    A[:, :, 7::37] *= (rng.random((nb, M, 1)) < 0.1)
    return A, Bm


def check(B, A, Bm):
    C = B.gemm(torch.from_numpy(A).cuda(), torch.from_numpy(Bm).cuda(), alpha=0.75)
    torch.cuda.synchronize()
    assert B.device_error() == 0
    K = A.shape[-1]
    rows = np.arange(0, A.shape[1], max(1, A.shape[1] // 40))
    A, C = A[:, rows], C.cpu().numpy()[:, rows]
    ref = 0.75 * np.matmul(A.astype(np.longdouble), Bm.astype(np.longdouble))
    scale = 0.75 * np.matmul(np.abs(A), np.abs(Bm))
    u = 2.0 ** -53
    assert np.all(np.abs(C - ref) <= 2 * K * u / (1 - K * u) * scale)


@pytest.mark.parametrize("nb, M, N, K", [
    (30, 127, 66, 33), (3, 300, 90, 96), (2, 97, 65, 1030), (120, 33, 50, 50), (1, 17, 1031, 250),
    (1, 1031, 17, 250), (1, 4099, 330, 270)])
@pytest.mark.parametrize("form, p", [(blocks, 0), (blocks, 8), (blocks, 13), (blocks, 40), (blocks, 200),
                                     (alternating, 7), (alternating, 40), (scattered, 12), (scattered, 80),
                                     (spiked, 20), (spiked, 70)])
def test_every_element_within_the_fp64_bound(B, form, p, nb, M, N, K):
    rng = np.random.default_rng(nb + 3 * M + 5 * N + 7 * K + p)
    check(B, *form(rng, nb, M, N, K, p))


def uniform_tt(d, n, r, seed):
    rng = np.random.default_rng(seed)
    ranks = [1] + [r] * (d - 1) + [1]
    return [rng.random((ranks[k], n, ranks[k + 1])) for k in range(d)]


def left_orthogonal(cores):
    out, carry = [], np.eye(1)
    for k, c in enumerate(cores):
        c = np.einsum("ab,bnc->anc", carry, c)
        if k + 1 == len(cores):
            return out + [c]
        q, carry = np.linalg.qr(c.reshape(-1, c.shape[2]))
        out.append(q.reshape(c.shape[0], c.shape[1], -1))


@pytest.mark.parametrize("d, r", [(20, 50), (12, 50), (20, 24)])
def test_a_tensor_minus_its_orthogonal_form_is_zero(B, d, r):
    y = uniform_tt(d, 32, r, d + r)
    Y = [torch.from_numpy(c).cuda() for c in y]
    X = [torch.from_numpy(np.ascontiguousarray(c)).cuda() for c in left_orthogonal(y)]
    D = B.tt_lincomb([Y, X], [1.0, -1.0])
    norm2 = float(B.tt_dot(Y, Y))
    assert abs(float(B.tt_dot(D, D))) <= 1e-12 * norm2
    rnd = B.Rounder(D, max_rank=0, tol=1e-10)
    rnd.run()
    torch.cuda.synchronize()
    R = rnd.result()
    assert float(B.tt_dot(R, R)) <= 1e-24 * norm2


@pytest.mark.parametrize("nb, M, N, K", [(3, 300, 90, 96), (1, 1031, 17, 250), (1, 4099, 330, 270)])
def test_infinities_stay_infinities(B, nb, M, N, K):
    """Infinities and NaN of an operand reach the outputs that FP64 arithmetic gives them, with
    their sign, and no others."""
    rng = np.random.default_rng(K)
    A, Bm = rng.standard_normal((nb, M, K)), rng.standard_normal((nb, K, N))
    A[0, 3, 1], A[-1, 7, K - 1], A[0, M - 1, K // 2] = np.inf, -np.inf, np.nan
    A[0, 12, 5], A[0, 12, 40] = np.inf, -np.inf
    Bm[0, 9, 2], Bm[-1, K - 3, N - 1] = -np.inf, np.inf
    Bm[0, 1, 5] = 0.0                                       # 0 inf
    C = B.gemm(torch.from_numpy(A).cuda(), torch.from_numpy(Bm).cuda())
    torch.cuda.synchronize()
    C = C.cpu().numpy()
    rows = sorted({3, 7, M - 1, 12} | set(range(0, M, max(1, M // 40))))
    A, C = A[:, rows], C[:, rows]
    with np.errstate(invalid="ignore"):
        ref = np.array([[[np.sum(a * b) for b in Bm[q].T] for a in A[q]] for q in range(nb)])
        scale = np.array([[[np.sum(np.abs(a * b)) for b in Bm[q].T] for a in A[q]] for q in range(nb)])
    assert np.isinf(ref).any() and np.isnan(ref).any()
    assert np.array_equal(np.isnan(C), np.isnan(ref))
    assert np.array_equal(C[np.isinf(ref)], ref[np.isinf(ref)])
    fine = np.isfinite(ref)
    u = 2.0 ** -53
    assert np.all(np.abs(C[fine] - ref[fine]) <= 4 * K * u * scale[fine])
