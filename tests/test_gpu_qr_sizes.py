"""Cholesky QR at the sizes where its panels, column slots and launch forms change
(odd and even column counts, multiples of 16 and 32, the last size of the
one-cluster form and the first of the whole-GPU form): orthonormal cores, the
oracle's result, and bitwise the launch-per-step form's.

Bounds: 6 (m c + c (c + 1)) u for |Q^T Q - I| (Cholesky QR2, Yamamoto et al. 2015),
the FP64 parity bar 1e-12 against the oracle."""
import hashlib
import json
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import hatt as ohatt
from oracle import tt as ott
from paper_2410_04385_gb300 import workloads as wl

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SIZES = [(1, 3), (2, 5), (3, 40), (4, 9), (15, 10), (16, 11), (17, 30), (31, 8), (32, 7), (33, 20), (50, 2),
         (50, 3), (63, 5), (64, 33), (65, 4), (96, 17), (97, 6), (127, 4), (128, 9)]


def result(c, n, graded=False):
    from paper_2410_04385_gb300 import binding
    r = max(2, int(np.ceil(np.sqrt(c))) + 1)
    dims = [max(4, c), n, max(4, c)]
    Y = wl.gaussian_tt(dims, [1, r, r, 1], 70 + c)
    Z = wl.gaussian_tt(dims, [1, r, r, 1], 71 + c)
    if graded:                                     # a wide spectrum: several passes, shifted ones among them
        for T in (Y, Z):
            T[1] = T[1] * (10.0 ** -np.linspace(0, 7, r))[:, None, None]
    X = binding.tt_hadamard_recompress([torch.from_numpy(x).cuda() for x in Y],
                                       [torch.from_numpy(x).cuda() for x in Z], sketch_rank=c, seed=c)
    return Y, Z, [x.cpu().numpy() for x in X]


@pytest.mark.parametrize("c, n", SIZES)
@pytest.mark.parametrize("graded", [False, True])
def test_orthonormal_and_the_oracles(c, n, graded):
    from paper_2410_04385_gb300 import binding
    Y, Z, X = result(c, n, graded)
    assert binding.device_error() == 0
    for x in X[:-1]:
        Q = x.reshape(-1, x.shape[2])
        m, k = Q.shape
        assert np.abs(Q.T @ Q - np.eye(k)).max() <= 6 * (m * k + k * (k + 1)) * 2.0 ** -53
    Xo = ohatt.hadamard_recompress(Y, Z, sketch_rank=c, seed=c)
    if not graded:
        assert ott.tt_diff_norm(X, Xo) <= 1e-12 * ott.tt_norm(Xo)
    A = ott.hadamard_pkp(Y, Z)
    assert ott.tt_rel_error(X, A) <= ott.tt_rel_error(Xo, A) + 1e-12


def test_launch_per_step_form_is_bitwise_the_same():
    script = ("import sys; sys.path.insert(0, %r)\nfrom tests import test_gpu_qr_sizes as T\nT.digest()" % ROOT)
    sha = []
    for form in ("steps", ""):
        p = subprocess.run([sys.executable, "-c", script], capture_output=True, text=True, timeout=600, cwd=ROOT,
                           env=dict(os.environ, HATT_QR_FORM=form))
        assert p.returncode == 0, p.stderr[-2000:]
        sha.append(json.loads(p.stdout.strip().splitlines()[-1]))
    assert sha[0] == sha[1]


def digest():
    out = []
    for c, n in SIZES:
        h = hashlib.sha256()
        for x in result(c, n)[2]:
            h.update(x.tobytes())
        out.append(h.hexdigest())
    print(json.dumps(out))
