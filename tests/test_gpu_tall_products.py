"""GPU tests of the m-sized products behind T at the edges of their tiles: the
Gram of T^T (8 x 8 blocks of the upper triangle, 32-row tiles, 64-row chunks)
and, in the 16-bit forms from 4096 snapshots on, the fold of the deferred factor
and the coefficients.

S = U0 diag(sigma) V0^T of exact rank l with sigma spread over 1 .. 1/2, so that
sigma comes out whole and C = U^T S.  Tolerances: sigma as in
tests/test_gpu_eig.py for its forms (FP16 as FP32, whose refinement pass it
shares); C carries the rounding of U (2^-21 of the lift in the 16-bit forms) and,
in the BF16 form, of the TF32 operands of T."""
import numpy as np
import pytest
import torch

import paper_2504_15350_gb300.rpod as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2504_15350_gb300.build import build
    build()
    R.load()


@pytest.mark.parametrize("compute,l,m", [
    ("f32", 1, 64), ("f32", 8, 65), ("f32", 9, 127), ("f32", 60, 9729), ("f32", 64, 33000),
    ("f32", 65, 500), ("f32", 120, 1000), ("f32", 121, 4097), ("f32", 128, 9728),
    ("bf16", 32, 4095), ("bf16", 33, 4096), ("bf16", 85, 4097), ("bf16", 128, 9730),
    ("f16", 31, 4098), ("f16", 85, 5001), ("f16", 120, 4100),
])
def test_small_svd_and_coefficients(compute, l, m):
    n, p = 512, 0 if l < 4 else 3
    rng = np.random.default_rng(l * 1000 + m % 1000)
    U0, _ = np.linalg.qr(rng.standard_normal((n, l)))
    V0, _ = np.linalg.qr(rng.standard_normal((m, l)))
    s = np.linspace(1.0, 0.5, l)
    S = torch.from_numpy((U0 * s) @ V0.T).float()
    flags = R.RPOD_FLAG_REFINE_FP32 if compute != "f32" else 0
    plan = R.Plan(n, m, l - p, p, 1, seed=4, compute=compute, flags=flags)
    U, sig, C = plan.basis(S.t().contiguous().cuda().t())
    rc, _ = plan.status()
    assert rc == R.RPOD_OK, R.rpod_strerror(rc)
    tol = 1e-3 if compute == "bf16" else 1e-5
    assert np.all(np.abs(sig.cpu().numpy() - s) <= tol * s)
    ref = U.double().cpu().numpy().T @ S.double().numpy()
    assert np.abs(C.double().cpu().numpy() - ref).max() <= tol * s[0]
