"""FP32 products with the l x l factors where the kernel changes: matrices up to 768
x 768 (one launch each) and above, l at the tile widths 32 and 64 and beside
them."""
import numpy as np
import pytest
import torch

import paper_2504_15350_gb300.rpod as R

pytestmark = pytest.mark.gpu


def _run(n, m, l, ld=None):
    rng = np.random.default_rng(n + l)
    s = 2.0 ** (-4.0 * np.arange(l) / l)
    U0, _ = np.linalg.qr(rng.standard_normal((n, l)))
    V0, _ = np.linalg.qr(rng.standard_normal((m, l)))
    S = torch.from_numpy((U0 * s) @ V0.T).float()
    plan = R.Plan(n, m, l, 0, 1, seed=1, compute="f32")
    U, sig, C = plan.basis(S.t().contiguous().cuda().t())
    rc, _ = plan.status()
    assert rc == R.RPOD_OK, R.rpod_strerror(rc)
    return s, S.double().numpy(), U.double().cpu().numpy(), sig.cpu().numpy(), C.double().cpu().numpy(), plan


@pytest.mark.parametrize("n,m", [(200, 150), (768, 140), (769, 300), (150, 768), (150, 769)])
@pytest.mark.parametrize("l", [1, 31, 32, 33, 64, 65, 128])
def test_bases_around_the_switch(n, m, l):
    s, S, U, sig, C, _ = _run(n, m, l)
    # FP32 rounding of sums of at most 769 terms, as the FP32 form's other tests
    assert np.abs(sig - s).max() <= 2e-6
    assert np.abs(U.T @ U - np.eye(l)).max() <= 4e-6
    assert np.linalg.norm(C - U.T @ S) <= 4e-6 * np.linalg.norm(C)


def test_small_factors_take_one_launch():
    # four applies, the fold, the lift and the coefficients: one launch each at
    # 600 x 250; the sketch pass, S^T Q and so on are the same at both sizes
    small = _run(600, 250, 30)[5].launches()
    large = _run(4200, 4200, 30)[5].launches()
    assert small <= large - 6, (small, large)
