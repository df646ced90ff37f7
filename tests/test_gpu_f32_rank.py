"""The FP32 form at and below its resolution: matrices of exact rank r < l are
reported and leave r correct values and columns, the rest at rounding level;
spectra that fall far below FP32's resolution within l keep the leading values
and the orthogonality, and are reported once the sampled columns are dependent
(less than 1e-13 of a squared norm left), not before."""
import numpy as np
import pytest
import torch

import paper_2504_15350_gb300.rpod as R
from tests.rpod_checks import max_angle, orth_err

pytestmark = pytest.mark.gpu


def _basis(n, m, s, k, p, q, seed):
    rng = np.random.default_rng(n + m)
    U0, _ = np.linalg.qr(rng.standard_normal((n, s.size)))
    V0, _ = np.linalg.qr(rng.standard_normal((m, s.size)))
    S = torch.from_numpy((U0 * s) @ V0.T).float().t().contiguous().cuda().t()
    plan = R.Plan(n, m, k, p, q, seed=seed, compute="f32", flags=R.RPOD_FLAG_RETURN_ALL_L)
    U, sig, _ = plan.basis(S)
    rc, warn = plan.status()
    assert rc == R.RPOD_OK, R.rpod_strerror(rc)
    return U0, U.double().cpu().numpy(), sig.cpu().numpy(), warn


@pytest.mark.parametrize("n,m,r,k,p", [(600, 250, 5, 20, 10), (2048, 400, 20, 30, 10),
                                       (1500, 6000, 5, 60, 5), (301, 203, 3, 100, 28)])
def test_exact_rank_is_reported(n, m, r, k, p):
    s = 1.0 / (1.0 + np.arange(r))
    U0, U, sig, warn = _basis(n, m, s, k, p, 1, 3)
    assert warn & R.RPOD_WARN_RANK_DEFICIENT
    # FP32 rounding (u = 6e-8) of sums over up to 6000 snapshots: the leading
    # values and vectors as in the FP32 form's other tests, the rest below 100 u
    # sigma_1
    assert np.all(np.abs(sig[:r] - s) <= 1e-5 * s)
    assert np.all(sig[r:] <= 1e-5 * s[0])
    assert max_angle(U0, U[:, :r]) <= 1e-4
    assert orth_err(U[:, :r]) <= 1e-5
    assert np.abs(U[:, :r].T @ U[:, r:]).max() <= 1e-5


@pytest.mark.parametrize("n,m", [(600, 250), (2048, 400), (3000, 1500)])
@pytest.mark.parametrize("e,reported", [(5, False), (7, True), (8, True)])
def test_falling_spectrum(n, m, e, reported):
    s = 10.0 ** (-e * np.arange(120) / 79)  # 10^-e sigma_1 at the l = 80th value
    for seed in range(3):
        _, U, sig, warn = _basis(n, m, s, 70, 10, 2, seed)
        # as above, and the part of the spectrum behind l that q = 2 leaves (a
        # few 1e-6 at e = 5)
        assert np.all(np.abs(sig - s[:80]) <= 3e-5), seed
        assert orth_err(U) <= 1e-5, seed
        assert bool(warn & R.RPOD_WARN_RANK_DEFICIENT) == reported, seed
