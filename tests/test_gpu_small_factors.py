"""Small factorizations at the edges of their kernels.

FP64 Cholesky factors up to l = 64 and above, of sampled matrices that are
regular, graded, and of exact rank below l (part of the columns dropped, part
kept).  The FP32 Gram of T^T in 32-row tiles, chunks of up to 256 rows and 4 x 4
blocks, at row counts around them and ranks that leave one to three columns of a
block."""
import numpy as np
import pytest
import torch

import paper_2504_15350_gb300.rpod as R
from tests.rpod_checks import max_angle, orth_err

pytestmark = pytest.mark.gpu


def _case(n, m, s, seed=0):
    rng = np.random.default_rng(seed + n + m)
    U0, _ = np.linalg.qr(rng.standard_normal((n, s.size)))
    V0, _ = np.linalg.qr(rng.standard_normal((m, s.size)))
    return U0, torch.from_numpy((U0 * s) @ V0.T)


def _basis(S, k, p, q, compute):
    plan = R.Plan(S.shape[0], S.shape[1], k, p, q, seed=4, compute=compute, flags=R.RPOD_FLAG_RETURN_ALL_L)
    U, sig, _ = plan.basis(S.t().contiguous().cuda().t())
    rc, warn = plan.status()
    assert rc == R.RPOD_OK, R.rpod_strerror(rc)
    return U.double().cpu().numpy(), sig.cpu().numpy(), warn


@pytest.mark.parametrize("l", [1, 2, 15, 16, 17, 63, 64, 65])
def test_fp64_graded(l):
    s = 10.0 ** (-6.0 * np.arange(l) / max(l - 1, 1))
    U0, S = _case(400, 200, s)
    U, sig, warn = _basis(S, l, 0, 1, "f64")
    # rank l exactly, values down to 1e-6 sigma_1: the bounds of the FP64 form
    assert np.all(np.abs(sig - s) <= 1e-10 * s + 1e-12)
    assert orth_err(U) <= 1e-12
    assert max_angle(U0, U) <= 1e-8
    assert not warn & R.RPOD_WARN_RANK_DEFICIENT


@pytest.mark.parametrize("l", [6, 17, 63, 64, 65])
def test_fp64_some_columns_dropped(l):
    s = np.array([5.0, 4.0, 3.0, 2.0, 1.0])
    U0, S = _case(400, 200, s)
    U, sig, warn = _basis(S, l, 0, 1, "f64")
    assert warn & R.RPOD_WARN_RANK_DEFICIENT
    # as tests/test_gpu_rpod.py for an exact rank
    assert np.allclose(sig[:5], s, rtol=1e-10)
    assert np.all(sig[5:] <= 1e-7 * s[0])
    assert max_angle(U0, U[:, :5]) <= 1e-8


@pytest.mark.parametrize("l", [1, 3, 30, 31, 86, 127, 128])
@pytest.mark.parametrize("m", [131, 255, 256, 257, 513, 4099])
def test_fp32_gram_of_t(m, l):
    s = 2.0 ** (-4.0 * np.arange(l) / l)
    _, S = _case(300, m, s)
    U, sig, _ = _basis(S.float(), l, 0, 1, "f32")
    # rank l exactly: sigma and U at FP32's rounding level, as the FP32 form's
    # other tests
    assert np.abs(sig - s).max() <= 2e-6
    assert orth_err(U) <= 4e-6
