"""GPU tests of the eigen start's cluster pass where its vectors spread over the
warps (vector g belongs to warp g mod 32): exact multiplicities whose clusters
end at, before and after multiples of 32, up to l = 128, and clusters at both
ends of the spectrum.  Tolerances: those of tests/test_gpu_eig.py for the FP32
form on the same kind of matrix."""
import numpy as np
import pytest
import torch

import paper_2504_15350_gb300.rpod as R
from tests.rpod_checks import max_angle, orth_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2504_15350_gb300.build import build
    build()
    R.load()


@pytest.mark.parametrize("groups,p", [
    ([(1.0, 2)], 2),
    ([(4.0, 31), (1.0, 1)], 1),
    ([(4.0, 1), (1.0, 32)], 2),
    ([(8.0, 33), (4.0, 2), (2.0, 30)], 4),
    ([(8.0, 64), (4.0, 3), (2.0, 29)], 8),
    ([(4.0, 97), (2.0, 3), (1.0, 20)], 8),
])
def test_large_clusters(groups, p):
    n, m = 2048, 600
    s = np.concatenate([np.full(c, v) for v, c in groups])
    J = s.size
    rng = np.random.default_rng(J)
    U0, _ = np.linalg.qr(rng.standard_normal((n, J)))
    V0, _ = np.linalg.qr(rng.standard_normal((m, J)))
    S = torch.from_numpy((U0 * s) @ V0.T)
    plan = R.Plan(n, m, J, p, 1, seed=3, compute="f32", flags=R.RPOD_FLAG_RETURN_ALL_L)
    U, sig, _ = plan.basis(S.t().contiguous().float().cuda().t())
    rc, _ = plan.status()
    assert rc == R.RPOD_OK, R.rpod_strerror(rc)
    sig, U = sig.cpu().numpy(), U.double().cpu().numpy()[:, :J]
    assert np.all(np.abs(sig[:J] - s) <= 1e-5 * s)
    assert orth_err(U) <= 1e-5
    c = 0
    for v, mult in groups:
        assert max_angle(U0[:, c:c + mult], U[:, c:c + mult]) <= 1e-4, (v, mult)
        c += mult
