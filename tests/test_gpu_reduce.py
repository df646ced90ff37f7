"""Sums of split l x l products at the counts where the kernel changes (one, up to
eight, more): bases whose Grams take 1, 2, 7, 8, 9 and 33 splits, ranks that
leave a partial CTA."""
import numpy as np
import pytest
import torch

import paper_2504_15350_gb300.rpod as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("compute", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("n,l", [(300, 11), (520, 12), (1800, 30), (2048, 45), (2304, 64), (8500, 20)])
def test_grams_of_few_splits(n, l, compute):
    m = 280
    rng = np.random.default_rng(n)
    s = 2.0 ** (-4.0 * np.arange(l) / l)
    U0, _ = np.linalg.qr(rng.standard_normal((n, l)))
    V0, _ = np.linalg.qr(rng.standard_normal((m, l)))
    S = torch.from_numpy((U0 * s) @ V0.T)
    S = S if compute == "f64" else S.float()
    flags = R.RPOD_FLAG_REFINE_FP32 if compute == "bf16" else 0
    plan = R.Plan(n, m, l - 2, 2, 1, seed=1, compute=compute, flags=flags)
    U, sig, _ = plan.basis(S.t().contiguous().cuda().t())
    rc, _ = plan.status()
    assert rc == R.RPOD_OK, R.rpod_strerror(rc)
    U = U.double().cpu().numpy()
    # rank l exactly: the forms' bounds on sigma and orthogonality
    tol = {"f64": 1e-11, "f32": 1e-5, "bf16": 1e-3}[compute]
    assert np.abs(sig.cpu().numpy()[:l - 2] - s[:l - 2]).max() <= tol
    assert np.abs(U.T @ U - np.eye(l - 2)).max() <= (1e-11 if compute == "f64" else 1e-5)
