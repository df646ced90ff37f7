"""FP32 products on the tensor cores (every value as an exact sum of three
bf16 parts) against FP64, through the calls that use them: projections with
every tile width (columns 1..128), row counts and depths around the 128 x 64
tiles, split and unsplit ranges of k, and snapshots that TMA cannot address;
bases of both operand orders at such sizes."""
import numpy as np
import pytest
import torch

import paper_2504_15350_gb300.rpod as R

pytestmark = pytest.mark.gpu


def colmajor(a, ld, device="cuda"):
    """a (rows x cols) as a column-major view with leading dimension ld."""
    buf = torch.full((a.shape[1], ld), float("nan"), dtype=a.dtype, device=device)
    buf[:, :a.shape[0]] = a.t().to(device)
    return buf[:, :a.shape[0]].t()


@pytest.mark.parametrize("n,kc,mn,pad", [
    (64, 1, 1, 0), (63, 5, 127, 1), (65, 16, 128, 3), (128, 33, 129, 0), (1000, 60, 401, 0),
    (1003, 64, 77, 0), (4096, 65, 500, 4), (4099, 96, 260, 0), (20000, 97, 130, 0),
    (30001, 128, 1000, 2), (16384, 100, 20000, 0)])
def test_projection_is_as_accurate_as_fp32(n, kc, mn, pad):
    g = torch.Generator().manual_seed(n + kc + mn)
    U = torch.randn(n, kc, generator=g) * torch.exp(torch.randn(n, kc, generator=g))
    S = torch.randn(n, mn, generator=g) * torch.exp(torch.randn(n, mn, generator=g))
    plan = R.Plan(n, max(kc, 8), kc, 0, 1, compute="f32")
    C = plan.project(U.t().contiguous().cuda().t(), colmajor(S, n + pad))
    assert plan.status()[0] == R.RPOD_OK
    Ud, Sd = U.double().cuda(), S.double().cuda()
    ref, size = Ud.t() @ Sd, Ud.abs().t() @ Sd.abs()
    err = (C.double() - ref).abs()
    # per entry: at most 24 truncated additions of 2^-23 within 64 values of
    # k and one rounding per 64 of them; in norm, random signs leave far less
    # (a product of parts left out would be at least 2^-18)
    assert bool((err <= (24 + n / 64) * 2.0 ** -23 * size).all())
    assert float(err.norm()) <= 2.0 ** -21 * float(ref.norm())


@pytest.mark.parametrize("n,m,k,p,pad", [(257, 129, 20, 4, 0), (1001, 333, 30, 10, 0), (640, 1217, 50, 14, 3),
                                         (5000, 301, 90, 10, 1), (300, 9000, 100, 28, 0)])
def test_basis_spans_and_values(n, m, k, p, pad):
    """A matrix of exact rank k + p with well separated singular values:
    sigma, U U^T and U C against FP64 at FP32's rounding level."""
    g = torch.Generator().manual_seed(n + m)
    r = k + p
    A = torch.linalg.qr(torch.randn(n, r, generator=g, dtype=torch.float64))[0]
    B = torch.linalg.qr(torch.randn(m, r, generator=g, dtype=torch.float64))[0]
    s = 2.0 ** (-4.0 * torch.arange(r, dtype=torch.float64) / r)
    S = ((A * s) @ B.t()).float()
    plan = R.Plan(n, m, k, p, 1, seed=3, compute="f32")
    U, sig, C = plan.basis(colmajor(S, n + pad))
    assert plan.status()[0] == R.RPOD_OK
    U, C, sig = U.double().cpu(), C.double().cpu(), sig.cpu()
    Ue, se, _ = torch.linalg.svd(S.double(), full_matrices=False)
    assert float((sig[:k] - se[:k]).abs().max()) <= 2e-6 * float(se[0])
    assert float((U.t() @ U - torch.eye(k, dtype=torch.float64)).abs().max()) <= 4e-6
    assert float((C - U.t() @ S.double()).norm()) <= 4e-6 * float(C.norm())
    # U_k spans the leading k directions up to rounding over the gap
    gap = float(se[k - 1] - se[k]) if k < r else float(se[k - 1])
    R_ = U - Ue[:, :k] @ (Ue[:, :k].t() @ U)
    assert float(torch.linalg.matrix_norm(R_, 2)) <= 2e-5 + 4e-6 / gap


def test_nonfinite_input_is_flagged():
    S = torch.randn(300, 200, device="cuda")
    S[37, 111] = float("inf")
    plan = R.Plan(200, 300, 10, 5, 1, compute="f32")
    plan.basis(S.t())
    assert plan.status()[0] == R.RPOD_ERR_NONFINITE
