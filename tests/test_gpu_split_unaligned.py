"""FP32 products with an operand that TMA cannot address (leading dimension or
base not a multiple of 16 bytes): the staged tiles at the edges of lines, rows
and k-blocks against FP64, and the time against the aligned product's."""
import numpy as np
import pytest
import torch

import paper_2504_15350_gb300.rpod as R

pytestmark = pytest.mark.gpu


def _shifted(rows, cols, shift, gen):
    """A rows x cols column-major view with leading dimension rows, starting
    `shift` elements into its buffer."""
    buf = torch.randn(shift + rows * cols, generator=gen, device="cuda")
    return buf[shift:].reshape(cols, rows).t()


@pytest.mark.parametrize("k", [1, 33, 65, 100])
@pytest.mark.parametrize("n,m,shift", [(63, 1, 1), (64, 127, 1), (65, 128, 0), (129, 129, 2), (191, 257, 3),
                                       (1027, 300, 0), (4096, 260, 1)])
def test_projection_of_unaligned_snapshots(n, m, shift, k):
    k = min(k, n - 1)
    gen = torch.Generator(device="cuda").manual_seed(n + m + k)
    plan = R.Plan(n, max(m, k + 1), k, 1, 0, compute="f32")
    S = _shifted(n, m, shift, gen)
    U = torch.randn(k, n, generator=gen, device="cuda").t()
    C = plan.project(U, S)
    ref = U.double().t() @ S.double()
    # FP32 products and sums of n terms, in 64-term chunks: 1e-6 of the terms'
    # root sum of squares
    scale = U.double().norm(dim=0)[:, None] * S.double().norm(dim=0)[None]
    assert bool(((C.double() - ref).abs() <= 1e-6 * scale).all())


@pytest.mark.parametrize("n,m,shift", [(257, 131, 0), (1030, 195, 0), (384, 257, 1)])
def test_basis_of_unaligned_snapshots(n, m, shift):
    gen = torch.Generator(device="cuda").manual_seed(n)
    s = 0.8 ** torch.arange(60, device="cuda", dtype=torch.float64)
    U0 = torch.linalg.qr(torch.randn(n, 60, generator=gen, device="cuda", dtype=torch.float64))[0]
    V0 = torch.linalg.qr(torch.randn(m, 60, generator=gen, device="cuda", dtype=torch.float64))[0]
    S = _shifted(n, m, shift, gen)
    S.copy_(((U0 * s) @ V0.t()).float())
    plan = R.Plan(n, m, 20, 20, 2, seed=1, compute="f32")
    U, sig, C = plan.basis(S)
    rc, _ = plan.status()
    assert rc == R.RPOD_OK, R.rpod_strerror(rc)
    assert bool(((sig[:20] - s[:20]).abs() <= 1e-5 * s[:20]).all())
    assert float((C.double() - U.double().t() @ S.double()).abs().max()) <= 1e-5
    assert np.abs((U.double().t() @ U.double()).cpu().numpy() - np.eye(20)).max() <= 1e-5


def test_unaligned_product_takes_about_as_long():
    times = {}
    for n in (65536, 65537):
        plan = R.Plan(n, 1000, 100, 10, 1, compute="f32")
        S = torch.ones(2000, n, device="cuda").t()
        U = torch.ones(100, n, device="cuda").t()
        out = plan.project(U, S)
        runs = []
        for _ in range(8):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            plan.project(U, S, out=out)
            b.record()
            b.synchronize()
            runs.append(a.elapsed_time(b))
        times[n] = min(runs)
    # 4-byte copies instead of TMA: a factor below 2 (3.5 with five copies in flight)
    assert times[65537] <= 2.5 * times[65536], times
