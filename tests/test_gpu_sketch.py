"""FP32 sketch against the FP64 one of the same words (the oracle's, Box-Muller
of Philox4x64-10): evaluated to 2^-32 before the one rounding to FP32, so every
entry lies within 1/2 + 2^-8 ulp of the FP64 value."""
import numpy as np
import pytest
import torch

import paper_2504_15350_gb300.rpod as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,l,seed", [(1, 1, 0), (3, 3, 5), (501, 12, 3), (64000, 60, 1), (90225, 85, 2)])
def test_fp32_sketch_is_the_rounded_fp64_sketch(m, l, seed):
    plan = R.Plan(max(m, 64), m, l, 0, 1, seed=seed, compute="f64" if m < 1000 else "f32")
    ref = plan.sketch(torch.float64).cpu().numpy()
    got = plan.sketch(torch.float32).cpu().numpy()
    ulp = np.spacing(np.abs(ref).astype(np.float32)).astype(np.float64)
    assert np.isfinite(got).all()
    assert (np.abs(got.astype(np.float64) - ref) / ulp).max() <= 0.5 + 2.0 ** -8
