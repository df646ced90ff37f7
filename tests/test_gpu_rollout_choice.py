"""Which kernels a rollout takes: many windows over few steps go to a
prediction's own kernels (one launch per phase), where the cluster kernel would
load the weights and run the whole window once per wave of samples; few windows
or many steps to one of the single-launch kernels.  All agree with the oracle."""
import numpy as np
import pytest
import torch

import oracle.lstm as OL
import paper_2504_15350_gb300.rpod as R
from tests.test_gpu_rollout_pipe import bf16_weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("I,H,L,O,T,B,steps,per_step", [
    (54, 256, 2, 50, 10, 512, 1, True), (54, 256, 2, 50, 10, 512, 10, True), (54, 256, 2, 50, 10, 64, 5, True),
    (54, 256, 2, 50, 10, 64, 60, False), (54, 256, 2, 50, 10, 8, 30, False), (14, 50, 3, 10, 10, 513, 3, True),
    (15, 51, 3, 11, 10, 16, 40, False)])
def test_rollout_choice(I, H, L, O, T, B, steps, per_step):
    rng = np.random.default_rng(H + B + steps)
    theta = (rng.uniform(-1.0, 1.0, OL.param_count(I, H, L, O)) / np.sqrt(H)).astype(np.float32)
    win = rng.standard_normal((B, T, I)).astype(np.float32)
    net = R.LSTM(I, H, L, O, T, max_batch=B, theta=theta)
    out = net.rollout(torch.from_numpy(win).cuda(), I - O, steps)
    assert net.status() == R.RPOD_OK
    assert (net.launches() > steps * (L + T - 1)) == per_step
    rows = np.unique(np.linspace(0, B - 1, 12).astype(int))
    ref = OL.rollout(bf16_weights(theta.astype(np.float64), I, H, L, O), win[rows].astype(np.float64),
                     I - O, steps, H, L, O)
    # as tests/test_gpu_rollout_pipe.py
    assert np.linalg.norm(out.cpu().numpy()[rows] - ref) <= 1e-5 * np.linalg.norm(ref)
