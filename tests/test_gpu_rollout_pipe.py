"""The pipelined rollout (a cluster per sample, all windows that share a row
advanced together) against the FP64 oracle at the edges of its shapes: units
that do not divide over the cluster, odd hidden and input sizes, one to four
layers, window lengths around the instantiated widths, more samples than
clusters run at once, a single step, and the shapes it hands to the other
kernels (window 17, FP32 weights too large for shared memory)."""
import numpy as np
import pytest
import torch

import oracle.lstm as OL
import paper_2504_15350_gb300.rpod as R

pytestmark = pytest.mark.gpu


def bf16_weights(theta, I, H, L, O):
    out, off = theta.copy(), 0
    for shp in OL.param_shapes(I, H, L, O):
        n = int(np.prod(shp))
        if len(shp) == 2:
            out[off:off + n] = torch.from_numpy(theta[off:off + n]).to(torch.bfloat16).double().numpy()
        off += n
    return out


@pytest.mark.parametrize("I,H,L,O,T,B,steps,fp32", [
    (7, 33, 1, 5, 4, 3, 9, False), (9, 50, 3, 7, 10, 2, 12, False), (6, 21, 2, 6, 5, 1, 1, False),
    (61, 100, 2, 57, 8, 5, 30, False), (5, 4, 1, 3, 11, 2, 7, False), (12, 65, 4, 9, 12, 2, 20, False),
    (54, 256, 2, 50, 10, 19, 25, False), (8, 48, 2, 8, 16, 2, 40, False), (5, 3, 2, 4, 1, 2, 6, False),
    (10, 130, 1, 8, 6, 4, 15, True), (9, 51, 3, 7, 10, 2, 12, True), (6, 40, 2, 5, 17, 2, 8, False),
    (54, 256, 2, 50, 10, 2, 8, True)])
def test_rollout_matches_oracle_at_shape_edges(I, H, L, O, T, B, steps, fp32):
    rng = np.random.default_rng(I + 3 * H + L + T + B)
    theta = (rng.uniform(-1.0, 1.0, OL.param_count(I, H, L, O)) / np.sqrt(H)).astype(np.float32)
    theta = theta.astype(np.float64)
    win = rng.standard_normal((B, T, I)).astype(np.float32)
    ref = OL.rollout(theta if fp32 else bf16_weights(theta, I, H, L, O), win.astype(np.float64), I - O,
                     steps, H, L, O)
    net = R.LSTM(I, H, L, O, T, max_batch=B, theta=theta, fp32_weights=fp32)
    out = net.rollout(torch.from_numpy(win).cuda(), I - O, steps)
    assert net.status() == R.RPOD_OK
    out = out.cpu().numpy()
    # FP32 gates and sums over K <= 2 H + I terms, 24 u per activation
    # (u = 2^-24), carried through steps of a contractive map
    assert np.linalg.norm(out - ref) <= 1e-5 * np.linalg.norm(ref)
