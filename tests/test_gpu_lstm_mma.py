"""The tensor-core LSTM cells and weight gradients against the FP64 oracle at
the edges of their tiles: batches around 16, 32 and 64, hidden, input and
output sizes that are odd or one past a tile, one to four layers, one-step
windows, dropout between layers."""
import numpy as np
import pytest
import torch

import oracle.lstm as OL
import paper_2504_15350_gb300.rpod as R
from tests.test_gpu_rollout_pipe import bf16_weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("I,H,L,O,T,B,p", [
    (1, 1, 1, 1, 1, 1, 0.0), (5, 33, 3, 4, 2, 33, 0.0), (7, 21, 2, 7, 4, 65, 0.3), (65, 64, 2, 63, 3, 32, 0.0),
    (20, 100, 4, 11, 6, 129, 0.1), (67, 17, 2, 66, 5, 17, 0.5), (12, 129, 1, 9, 7, 64, 0.0),
    (33, 48, 2, 32, 12, 100, 0.0)])
def test_forward_loss_and_gradients(I, H, L, O, T, B, p):
    rng = np.random.default_rng(I + H + L + B)
    theta = (rng.uniform(-1.0, 1.0, OL.param_count(I, H, L, O)) / np.sqrt(H)).astype(np.float32)
    theta = theta.astype(np.float64)
    X = rng.standard_normal((B, T, I)).astype(np.float32)
    Y = rng.standard_normal((B, O)).astype(np.float32)
    te = bf16_weights(theta, I, H, L, O)
    net = R.LSTM(I, H, L, O, T, max_batch=B + 3, theta=theta)
    Xd, Yd = torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()
    y_o, _ = OL.forward(te, X.astype(np.float64), H, L, O)
    # FP32 rounding (u = 6e-8) over sums of at most 300 terms and the gates'
    # fast exponential, carried through T L cells and back: 2e-5 of a block's
    # largest entry, as the start of the chain leaves 24 u
    assert np.abs(net.forward(Xd).cpu().numpy() - y_o).max() <= 2e-5 * np.abs(y_o).max()
    drop = None
    if p > 0.0:
        net.set_dropout(p, 77)
        drop = (p, 77, 0)
    y_o, cache = OL.forward(te, X.astype(np.float64), H, L, O, dropout=drop)
    loss_o, dy = OL.mse(y_o, Y.astype(np.float64))
    g_o = OL.backward(te, cache, dy, H, L, O)
    loss, g = net.loss_grad(Xd, Yd)
    assert abs(loss.item() - loss_o) <= 1e-5 * loss_o
    g, off = g.cpu().numpy(), 0
    for shp in OL.param_shapes(I, H, L, O):
        n = int(np.prod(shp))
        ref = g_o[off:off + n]
        assert np.abs(g[off:off + n] - ref).max() <= 2e-5 * max(np.abs(ref).max(), 1e-30), shp
        off += n
