"""Windows and targets with infinite entries.  An infinite input saturates the
gates of its step (W_x has no zeros), so the prediction and the loss stay
finite and every gradient stays finite but the columns of the first W_x that
the infinite inputs multiply (zero times infinity); an infinite target makes
the loss and its own bias gradient infinite.  Both batch tilings, odd sizes."""
import numpy as np
import pytest
import torch

import oracle.lstm as OL
import paper_2504_15350_gb300.rpod as R
from tests.test_gpu_rollout_pipe import bf16_weights

pytestmark = pytest.mark.gpu


def _case(I, H, L, O, T, B):
    rng = np.random.default_rng(H + B)
    theta = (rng.uniform(-1.0, 1.0, OL.param_count(I, H, L, O)) / np.sqrt(H)).astype(np.float32)
    theta = theta.astype(np.float64)
    X = rng.standard_normal((B, T, I)).astype(np.float32)
    Y = rng.standard_normal((B, O)).astype(np.float32)
    return theta, X, Y, R.LSTM(I, H, L, O, T, max_batch=B, theta=theta)


@pytest.mark.parametrize("I,H,L,O,T,B", [(6, 32, 2, 4, 5, 3), (6, 32, 2, 4, 5, 40), (7, 33, 1, 5, 4, 65)])
def test_infinite_window_entries_saturate(I, H, L, O, T, B):
    theta, X, Y, net = _case(I, H, L, O, T, B)
    X[1, T - 1, 3], X[2, 0, 1] = np.inf, -np.inf
    te = bf16_weights(theta, I, H, L, O)
    with np.errstate(over="ignore", invalid="ignore"):
        y_o, cache = OL.forward(te, X.astype(np.float64), H, L, O)
        loss_o, dy = OL.mse(y_o, Y.astype(np.float64))
        g_o = OL.backward(te, cache, dy, H, L, O)
    assert np.isfinite(y_o).all()
    Xd, Yd = torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()
    # the tolerances of the finite case (tests/test_gpu_lstm_mma.py): a saturated
    # gate is exact
    assert np.abs(net.forward(Xd).cpu().numpy() - y_o).max() <= 2e-5 * np.abs(y_o).max()
    loss, g = net.loss_grad(Xd, Yd)
    assert abs(loss.item() - loss_o) <= 1e-5 * loss_o
    g, off = g.cpu().numpy(), 0
    hit = np.zeros(g.size, bool)
    hit[:4 * H * I].reshape(4 * H, I)[:, [1, 3]] = True
    assert np.isfinite(g[~hit]).all() and not np.isfinite(g[hit]).any()
    for shp in OL.param_shapes(I, H, L, O):
        n = int(np.prod(shp))
        keep = ~hit[off:off + n]
        ref = g_o[off:off + n][keep]
        assert np.abs(g[off:off + n][keep] - ref).max() <= 2e-5 * max(np.abs(ref).max(), 1e-30), shp
        off += n


def test_infinite_target():
    I, H, L, O, T, B = 6, 32, 2, 4, 5, 40
    theta, X, Y, net = _case(I, H, L, O, T, B)
    Y[1, 2] = np.inf
    loss, g = net.loss_grad(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda())
    assert loss.item() == np.inf
    by = g[-O:].cpu().numpy()
    assert by[2] == -np.inf and np.isfinite(by[[0, 1, 3]]).all()
