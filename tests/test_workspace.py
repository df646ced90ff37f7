"""Workspace sizes (no GPU needed): the FP32 form's plans hold the partial sums that
their products use, in a batch as alone, and an LSTM the buffers of its own
weight type."""
import pytest

import paper_2504_15350_gb300.rpod as R
from paper_2504_15350_gb300.build import build


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build()
    R.load()


def _batch_bytes(n, m, k, p, compute):
    # nothing is read through the pointers before a run
    inst = R.Instance(n, m, k, p, 1, 0, 256, n, None, 0, 256, n, 256, 256, k)
    h = R.rpod_batch_create([inst], compute, 0, compute)
    try:
        return R.rpod_batch_workspace_bytes(h)
    finally:
        R.rpod_batch_destroy(h)


@pytest.mark.parametrize("n,m,k,p", [(262144, 1000, 50, 10), (65536, 4000, 100, 20), (8192, 1500, 30, 10)])
def test_fp32_partials_are_those_of_its_products(n, m, k, p):
    h = R.rpod_plan_create(n, m, k, p, 1, 0, R.RPOD_F32)
    alone = R.rpod_workspace_bytes(h)
    R.rpod_plan_destroy(h)
    # no launch scale above 100 %, so no more room in a batch
    assert _batch_bytes(n, m, k, p, R.RPOD_F32) == alone
    # Y, Q, the three parts of an operand of n rows, Z, T, the sketch and the
    # l x l work: the rest is partial sums, of 128-row tiles on 152 SMs
    l = k + p
    fixed = 4 * l * (2 * n + 4 * m) + 6 * l * (n + 63) + 8 * 40 * l * l + 16 * 304 * l * l + (1 << 20)
    tiles = -(-m // 128)
    assert alone <= fixed + 4 * l * m * (2 * 152 // tiles + 2), (alone, fixed)


@pytest.mark.parametrize("dims", [(54, 256, 2, 50, 10, 512), (14, 50, 3, 10, 10, 64), (9, 33, 1, 5, 4, 7)])
def test_lstm_buffers_are_those_of_its_weight_type(dims):
    I, H, L, O, T, B = dims
    size = {}
    for flags in (0, R.RPOD_LSTM_FP32_WEIGHTS):
        h = R.rpod_lstm_create(*dims, flags)
        size[flags] = R.rpod_lstm_workspace_bytes(h)
        P = R.rpod_lstm_param_count(h)
        R.rpod_lstm_destroy(h)
    rows, H8, slack = T * B, (H + 7) // 8 * 8, 1 << 15
    # parameters, moments, gradient and BF16 copy; three windows; gates, c and h
    both = 18 * P + 12 * rows * I + 16 * L * rows * H + 8 * L * (T + 1) * B * H + 12 * B * O
    # three BF16 parts of x, h, masked h, dz and dy, dropout masks, dc
    bf16 = 6 * (rows * ((I + 7) // 8 * 8 + (2 * L - 1) * H8 + 4 * L * H8) + B * (O + 8)) + (L - 1) * rows * H
    # input projections, dz, dh, masked h, split sums of the weight gradients
    fp32 = 4 * (4 * L * rows * H + 4 * rows * H + rows * max(I, H) + (L - 1) * rows * H + 128 * H * max(I, H))
    assert size[0] <= both + bf16 + 4 * L * B * H + slack
    assert size[R.RPOD_LSTM_FP32_WEIGHTS] <= both + fp32 + 12 * B * max(H, O) + slack
