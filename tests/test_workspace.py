"""Workspace sizes (no GPU needed): the FP32 form's plans hold the partial sums that
their products use, in a batch as alone."""
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
