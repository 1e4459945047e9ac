"""GPU: batched filters of tables below a block's rows (fewer steps per warp) and few-groups plans on both sides of the
rows from which their blocks are larger, against the oracle."""
import numpy as np
import pytest

import oracle
from tests.plan_util import compare, gpu_plan_collect, gpu_plan_prepare

pytestmark = pytest.mark.gpu


def _run(specs):
    import paper_2203_01877_gb300 as tqp
    prep = [gpu_plan_prepare(**s) for s in specs]
    ctx = tqp.Context(0, 1 << 30)
    try:
        b = tqp.tqp_batch_create(ctx, [p[0] for p in prep], [p[1] for p in prep])
        tqp.tqp_batch_run(b)
        ctx.check()
        tqp.tqp_batch_destroy(b)
    finally:
        ctx.close()
    for s, (_, _, bufs, _, shape) in zip(specs, prep):
        want = oracle.run_plan(want_pairs=False, cap_groups=None, want_row_ids=bool(s.get("want_row_ids")),
                               **{k: v for k, v in s.items() if k not in ("want_row_ids", "capacity_groups")})
        compare(dict(gpu_plan_collect(bufs, shape), status=0), want, s)


def test_small_filters():
    specs = []
    for n in (1, 127, 128, 129, 511, 1023, 1024, 1025, 2047, 2048, 2049, 4095, 4096, 4097, 8193):
        rng = np.random.default_rng(n)
        specs.append(dict(fact=[rng.integers(0, 1000, n).astype(np.int32), rng.integers(-10**9, 10**9, n)],
                          preds=[(0, "lt", 10 + n % 900)], sum_expr=[("col", 1)], want_row_ids=True))
    _run(specs)


@pytest.mark.parametrize("rows", [(1 << 24) - 4096, 1 << 24])
def test_few_groups(rows):
    rng = np.random.default_rng(rows)
    specs = []
    for n in (rows // 2 + 33, rows // 2 - 33):
        specs.append(dict(fact=[rng.integers(0, 3, n).astype(np.uint8), rng.integers(0, 1000, n)],
                          preds=[(1, "lt", 700)], group_cols=[0], aggs=[("sum", [("col", 1)]), ("count", None)],
                          capacity_groups=16))
    _run(specs)
