"""GPU: shared scans on both sides of the line between few queries (totals per row, in registers) and many (a
row queue and transposed masks), with few and many passing rows per step, and the launch shapes and batches
that leave them little shared memory."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import up

pytestmark = pytest.mark.gpu

SUMS = [[("col", 0)], [("col", 0), ("const", 7), ("col", 1), "sub", "mul"]]


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 256 << 20)
    yield c
    c.close()


def _run(ctx, cols, queries):
    import torch
    import paper_2203_01877_gb300 as tqp
    T = tqp.TableRef([up(c) for c in cols])
    outs = [(torch.full((1,), -7, dtype=torch.int64, device="cuda"),
             torch.full((1,), -7, dtype=torch.int64, device="cuda") if e else None) for _, e in queries]
    launch = tqp.tqp_filter_shared(ctx, T, [(p, e, c, s) for (p, e), (c, s) in zip(queries, outs)])
    ctx.check()
    for (p, e), (c, s) in zip(queries, outs):
        ids, total = oracle.filter_rows(cols, p, e)
        assert int(c.item()) == len(ids) and (e is None or int(s.item()) == total), (p, e)
    return launch


@pytest.mark.parametrize("n", [1, 33, 1023, 1025, 70_003])
@pytest.mark.parametrize("nq", [3, 4, 5, 8, 9, 32])
@pytest.mark.parametrize("nexpr", [0, 1, 2])
@pytest.mark.parametrize("span", [2, 120, 1000])
def test_few_and_many(ctx, n, nq, nexpr, span):
    rng = np.random.default_rng(n + nq + span)
    cols = [rng.integers(-2**30, 2**30, n), rng.integers(0, 1000, n).astype(np.int32),
            rng.integers(0, 1000, n).astype((np.int32, np.int64)[nq % 2]), rng.integers(0, 250, n).astype(np.uint8)]
    queries = [([(1 + q % 3, "between", 7 * q % 200, 7 * q % 200 + span)], SUMS[q % nexpr] if nexpr else None)
               for q in range(nq)]
    assert _run(ctx, cols, queries) == [0] * nq


def _wide(n, ncols, extra=()):
    rng = np.random.default_rng(ncols)
    return [rng.integers(0, 8, n) for _ in range(ncols)] + [rng.integers(0, 8, n).astype(t) for t in extra]


@pytest.mark.parametrize("nq", [4, 6, 12])
def test_a_callers_shape_to_the_last_kilobyte(ctx, nq):
    # 37 bytes a row: 2 stages of 3072 rows take 227,328 bytes of shared memory
    cols = _wide(50_001, 4, (np.int32, np.uint8))
    queries = [([(q % 6, "le", 1 + q % 4)], [("col", 0)]) for q in range(nq)]
    try:
        ctx.set_tuning(3072, 2, 1)
        _run(ctx, cols, queries)
    finally:
        ctx.set_tuning(0, 0, 0)


@pytest.mark.parametrize("nq", [4, 16])
@pytest.mark.parametrize("how", ["plans", "batch"])
def test_batched_scans_of_64_byte_rows(ctx, nq, how):
    import paper_2203_01877_gb300 as tqp
    from tests.plan_util import compare, gpu_plan_collect, gpu_plan_prepare
    cols = _wide(20_003, 8)
    ref = tqp.TableRef([up(c) for c in cols])
    specs = [dict(fact=cols, preds=[(q % 8, "le", 1 + q % 5)], sum_expr=[("col", (q + 1) % 2)]) for q in range(nq)]
    prep = [gpu_plan_prepare(fact_ref=ref, **s) for s in specs]
    if how == "batch":
        b = tqp.tqp_batch_create(ctx, [p[0] for p in prep], [p[1] for p in prep])
        tqp.tqp_batch_run(b)
        ctx.check()
        tqp.tqp_batch_destroy(b)
    else:
        tqp.tqp_run_plans(ctx, [p[0] for p in prep], [p[1] for p in prep])
        ctx.check()
    for s, (_, _, bufs, _, shape) in zip(specs, prep):
        compare(dict(gpu_plan_collect(bufs, shape), status=0),
                oracle.run_plan(want_pairs=False, cap_groups=None, want_row_ids=False, **s), s)
