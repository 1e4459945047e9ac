"""GPU: the autotuner's choice for a plan does not select the form of the filter inside it: the plain-load scan, which
has no device-side wait, runs there (the staged one would report an expired wait under a limit of one poll)."""
import numpy as np
import pytest

import datagen
import oracle
from tests.plan_util import compare, gpu_plan_collect, gpu_plan_prepare

pytestmark = pytest.mark.gpu


def test_filter_of_a_tuned_plan():
    import paper_2203_01877_gb300 as tqp
    t = datagen.fact_table(1_500_003, seed=3, cols=["date", "discount", "quantity", "price"])
    spec = dict(fact=[t[c] for c in ("date", "discount", "quantity", "price")], preds=[(0, "le", 2450)],
                sum_expr=[("col", 3), ("col", 1), "mul"], want_row_ids=True)
    want = oracle.run_plan(want_pairs=False, cap_groups=None, **spec)
    plan, res, bufs, keep, shape = gpu_plan_prepare(**spec)
    ctx = tqp.Context(0, 1 << 30)
    try:
        ctx.set_autotune(True)
        tqp.tqp_run_plan(ctx, plan, res)
        ctx.check()
        assert ctx.tuned_count == 1
        bufs["row_ids"].fill_(-7)
        ctx.set_wait_limit(1)
        tqp.tqp_run_plan(ctx, plan, res)
        assert ctx.status() == 0
        compare(dict(gpu_plan_collect(bufs, shape), status=0), want, spec)
    finally:
        ctx.close()


def test_tuned_hash_join():
    import torch
    import paper_2203_01877_gb300 as tqp
    from tests.gpu_util import up
    rng = np.random.default_rng(1)
    bk, pk = rng.permutation(60_000).astype(np.int32) * 11, (rng.integers(0, 90_000, 700_001) * 11).astype(np.int32)
    wb, wp = oracle.join_pairs(bk, pk)
    B, P = tqp.TableRef([up(bk)]), tqp.TableRef([up(pk)])
    ob, op = (torch.zeros(len(wb), dtype=torch.int32, device="cuda") for _ in range(2))
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    ctx = tqp.Context(0, 512 << 20)
    try:
        ctx.set_autotune(True)
        for _ in range(2):
            tqp.tqp_hash_join(ctx, B, 0, P, 0, ob, op, len(wb), cnt)
            ctx.check()
            assert int(cnt.item()) == len(wb)
            assert np.array_equal(ob.cpu().numpy(), wb) and np.array_equal(op.cpu().numpy(), wp)
    finally:
        ctx.close()
