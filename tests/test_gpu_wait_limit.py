"""GPU: the context's wait limit bounds every device-side wait. With a limit of one poll the built-in pair join
(look-back over tiles, and the sort of repeated build keys), the sort-based join and group-by, and the radix
select of a top-k give up and report TQP_ERR_TIMEOUT (the look-back's count exact or -1, the select's -1); with
the default limit restored the same call gives the oracle's result, also while the earlier time-out is still latched."""
import numpy as np
import pytest

import datagen
import oracle
from tests.gpu_util import up
from tests.plan_util import compare, gpu_plan_collect, gpu_plan_prepare

pytestmark = pytest.mark.gpu

DEFAULT_WAIT = 1 << 22


@pytest.fixture()
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 1 << 30)
    yield c
    c.close()


@pytest.mark.parametrize("variant", [-1, 1])
@pytest.mark.parametrize("dup", [1, 7])
def test_join(ctx, variant, dup):
    import torch
    import paper_2203_01877_gb300 as tqp
    rng = np.random.default_rng(dup)
    bk = np.repeat(rng.permutation(10 * 50_000)[:50_000], dup).astype(np.int32) * 1001
    rng.shuffle(bk)
    pk = (rng.integers(0, 10 * 50_000, 3_000_000) * 1001).astype(np.int32)
    wb, wp = oracle.join_pairs(bk, pk)
    cap = len(wb) + 16
    B, P = tqp.TableRef([up(bk)]), tqp.TableRef([up(pk)])
    ob, op = (torch.full((cap,), -9, dtype=torch.int32, device="cuda") for _ in range(2))
    cnt = torch.full((1,), -7, dtype=torch.int64, device="cuda")
    ctx.set_variant(variant)
    ctx.set_wait_limit(1)
    for _ in range(3):
        tqp.tqp_hash_join(ctx, B, 0, P, 0, ob, op, cap, cnt)
        assert ctx.status() == tqp.ERR_TIMEOUT
        if variant != 1:
            assert int(cnt.item()) in (-1, len(wb)) or dup > 1
    ctx.set_wait_limit(DEFAULT_WAIT)
    tqp.tqp_hash_join(ctx, B, 0, P, 0, ob, op, cap, cnt)
    assert ctx.status() == 0 and int(cnt.item()) == len(wb)
    assert np.array_equal(ob[:len(wb)].cpu().numpy(), wb) and np.array_equal(op[:len(wb)].cpu().numpy(), wp)


def test_sorted_group_by(ctx):
    import torch
    import paper_2203_01877_gb300 as tqp
    rng = np.random.default_rng(3)
    n = 400_003
    cols = [rng.integers(-2**31, 2**31, 5000)[rng.integers(0, 5000, n)].astype(np.int32), rng.integers(-9, 9, n)]
    T = tqp.TableRef([up(c) for c in cols])
    z = lambda m: torch.full((m,), -7, dtype=torch.int64, device="cuda")  # noqa: E731
    keys, iv, ng = z(8192), z(8192), z(1)
    run = lambda: tqp.tqp_groupby_agg(ctx, T, [], [0], [("min", [("col", 1)])], keys, iv, None, 8192, ng)  # noqa: E731
    ctx.set_wait_limit(1)
    run()
    assert ctx.status() == tqp.ERR_TIMEOUT
    ctx.set_wait_limit(DEFAULT_WAIT)
    run()
    assert ctx.status() == 0
    want = oracle.run_plan(fact=cols, group_cols=[0], aggs=[("min", [("col", 1)])], want_pairs=False,
                           cap_groups=None, want_row_ids=False)
    g = int(ng.item())
    assert g == want["num_groups"] and np.array_equal(keys[:g].cpu().numpy(), want["keys"][:, 0])
    assert np.array_equal(iv[:g].cpu().numpy(), want["ivals"][:, 0])


def _topk_spec():
    d = datagen.dim_table(300_000, 200_000, seed=5)
    pr = datagen.probe_table(600_000, 300_000, seed=5)
    return dict(fact=[pr["fk"], pr["value"]], dim=[d["key"], d["payload"]], fact_fk=0, dim_key=0, group_cols=[3],
                aggs=[("sum", [("col", 1)]), ("count", None)], topk=40, topk_agg=0)


@pytest.mark.parametrize("batch", [False, True])
def test_topk_select(ctx, batch):
    import paper_2203_01877_gb300 as tqp
    spec = _topk_spec()
    want = oracle.run_plan(want_pairs=False, cap_groups=None, want_row_ids=False, **spec)
    plan, res, bufs, keep, shape = gpu_plan_prepare(**spec)
    ctx.set_wait_limit(1)
    if batch:
        b = tqp.tqp_batch_create(ctx, [plan], [res])
        tqp.tqp_batch_run(b)
        assert ctx.status() == tqp.ERR_TIMEOUT and int(bufs["num_groups"].item()) == -1
        tqp.tqp_batch_destroy(b)
        ctx.set_wait_limit(DEFAULT_WAIT)
        b = tqp.tqp_batch_create(ctx, [plan], [res])
        tqp.tqp_batch_run(b)
        assert ctx.status() == 0
        got = dict(gpu_plan_collect(bufs, shape), status=0)
        tqp.tqp_batch_destroy(b)
    else:
        tqp.tqp_run_plan(ctx, plan, res)
        assert int(bufs["num_groups"].item()) == -1
        ctx.set_wait_limit(DEFAULT_WAIT)
        tqp.tqp_run_plan(ctx, plan, res)  # (the time-out is still latched)
        got = dict(gpu_plan_collect(bufs, shape), status=0)
        assert ctx.status() == tqp.ERR_TIMEOUT and ctx.status() == 0
    compare(got, want, spec)
