"""GPU: calls in the smallest arena they have been accepted in (bytes measured before the plain-load forms, whose
padded key entries, wider range passes and block maps must not raise it), with the results of a large one."""
import numpy as np
import pytest

from tests.plan_util import gpu_plan_collect, gpu_plan_prepare

pytestmark = pytest.mark.gpu

SUM, SUM2, COUNT = ("sum", [("col", 1)]), ("sum", [("col", 2)]), ("count", None)


def _join(nf, nd, ng, topk):
    rng = np.random.default_rng(nd)
    return dict(fact=[rng.integers(0, nd, nf).astype(np.int32), rng.integers(0, 1000, nf),
                      rng.integers(0, 100, nf).astype(np.int32)],
                dim=[np.arange(nd, dtype=np.int32), rng.integers(0, ng, nd).astype(np.int32)], fact_fk=0, dim_key=0,
                group_cols=[4], aggs=[SUM, SUM2, COUNT], topk=topk, topk_agg=0, capacity_groups=topk)


def _scan(n, group_cols, cap, topk):
    rng = np.random.default_rng(n)
    return dict(fact=[rng.integers(0, 1000, n).astype(np.int32), rng.integers(0, 1000, n),
                      rng.integers(0, 4, n).astype(np.uint8), rng.integers(0, 3, n).astype(np.uint8)],
                preds=[(0, "lt", 500)], group_cols=group_cols, aggs=[SUM, COUNT], topk=topk, topk_agg=0,
                capacity_groups=topk or cap, max_groups=cap)


CASES = {  # spec, bytes of: one plan, run_plans, a batch
    "key entries of three words": (_join(200_000, 50_000, 20_000, 10), 5940736, 9095616, 9095616),
    "the same, few rows": (_join(1000, 100, 10, 10), 79424, 87360, 87488),
    "few groups, top-k": (_scan(10_000_000, [2, 3], 16, 10), 72256, 74816, 74944),
    "many groups": (_scan(1000, [0, 2], 20_000, 0), 3168512, 3170048, 3169984),
}


@pytest.mark.parametrize("how", ["plan", "plans", "batch"])
@pytest.mark.parametrize("name", CASES)
def test_accepted_in_the_smallest_arena(name, how):
    import paper_2203_01877_gb300 as tqp
    spec, *need = CASES[name]
    need = need[("plan", "plans", "batch").index(how)]
    plan, res, bufs, keep, shape = gpu_plan_prepare(**spec)
    got = []
    for arena in (1 << 28, need):
        for v in bufs.values():
            if v is not None:
                v.fill_(-7)
        ctx = tqp.Context(0, arena)
        try:
            if how == "plan":
                tqp.tqp_run_plan(ctx, plan, res)
            elif how == "plans":
                tqp.tqp_run_plans(ctx, [plan], [res])
            else:
                b = tqp.tqp_batch_create(ctx, [plan], [res])
                tqp.tqp_batch_run(b)
                ctx.check()
                tqp.tqp_batch_destroy(b)
            ctx.check()
            got.append(gpu_plan_collect(bufs, shape))
        finally:
            ctx.close()
    for k in got[0]:
        assert np.array_equal(np.asarray(got[0][k]), np.asarray(got[1][k])), k
