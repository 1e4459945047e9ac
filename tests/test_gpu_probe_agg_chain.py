"""GPU: the probe of joined aggregations where every fact row matches many build rows of one group, so that one
block adds far more joined rows to a group than it reads fact rows. Expected values in closed form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# 1024 fact rows (one block), times 2^22 build rows: 2^32 joined rows in one group; 3 more build rows: past it
@pytest.mark.parametrize("n,m", [(1024, 1 << 12), (1024, 1 << 22), (1021, (1 << 22) + 16_003)])
def test_group_count_past_32_bits(n, m):
    import torch
    import paper_2203_01877_gb300 as tqp
    rng = np.random.default_rng(n)
    value = rng.integers(-10**12, 10**12, n)
    F = tqp.TableRef([torch.full((n,), 7, dtype=torch.int32, device="cuda"), torch.from_numpy(value).cuda()])
    D = tqp.TableRef([torch.full((m,), 7, dtype=torch.int32, device="cuda"),
                      torch.full((m,), 3, dtype=torch.int32, device="cuda")])
    z = lambda k: torch.full((k,), -7, dtype=torch.int64, device="cuda")  # noqa: E731
    keys, iv, ng, tot, joined = z(4), z(8), z(1), z(1), z(1)
    ctx = tqp.Context(0, 512 << 20)
    try:
        plan = tqp.make_plan(F, (), D, 0, 0, [3], [("count", None), ("sum", [("col", 1)])], max_groups=4)
        res = tqp.make_result(None, 0, None, None, keys, iv, None, 4, ng, tot, joined)
        tqp.tqp_run_plan(ctx, plan, res)
        ctx.check()
    finally:
        ctx.close()
    assert int(joined.item()) == n * m
    assert int(ng.item()) == 1 and int(keys[0].item()) == 3
    assert int(iv[0].item()) == n * m
    want = int(value.sum()) * m
    assert int(iv[1].item()) == (want + 2**63) % 2**64 - 2**63  # (sums wrap modulo 2^64)
