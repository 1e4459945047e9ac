"""GPU: the shared scan's per-warp queue of passing rows against the oracle: queries that all rows, few rows and no row
pass (the queue filling in every step, across tiles and chunks, and left partly full), 3 to 32 queries, one and two sum
expressions and none, and row counts at the edges of a step and a tile."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
EXPRS = [[("col", 1), ("col", 2), "mul"], [("col", 2)]]


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 64 << 20)
    yield c
    c.close()


@pytest.mark.parametrize("n", [1, 127, 129, 1025, 8191, 400_003])
@pytest.mark.parametrize("nq", [3, 31, 32])
@pytest.mark.parametrize("share", [0, 1, 30, 1000])
@pytest.mark.parametrize("nexpr", [0, 1, 2])
def test_queue(ctx, n, nq, share, nexpr):
    import paper_2203_01877_gb300 as tqp
    from tests.gpu_util import up
    rng = np.random.default_rng(n + nq + share)
    cols = [rng.integers(0, 1000, n).astype(np.int32), rng.integers(-2**20, 2**20, n), rng.integers(0, 50, n).astype(np.int32)]
    cnt = torch.full((nq,), -7, dtype=torch.int64, device="cuda")
    tot = torch.full((nq,), -7, dtype=torch.int64, device="cuda")
    specs = []
    for i in range(nq):
        lo = int(rng.integers(0, 1001 - share))
        preds = [(0, "ge", lo), (0, "lt", lo + share)] + ([(2, "lt", 10 + i)] if i % 3 == 2 else [])
        specs.append((preds, EXPRS[i % nexpr] if nexpr else None))
    qs = [(p, e, cnt[i:i + 1], tot[i:i + 1] if e else None) for i, (p, e) in enumerate(specs)]
    tqp.tqp_filter_shared(ctx, tqp.TableRef([up(c) for c in cols]), qs)
    assert ctx.status() == 0
    for i, (p, e) in enumerate(specs):
        ids, s = oracle.filter_rows(cols, p, e)
        assert int(cnt[i]) == len(ids) and (e is None or int(tot[i]) == s), (i, p, e)
