"""GPU: the radix sort on both sides of the size where its passes leave the shared launch (3 * 2^20 items), through the
sort-based group-by (64-bit keys: eight passes) and the sort-based join (repeated build keys in canonical order)."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import up
from tests.test_gpu_groupby import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 1 << 30)
    c.set_variant(1)
    yield c
    c.close()


@pytest.mark.parametrize("n", [(3 << 20) - 1, 3 << 20, (3 << 20) + 1, (3 << 20) + 4097])
def test_group_by(ctx, n):
    rng = np.random.default_rng(n)
    pool = rng.integers(-2**62, 2**62, 700)
    cols = [pool[rng.integers(0, 700, n)], rng.integers(-1000, 1000, n)]
    check(ctx, cols, [(1, "gt", -900)], [0], [("sum", [("col", 1)]), ("count", None)], capacity=700)


@pytest.mark.parametrize("n", [3 << 20, (3 << 20) + 4097])
def test_join(ctx, n):
    import torch
    import paper_2203_01877_gb300 as tqp
    rng = np.random.default_rng(n)
    bk = (rng.integers(0, n // 3, n) * 331).astype(np.int32)
    pk = (rng.integers(0, n // 3, 50_000) * 331).astype(np.int32)
    wb, wp = oracle.join_pairs(bk, pk)
    cap = len(wb)
    ob, op = (torch.full((cap,), -9, dtype=torch.int32, device="cuda") for _ in range(2))
    cnt = torch.full((1,), -7, dtype=torch.int64, device="cuda")
    for variant in (1, 0):
        ctx.set_variant(variant)
        tqp.tqp_hash_join(ctx, tqp.TableRef([up(bk)]), 0, tqp.TableRef([up(pk)]), 0, ob, op, cap, cnt)
        ctx.set_variant(1)
        ctx.check()
        assert int(cnt.item()) == cap
        assert np.array_equal(ob.cpu().numpy(), wb) and np.array_equal(op.cpu().numpy(), wp)
