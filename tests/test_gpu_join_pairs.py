"""GPU: the one-pass pair-output join against the oracle, at the edges of its 8192-row tiles and of the 128 tiles its
look-back reads at a time, for every join kind, table form (indexed by key, buckets, 64-bit slots), mix of key types,
full buckets, repeated keys (runs that straddle a warp's rounds, one key for every row) and capacities."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
KINDS = ["inner", "semi", "anti", "left_outer"]


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 256 << 20)
    yield c
    c.close()


def check(ctx, bk, pk, kind, short=0):
    import torch
    import paper_2203_01877_gb300 as tqp
    from tests.gpu_util import up
    wb, wp = oracle.join_pairs(bk, pk, join_kind=kind)
    cap = max(len(wb) - short, 0)
    ob = torch.full((cap + 4,), -7, dtype=torch.int32, device="cuda")
    op = torch.full((cap + 4,), -7, dtype=torch.int32, device="cuda")
    cnt = torch.full((1,), -7, dtype=torch.int64, device="cuda")
    tqp.tqp_hash_join_kind(ctx, tqp.TableRef([up(bk)]), 0, tqp.TableRef([up(pk)]), 0, kind, ob, op, cap, cnt)
    assert ctx.status() == (tqp.ERR_CAPACITY if short else 0)
    assert int(cnt.item()) == len(wb)
    assert np.array_equal(ob[:cap].cpu().numpy(), wb[:cap]) and np.array_equal(op[:cap].cpu().numpy(), wp[:cap])
    assert bool((ob[cap:] == -7).all()) and bool((op[cap:] == -7).all())  # nothing past the capacity
    return len(wb)


@pytest.mark.parametrize("n", [1, 31, 33, 511, 8191, 8192, 8193, 128 * 8192 + 1])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("spread,dup", [(1, 1), (1_000_003, 1), (1, 3), (1_000_003, 3)])
def test_sizes(ctx, n, kind, spread, dup):
    rng = np.random.default_rng(n + dup)
    bk = (rng.permutation(900) // dup * spread).astype(np.int32)
    pk = (rng.integers(0, 1200 // dup, n) * spread).astype(np.int32)
    check(ctx, bk, pk, kind)


@pytest.mark.parametrize("bt", [np.uint8, np.int32, np.int64])
@pytest.mark.parametrize("pt", [np.uint8, np.int32, np.int64])
@pytest.mark.parametrize("kind", KINDS)
def test_key_types(ctx, bt, pt, kind):
    def keys(dt, n, seed):
        i = np.iinfo(dt)
        special = [i.min, i.max, 0, 255, 256, -1, 2**31 - 1, -2**31, 2**32 - 1, 2**32 + 5, 5]
        pool = np.array([s for s in special if i.min <= s <= i.max], dtype=dt)
        return pool[np.random.default_rng(seed).integers(0, len(pool), n)]
    check(ctx, keys(bt, 40, 1), keys(pt, 9001, 2), kind)
    check(ctx, np.unique(keys(bt, 40, 3)), keys(pt, 9001, 4), kind)


@pytest.mark.parametrize("kind", ["inner", "left_outer"])
def test_full_buckets(ctx, kind):
    """60,000 scattered keys in 131,072 slots: about one bucket in six overflows into the next."""
    rng = np.random.default_rng(3)
    bk = rng.choice(2**31 - 1, 60_000, replace=False).astype(np.int32)
    pk = np.where(rng.random(200_000) < 0.6, bk[rng.integers(0, len(bk), 200_000)],
                  rng.integers(-2**31, 2**31 - 1, 200_000)).astype(np.int32)
    check(ctx, bk, pk, kind)


@pytest.mark.parametrize("kind", ["inner", "left_outer", "semi"])
def test_runs(ctx, kind):
    rng = np.random.default_rng(4)
    bk = np.repeat(np.array([5, 10**9, -3, 77], np.int32), [1, 33, 400, 2])
    rng.shuffle(bk)
    check(ctx, bk, rng.choice(np.array([5, 10**9, -3, 77, 6], np.int32), 9000), kind)
    check(ctx, np.full(700, 9, np.int32), np.full(8193, 9, np.int32), kind)


@pytest.mark.parametrize("short", [1, 100, 9000])
def test_capacity(ctx, short):
    rng = np.random.default_rng(5)
    check(ctx, rng.permutation(5000).astype(np.int32), rng.integers(0, 5000, 20_000).astype(np.int32), "inner", short)
    check(ctx, np.arange(5000, dtype=np.int32) // 2, rng.integers(0, 2500, 20_000).astype(np.int32), "inner", short)
