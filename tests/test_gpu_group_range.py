"""GPU: the group-by over key ranges (more than 64 groups) against the oracle, at the edges of its 128-row warp steps
and 4096-entry output blocks, for ranges at and just past what its entries hold (the hash path then answers), tables in
shared memory and in L2, every number of sums, hot keys, key types, signs and predicates."""
import numpy as np
import pytest

from tests.test_gpu_groupby import check, gpu_groupby

pytestmark = pytest.mark.gpu

SUMS = {0: [("count", None)], 1: [("sum", [("col", 2)]), ("count", None), ("avg", [("col", 2)])],
        2: [("sum", [("col", 2)]), ("sum", [("col", 2), ("const", 100), ("col", 3), "sub", "mul"])],
        3: [("sum", [("col", 3)]), ("avg", [("col", 2)]), ("sum", [("col", 2), ("col", 3), "mul"]), ("count", None)]}


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 512 << 20)
    yield c
    c.close()


def table(n, groups, seed, first, dtype=np.int32, hot=0.0):
    rng = np.random.default_rng(seed)
    key = rng.integers(0, groups, n)
    key[:2] = [0, groups - 1][:n]
    if hot:
        key = np.where(rng.random(n) < hot, groups // 3, key)
        key = np.where(rng.random(n) < hot / 2, groups // 2, key)
    return [(key + first).astype(dtype), rng.integers(0, 9, n).astype(np.uint8),
            rng.integers(-2**54, 2**54, n) // n, rng.integers(-50, 50, n).astype(np.int32)]


@pytest.mark.parametrize("n", [1, 127, 129, 3073, 70_003])
@pytest.mark.parametrize("nsum", [0, 1, 2, 3])
@pytest.mark.parametrize("groups,capacity", [(70, 70), (4096, 4100), (4097, 8192), (60_001, 60_001)])
def test_sizes(ctx, n, nsum, groups, capacity):
    cols = table(n, groups, n + nsum, -groups // 2, (np.int32, np.int64)[n % 2])
    check(ctx, cols, [(1, "lt", 7), (3, "ne", 4)] if nsum % 2 else [], [0], SUMS[nsum], capacity=capacity)


@pytest.mark.parametrize("extra", [0, 1, 2])
def test_range_at_the_entries(ctx, extra):
    """300 groups have a table of 1024 + 1 entries: ranges of 1024, 1025 and (hashed) 1026 keys."""
    cols = table(50_000, 300, 3, 0)
    cols[0][7] = 1023 + extra
    check(ctx, cols, [], [0], SUMS[1], capacity=301)


@pytest.mark.parametrize("first,dtype", [(2**31 - 2000, np.int32), (-2**31, np.int32), (2**63 - 2000, np.int64),
                                         (-2**63, np.int64), (-1000, np.int64)])
@pytest.mark.parametrize("n", [20_000, 600_000])
def test_extreme_keys(ctx, first, dtype, n):
    rng = np.random.default_rng(n)
    key = (rng.integers(0, 2000, n).astype(np.int64) + np.int64(first)).astype(dtype)
    val = rng.integers(-2**62, 2**62, n) // n
    check(ctx, [key, val], [], [0], [("sum", [("col", 1)]), ("count", None)], capacity=2000)
    key[5] = np.iinfo(dtype).min if first > 0 else np.iinfo(dtype).max  # the widest range: hashed
    check(ctx, [key, val], [], [0], [("sum", [("col", 1)]), ("count", None)], capacity=2001)


@pytest.mark.parametrize("groups", [1500, 200_000])
@pytest.mark.parametrize("hot", [0.05, 0.4, 0.95])
def test_hot_keys(ctx, groups, hot):
    cols = table(900_001, groups, 5, 17, hot=hot)
    for nsum in (1, 3):
        check(ctx, cols, [(1, "le", 6)], [0], SUMS[nsum], capacity=groups)


def test_several_keys(ctx):
    rng = np.random.default_rng(2)
    n = 300_007
    a, b = rng.integers(-30, 30, n).astype(np.int32), rng.integers(3, 250, n).astype(np.uint8)
    c, v = rng.integers(2**31 - 4, 2**31 - 1, n).astype(np.int32), rng.integers(0, 10**7, n)
    aggs = [("sum", [("col", 3)]), ("count", None)]
    check(ctx, [a, b, b, v], [], [0, 1], aggs, capacity=60 * 247)
    check(ctx, [a, b, c, v], [(3, "lt", 9_000_000)], [1, 2], aggs, capacity=3 * 247)
    check(ctx, [b, b, b, v], [], [0, 1, 2], aggs, capacity=300)  # the product of the ranges is past the entries
    check(ctx, [a, b, c, v], [(3, "lt", -1)], [1, 2], aggs, capacity=3 * 247)  # no row passes


def test_capacity_exceeded(ctx):
    import paper_2203_01877_gb300 as tqp
    key = np.arange(100, dtype=np.int32)
    st, g, *_ = gpu_groupby(ctx, [key], [], [0], [("count", None)], capacity=99)
    assert st == tqp.ERR_CAPACITY and g == -1
    check(ctx, [key], [], [0], [("count", None)], capacity=100)
