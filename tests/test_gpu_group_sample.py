"""GPU: the group-by over key ranges where the sample of 256 rows and the whole range pass disagree, with tables on
both sides of the sizes that are cleared before the range is known and that have a kernel of their own in L2."""
import numpy as np
import pytest

from tests.test_gpu_groupby import check, gpu_groupby

pytestmark = pytest.mark.gpu

AGGS = [("sum", [("col", 1)]), ("count", None)]


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 1 << 30)
    yield c
    c.close()


@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 20_000, 300_001])
@pytest.mark.parametrize("where", ["none", "sampled", "unsampled", "last", "filtered"])
@pytest.mark.parametrize("groups", [90, 3000, 60_000])
def test_one_outlier(ctx, n, where, groups):
    rng = np.random.default_rng(n + groups)
    cols = [rng.integers(0, groups, n).astype(np.int32), rng.integers(-10**9, 10**9, n),
            rng.integers(0, 9, n).astype(np.uint8)]
    row = {"none": None, "sampled": n * 17 // 256 if n > 256 else 0, "unsampled": min(n - 1, 1), "last": n - 1,
           "filtered": n // 2}[where]
    if row is not None:
        cols[0][row] = 2**31 - 1
        cols[2][row] = 8 if where == "filtered" else 0
    check(ctx, cols, [(2, "lt", 8)], [0], AGGS, capacity=groups + 1)


@pytest.mark.parametrize("groups", [5_000, 70_000])
@pytest.mark.parametrize("scattered", [False, True])
def test_many_rows(ctx, groups, scattered):
    n = (1 << 23) + 70_001
    rng = np.random.default_rng(groups)
    pool = rng.permutation(2**20)[:groups] * (2003 if scattered else 1) if scattered else np.arange(groups)
    cols = [pool[rng.integers(0, groups, n)].astype(np.int32), rng.integers(-10**9, 10**9, n)]
    check(ctx, cols, [], [0], AGGS, capacity=groups)


def test_capacity_exceeded(ctx):
    import paper_2203_01877_gb300 as tqp
    key = np.arange(10_000, dtype=np.int32)
    st, g, *_ = gpu_groupby(ctx, [key], [], [0], [("count", None)], capacity=9_999)
    assert st == tqp.ERR_CAPACITY and g == -1
    check(ctx, [key], [], [0], [("count", None)], capacity=10_000)
