"""GPU: the one-launch radix sort behind group-by output, join runs and the sort-based forms: item counts at the edges of
its 4096-item tiles and past one tile per resident block, one to eight 8-bit passes, and inputs it finds empty."""
import numpy as np
import pytest

from tests.test_gpu_groupby import check as check_groupby
from tests.test_gpu_join_pairs import check as check_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 2 << 30)
    yield c
    c.close()


@pytest.mark.parametrize("n", [1, 4095, 4096, 4097, 70_001, 3_000_001])
@pytest.mark.parametrize("dtype,spread", [(np.int32, 2**31), (np.int64, 2**62)])
def test_group_keys_in_order(ctx, n, dtype, spread):
    """Scattered keys, nearly all distinct: as many groups to sort as rows, over 32 and 64 bits."""
    key = np.random.default_rng(n).integers(-spread, spread, n).astype(dtype)
    check_groupby(ctx, [key, np.arange(n, dtype=np.int64)], [], [0], [("sum", [("col", 1)])], capacity=max(n, 5000))


def test_no_passing_row(ctx):
    key = np.random.default_rng(1).integers(-2**31, 2**31, 50_000).astype(np.int32)
    check_groupby(ctx, [key], [(0, "gt", 2**40)], [0], [("count", None)], capacity=50_000)


@pytest.mark.parametrize("nb", [2, 4096, 4098, 700_001])
def test_runs_of_repeated_keys(ctx, nb):
    rng = np.random.default_rng(nb)
    bk = (rng.integers(0, max(1, nb // 3), nb) * 1_000_003 % 2**31).astype(np.int32)
    check_pairs(ctx, bk, bk[rng.integers(0, nb, 20_000)], "inner")
