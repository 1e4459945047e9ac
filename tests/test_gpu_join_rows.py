"""GPU: the pair-output join at the sizes where a lane's rows change (1, 4 and 16), at the edges of each form's tiles,
with runs much longer than a tile's rows, and with capacities that end before, inside and behind such a run."""
import numpy as np
import pytest

from tests.test_gpu_join_pairs import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 256 << 20)
    yield c
    c.close()


def _sizes():
    one = 2 * 152 * 512  # rows that two blocks per SM take at one per lane
    return [512, 513, one, one + 1, one + 2049, 4 * one, 4 * one + 1, 4 * one + 8193]


@pytest.mark.parametrize("n", _sizes())
@pytest.mark.parametrize("kind", ["inner", "semi", "anti", "left_outer"])
@pytest.mark.parametrize("bt,dup", [(np.int32, 1), (np.int32, 3), (np.int64, 1), (np.int64, 3)])
def test_sizes(ctx, n, kind, bt, dup):
    rng = np.random.default_rng(n + dup)
    bk = (rng.permutation(3000) // dup * 1_000_003 % 2**31).astype(bt)
    pk = (rng.integers(0, 4000 // dup, n) * 1_000_003 % 2**31).astype((np.int32, np.int64)[n % 2])
    check(ctx, bk, pk, kind)


@pytest.mark.parametrize("n", [200, 3000, 160_000])
@pytest.mark.parametrize("short", [0, 1, 20_000, 39_999, 10**9])
def test_long_runs(ctx, n, short):
    rng = np.random.default_rng(n)
    bk = np.concatenate([np.full(20_000, 7), np.arange(100, 1100), np.full(33, -5)]).astype(np.int32)
    rng.shuffle(bk)
    pk = rng.integers(100, 1100, n).astype(np.int32)
    pk[rng.integers(0, n, 3)] = 7
    pk[n - 1] = 7
    pk[rng.integers(0, n - 1, n // 10)] = -5
    check(ctx, bk, pk, "inner", short)
