"""GPU: IN lists on both sides of the row counts (2^19 and 3 * 2^19) that decide which lists are compared value by
value, against numpy."""
import numpy as np
import pytest

from tests.gpu_util import gpu_filter

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 64 << 20)
    yield c
    c.close()


def _check(ctx, col, values, want):
    ids, k, _, st = gpu_filter(ctx, [col], [(0, "in", values)])
    assert st == 0 and k == len(want) and np.array_equal(ids, want)


@pytest.mark.parametrize("n", [1000, (1 << 19) - 1, 1 << 19, 3 * (1 << 19) - 1, 3 * (1 << 19)])
@pytest.mark.parametrize("count", [4, 10, 11, 32, 33])
def test_lists(ctx, n, count):
    rng = np.random.default_rng(n + count)
    which = rng.integers(0, 80, n)
    for width in (8, 11, 24, 27):
        words = np.zeros((80, width), np.uint8)
        for i in range(80):  # distinct: the number in two letters, then letters up to a length
            words[i, :2] = 97 + i // 26, 97 + i % 26
            words[i, 2:rng.integers(2, width + 1)] = 100 + i % 3
        _check(ctx, words[which], [bytes(w).rstrip(b"\0") for w in words[:count]], np.flatnonzero(which < count))
    for dtype in (np.int32, np.int64):
        _check(ctx, which.astype(dtype), list(range(count)), np.flatnonzero(which < count))
