"""GPU: the plain-load filter with two and four steps per warp and a ragged end, and the shapes and sizes on both sides
of its line with the staged scan (2^23 rows, no sum), against the oracle; the smallest arena it took serves both."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import gpu_filter

pytestmark = pytest.mark.gpu

# int64, int64, int32, int32, uint8
SHAPES = {"two wide": [(0, "lt", 300), (1, "ge", 500)], "wide and two words": [(0, "lt", 600), (2, "ge", 200), (3, "lt", 700)],
          "wide, word, byte": [(0, "lt", 600), (2, "ge", 200), (4, "lt", 150)], "one wide": [(0, "lt", 30)],
          "two words": [(2, "ge", 200), (3, "ne", 700)]}


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 64 << 20)
    yield c
    c.close()


def _cols(n):
    rng = np.random.default_rng(n)
    return [rng.integers(0, 1000, n), rng.integers(0, 1000, n), rng.integers(0, 1000, n).astype(np.int32),
            rng.integers(0, 1000, n).astype(np.int32), rng.integers(0, 200, n).astype(np.uint8)]


def _check(ctx, cols, preds, ex):
    want, wsum = oracle.filter_rows(cols, preds, ex)
    ids, k, s, st = gpu_filter(ctx, cols, preds, ex)
    assert st == 0 and k == len(want) and np.array_equal(ids, want) and (ex is None or s == wsum)
    _, k, s, st = gpu_filter(ctx, cols, preds, ex, want_ids=False)
    assert st == 0 and k == len(want) and (ex is None or s == wsum)


@pytest.mark.parametrize("n", [1_300_001, 2_490_368, 2_490_369, 2_600_511, (1 << 23) - 1, 1 << 23])
@pytest.mark.parametrize("shape", SHAPES)
def test_sizes(ctx, n, shape):
    cols = _cols(n)
    for ex in (None, [("col", 1)]) if n < 4_000_000 else (None,):
        _check(ctx, cols, SHAPES[shape], ex)


def test_smallest_arena():
    import paper_2203_01877_gb300 as tqp
    n = (1 << 23) + 130
    cols = _cols(n)
    # counters and block totals (129 of 65,536 rows), then one mask bit per row of whole 128-row steps
    need = 256 + (32 + 129 * 4 + 255) // 256 * 256 + (n + 127) // 128 * 16
    ctx = tqp.Context(0, need)
    try:
        _check(ctx, cols, SHAPES["two wide"], None)
    finally:
        ctx.close()
