"""GPU: filters without a sum on both sides of the lines between the plain loads and the staged scan, by mix of
condition types and row count, against the oracle."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import gpu_filter

pytestmark = pytest.mark.gpu

# int64, int64, int32 x 3, uint8 x 2
D, W, U = [(0, "lt", 600), (1, "ge", 300)], [(2, "ge", 200), (3, "lt", 700), (4, "ne", 5)], [(5, "lt", 150), (6, "ge", 20)]
MIXES = {"2d": D, "2d u": D + U[:1], "2d w": D + W[:1], "d w": D[:1] + W[:1], "d 2w": D[:1] + W[:2], "d 3w": D[:1] + W,
         "d w u": D[:1] + W[:1] + U[:1], "d 2w u": D[:1] + W[:2] + U[:1], "d w 2u": D[:1] + W[:1] + U}
LINES = {5 << 20: MIXES, 1 << 25: ("d w", "d w 2u"), 1 << 26: ("d w", "d w u", "d 2w u")}


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 64 << 20)
    yield c
    c.close()


@pytest.mark.parametrize("line", LINES)
def test_both_sides(ctx, line):
    rng = np.random.default_rng(line)
    types = [np.int64] * 2 + [np.int32] * 3 + [np.uint8] * 2
    full = [rng.integers(0, 200 if t == np.uint8 else 1000, line, dtype=t) for t in types]
    for n in (line - 1, line):
        cols = [c[:n] for c in full]
        for mix in LINES[line]:
            preds = MIXES[mix]
            want, _ = oracle.filter_rows(cols, preds, None)
            ids, k, _, st = gpu_filter(ctx, cols, preds, None)
            assert st == 0 and k == len(want) and np.array_equal(ids, want), (n, mix)
            _, k, _, st = gpu_filter(ctx, cols, preds, None, want_ids=False)
            assert st == 0 and k == len(want), (n, mix)
