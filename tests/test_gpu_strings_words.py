"""GPU: LIKE, NOT LIKE and IN on strings of at most 32 bytes (words in registers) against the oracle: every way a width
splits into words, patterns at the chunk and width edges, matches that would run past the string's end, bytes after its
first zero, and values at the edges of the short list (longer lists and wider strings take the byte-wise form)."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import gpu_filter

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 64 << 20)
    yield c
    c.close()


def strings(n, width, seed, garbage=False):
    rng = np.random.default_rng(seed)
    x = rng.integers(97, 100, (n, width)).astype(np.uint8)  # a, b, c: repeats and near matches
    ln = rng.integers(0, width + 1, n)
    x[np.arange(width)[None, :] >= ln[:, None]] = 0
    if garbage:  # bytes after the first zero are not part of the string
        tail = np.arange(width)[None, :] > ln[:, None]
        x[tail] = rng.integers(97, 100, int(tail.sum()))
    return x


def check(ctx, x, op, arg):
    cols = [x, np.arange(len(x), dtype=np.int64)]
    preds = [(0, op, arg)]
    want, wsum = oracle.filter_rows(cols, preds, [("col", 1)])
    ids, k, s, st = gpu_filter(ctx, cols, preds, [("col", 1)])
    assert st == 0 and k == len(want) and s == wsum and np.array_equal(ids, want), (op, arg, x.shape)


@pytest.mark.parametrize("width", [1, 3, 4, 5, 7, 8, 12, 15, 16, 20, 23, 24, 27, 28, 31, 32, 33])
@pytest.mark.parametrize("n", [1, 31, 2051])
def test_like(ctx, width, n):
    x = strings(n, width, width + n, garbage=n > 100)
    full = bytes(x[0][:max(1, int(np.argmax(x[0] == 0)) if (x[0] == 0).any() else width)]).replace(b"\0", b"a").decode()
    for p in ("%ab%", "ab%", "%ab", "a%b", "%a_c%", "%", "%%", "", "_", "%_%", "%abca%", "%abcab%", "ab%ca%b", "%a%b%c%",
              "%abc%abc%", "_b%_", full, full + "%", "%" + full, "%" + full + "%", "_" * width, "_" * width + "%",
              "%" + "_" * width, "a" * (width + 1), "%" + "a" * (width + 1), "%a%a%a%a%a%a%a%a%", "%a%a%a%a%a%a%a%a%a%"):
        check(ctx, x, "like", p)
        check(ctx, x, "not_like", p)


@pytest.mark.parametrize("width", [1, 4, 6, 8, 24, 27, 32])
@pytest.mark.parametrize("count", [0, 1, 32, 33])
def test_in(ctx, width, count):
    x = strings(3001, width, width)
    pick = [bytes(r).rstrip(b"\0").decode() for r in x[:count]]
    check(ctx, x, "in", pick)


@pytest.mark.parametrize("count", [1, 32, 33])
def test_in_numbers_with_like(ctx, count):
    rng = np.random.default_rng(count)
    x, v = strings(5003, 24, 9), rng.integers(-60, 60, 5003).astype(np.int32)
    cols = [x, v]
    preds = [(0, "like", "%ab%"), (1, "in", [int(i) - count // 2 for i in range(count)])]
    want, _ = oracle.filter_rows(cols, preds, None)
    ids, k, _, st = gpu_filter(ctx, cols, preds)
    assert st == 0 and np.array_equal(ids, want)
