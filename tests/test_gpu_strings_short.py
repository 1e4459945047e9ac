"""GPU: LIKE segments of one and two bytes (found byte by byte: bytes on both sides of 0x80, neighbours that differ in
one bit, `_` beside a literal) and IN lists on both sides of the length that is compared value by value, for every way
a width splits into words."""
import numpy as np
import pytest

from tests.test_gpu_strings_words import check, ctx  # noqa: F401

pytestmark = pytest.mark.gpu
WIDTHS = [1, 2, 3, 4, 7, 8, 12, 13, 16, 20, 21, 24, 25, 28, 31, 32]


@pytest.mark.parametrize("width", WIDTHS)
@pytest.mark.parametrize("pool", [b"ab", b"\x01\x80\x81\xff\x7f", b"`abA\xe1"])
def test_short_segments(ctx, width, pool):  # noqa: F811
    rng = np.random.default_rng(width)
    x = np.frombuffer(pool, np.uint8)[rng.integers(0, len(pool), (1500, width))].copy()
    ln = rng.integers(0, width + 1, len(x))
    x[np.arange(width)[None, :] >= ln[:, None]] = 0
    x[::7, width // 2:] = rng.integers(0, 3, (len(x[::7]), width - width // 2))  # bytes behind the first zero
    a, b, c = pool[:1], pool[1:2], pool[-1:]
    for p in (b"%" + a + b"%", b"%" + b + b"%", b"%" + a + b + b"%", b"%" + c + c + b"%", b"%_" + b + b"%",
              b"%" + c + b"_%", b"%__%", a + b"%" + b + b"%" + c, b"%" + a + b"%" + b + a + b"%" + c + b"%",
              b"%" + b + b"%" + b + b"%" + b + b"%" + a, a + b"%" + b"_" + b + b"%" + c + b"_%"):
        check(ctx, x, "like", p)
        check(ctx, x, "not_like", p)


@pytest.mark.parametrize("width", WIDTHS)
@pytest.mark.parametrize("count", [4, 5, 6, 7, 8, 9, 10, 11, 14, 15, 16, 17, 31, 33])
def test_in_lists(ctx, width, count):  # noqa: F811
    rng = np.random.default_rng(width + count)
    x = rng.integers(97, 101, (2003, width)).astype(np.uint8)
    x[np.arange(width)[None, :] >= rng.integers(0, width + 1, len(x))[:, None]] = 0
    check(ctx, x, "in", [bytes(r).rstrip(b"\0") for r in x[:count]])


@pytest.mark.parametrize("count", [9, 10, 11, 33])
@pytest.mark.parametrize("dtype", [np.uint8, np.int32, np.int64])
def test_number_lists(ctx, count, dtype):  # noqa: F811
    import oracle
    from tests.gpu_util import gpu_filter
    rng = np.random.default_rng(count)
    cols = [rng.integers(0, 120, 5003).astype(dtype)]
    preds = [(0, "in", [int(v) for v in rng.permutation(140)[:count]])]
    want, _ = oracle.filter_rows(cols, preds, None)
    ids, k, _, st = gpu_filter(ctx, cols, preds)
    assert st == 0 and k == len(want) and np.array_equal(ids, want)
