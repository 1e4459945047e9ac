"""GPU: the plain-load filter scan (built-in for one to four conditions) against the oracle: row counts at the edges of
its 128-row warp steps, 1024-row segments and 65536-row mask blocks, every column type, 64-bit columns on 16- and
32-byte boundaries, selectivities on both sides of its queue, and every form of the sum."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import gpu_filter, up, zeros

pytestmark = pytest.mark.gpu

SUMS = [None, [("col", 3)], [("col", 3), ("col", 1), "mul"], [("col", 2), ("const", 100), ("col", 0), "sub", "mul"],
        [("const", 7)], [("col", 0), ("const", -3), "mul", ("const", 5), "add"]]
PREDS = [[(0, "lt", 20)], [(0, "ge", 2), (1, "ne", 3)], [(0, "lt", 90), (1, "lt", 250), (2, "ge", -2**33)],
         [(0, "between", 1, 98), (0, "ne", 50), (2, "lt", 2**33), (3, "gt", -10**6)], [(2, "eq", 1 << 60)]]


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 64 << 20)
    yield c
    c.close()


def columns(n, seed):
    rng = np.random.default_rng(seed)
    return [rng.integers(0, 100, n).astype(np.int32), rng.integers(0, 256, n).astype(np.uint8),
            rng.integers(-2**34, 2**34, n), rng.integers(-10**6, 10**6, n).astype(np.int32)]


@pytest.mark.parametrize("n", [1, 5, 127, 128, 129, 1023, 1025, 8193, 65535, 65537, 300_003])
@pytest.mark.parametrize("preds", range(len(PREDS)))
def test_sizes(ctx, n, preds):
    cols = columns(n, n + preds)
    for e in SUMS:
        for ids in (True, False):
            want, wsum = oracle.filter_rows(cols, PREDS[preds], e)
            got, k, s, st = gpu_filter(ctx, cols, PREDS[preds], e, want_ids=ids)
            assert st == 0 and k == len(want)
            assert e is None or s == wsum
            assert not ids or np.array_equal(got, want)


@pytest.mark.parametrize("share", [1, 24, 26, 60, 99])
def test_selectivity(ctx, share):
    cols = columns(200_001, share)
    want, wsum = oracle.filter_rows(cols, [(0, "lt", share)], SUMS[3])
    got, k, s, st = gpu_filter(ctx, cols, [(0, "lt", share)], SUMS[3])
    assert st == 0 and k == len(want) and s == wsum and np.array_equal(got, want)


def test_int64_on_a_16_byte_boundary(ctx):
    import torch
    import paper_2203_01877_gb300 as tqp
    n = 70_001
    cols = columns(n, 3)
    dev = [up(c) for c in cols]
    buf = torch.zeros(n + 2, dtype=torch.int64, device="cuda")
    buf[2:] = dev[2]
    dev[2] = buf[2:]
    assert dev[2].data_ptr() % 32 == 16
    preds, e = PREDS[2], SUMS[3]
    ids, cnt, s = zeros(n, torch.int32), zeros(1, torch.int64), zeros(1, torch.int64)
    tqp.tqp_filter(ctx, tqp.TableRef(dev), preds, e, s, ids, n, cnt)
    want, wsum = oracle.filter_rows(cols, preds, e)
    assert ctx.status() == 0 and int(cnt.item()) == len(want) and int(s.item()) == wsum
    assert np.array_equal(ids[:len(want)].cpu().numpy(), want)


def test_capacity(ctx):
    import paper_2203_01877_gb300 as tqp
    cols = columns(100_000, 4)
    want, _ = oracle.filter_rows(cols, [(0, "lt", 90)], None)
    got, k, _, st = gpu_filter(ctx, cols, [(0, "lt", 90)], capacity=5000)
    assert st == tqp.ERR_CAPACITY and k == len(want) and np.array_equal(got, want[:5000])
