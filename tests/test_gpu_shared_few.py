"""GPU: shared scans of few queries whose steps of 128 rows pass about as many rows as the queue's line (64), and
over wide rows, where the row queues would cost a resident CTA and are left out."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import up

pytestmark = pytest.mark.gpu

SUMS = [[("col", 0)], [("col", 0), ("const", 7), ("col", 1), "sub", "mul"]]


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 64 << 20)
    yield c
    c.close()


def _run(ctx, cols, queries):
    import torch
    import paper_2203_01877_gb300 as tqp
    T = tqp.TableRef([up(c) for c in cols])
    outs = [(torch.full((1,), -7, dtype=torch.int64, device="cuda"),
             torch.full((1,), -7, dtype=torch.int64, device="cuda")) for _ in queries]
    assert tqp.tqp_filter_shared(ctx, T, [(p, e, c, s) for (p, e), (c, s) in zip(queries, outs)]) == [0] * len(queries)
    ctx.check()
    for (p, e), (c, s) in zip(queries, outs):
        ids, total = oracle.filter_rows(cols, p, e)
        assert int(c.item()) == len(ids) and int(s.item()) == total, (p, e)


@pytest.mark.parametrize("n", [127, 1024, 1025, 70_003])
@pytest.mark.parametrize("nq", [3, 8])
@pytest.mark.parametrize("nexpr", [1, 2])
@pytest.mark.parametrize("percent", [25, 45, 50, 55])
def test_about_half_a_step(ctx, n, nq, nexpr, percent):
    rng = np.random.default_rng(n + nq + percent)
    cols = [rng.integers(-2**30, 2**30, n), rng.integers(0, 1000, n).astype(np.int32)]
    w = 10 * percent // nq
    _run(ctx, cols, [([(1, "between", q * w, q * w + w - 1)], SUMS[q % nexpr]) for q in range(nq)])


@pytest.mark.parametrize("n", [1, 1023, 1025, 400_003])
@pytest.mark.parametrize("span", [1, 40, 150])
@pytest.mark.parametrize("nexpr", [1, 2])
def test_six_wide_columns(ctx, n, span, nexpr):
    rng = np.random.default_rng(n + span)
    cols = [rng.integers(0, 300, n) for _ in range(6)]
    queries = [([(q, "between", q * span, q * span + span - 1), (q + 3, "lt", 200)], SUMS[q % nexpr]) for q in range(3)]
    _run(ctx, cols, queries + [([(c, "lt", 250) for c in range(6)], SUMS[0])])
