"""GPU: the plain-load probe of joined aggregations (variant 1 without a launch-shape override) against the
oracle, at the edges of its 128-row warp steps and 1024-row blocks, for every entry width (one to four words),
key type, table form (direct-mapped, hashed, several build rows per key) and predicates."""
import numpy as np
import pytest

import oracle
from tests.plan_util import compare, gpu_plan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2203_01877_gb300 as tqp
    c = tqp.Context(0, 256 << 20)
    yield c
    c.close()


AGGS = {0: [("count", None)], 1: [("sum", [("col", 1)]), ("count", None)],
        2: [("sum", [("col", 1)]), ("sum", [("col", 1), ("const", 100), ("col", 2), "sub", "mul"]), ("count", None)]}


@pytest.mark.parametrize("n", [1, 127, 128, 129, 1023, 1025, 70_003])
@pytest.mark.parametrize("nsum,total", [(0, False), (0, True), (1, False), (1, True), (2, False), (2, True)])
@pytest.mark.parametrize("table", ["dense", "hashed", "dup_dense", "dup_hashed"])
def test_probe_agg_matches_oracle(ctx, n, nsum, total, table):
    rng = np.random.default_rng(n * 31 + nsum * 7 + total + len(table))
    nb = 300
    idx = np.arange(nb) // (3 if table.startswith("dup") else 1)
    spread = 1 if table.endswith("dense") else 1_000_003
    kt = (np.int32, np.int64)[n % 2]
    fact = [(rng.integers(0, 340, n) * spread).astype(kt), rng.integers(-10**7, 10**7, n),
            rng.integers(0, 50, n).astype((np.int32, np.uint8)[nsum % 2]), rng.integers(0, 9, n).astype(np.uint8)]
    dim = [(idx * spread).astype(np.int32), rng.integers(0, 17, nb).astype(np.int32)]
    spec = dict(fact=fact, dim=dim, fact_fk=0, dim_key=0, group_cols=[5], aggs=AGGS[nsum], capacity_groups=64,
                preds=[(3, "lt", 7), (2, "ne", 4)] if n % 3 else [],
                sum_expr=[("col", 1), ("col", 2), "mul"] if total else None)
    want = oracle.run_plan(want_pairs=False, cap_groups=None, want_row_ids=False,
                           **{k: v for k, v in spec.items() if k != "capacity_groups"})
    try:
        ctx.set_variant(1)
        got = gpu_plan(ctx, **spec)
    finally:
        ctx.set_variant(-1)
    compare(got, want, spec)
