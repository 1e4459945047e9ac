"""GPU: two contexts on two streams from two host threads, each running calls whose kernels have barriers over a whole
chip of blocks (radix sort, radix select): neither waits for the other's blocks beyond its limit, and every result is
right."""
import threading

import numpy as np
import pytest

import datagen
import oracle
from tests.gpu_util import up
from tests.plan_util import compare, gpu_plan_collect, gpu_plan_prepare

pytestmark = pytest.mark.gpu


def test_sorts_and_selects_side_by_side():
    import torch
    import paper_2203_01877_gb300 as tqp
    rng = np.random.default_rng(1)
    nb = 2_600_000  # 608 blocks of the sort
    bk = (rng.integers(0, nb // 4, nb) * 331).astype(np.int32)
    pk = (rng.integers(0, nb // 4, 100_000) * 331).astype(np.int32)
    wb, wp = oracle.join_pairs(bk, pk)
    d = datagen.dim_table(600_000, 500_000, seed=5)
    pr = datagen.probe_table(1_300_000, 600_000, seed=5)
    spec = dict(fact=[pr["fk"], pr["value"]], dim=[d["key"], d["payload"]], fact_fk=0, dim_key=0, group_cols=[3],
                aggs=[("sum", [("col", 1)]), ("count", None)], topk=40, topk_agg=0)
    want = oracle.run_plan(want_pairs=False, cap_groups=None, want_row_ids=False, **spec)
    errors = []

    def work(k):
        try:
            stream = torch.cuda.Stream()
            ctx = tqp.Context(0, 1 << 30)
            B, P = tqp.TableRef([up(bk)]), tqp.TableRef([up(pk)])
            ob, op = (torch.empty(len(wb), dtype=torch.int32, device="cuda") for _ in range(2))
            cnt = torch.empty(1, dtype=torch.int64, device="cuda")
            plan, res, bufs, keep, shape = gpu_plan_prepare(**spec)
            torch.cuda.synchronize()
            for i in range(25):
                if (i + k) % 2:
                    for t in (ob, op, cnt):
                        with torch.cuda.stream(stream):
                            t.fill_(-9)
                    ctx.set_variant(1 if i % 3 == 0 else -1)
                    tqp.tqp_hash_join(ctx, B, 0, P, 0, ob, op, len(wb), cnt, stream)
                    assert ctx.status(stream) == 0
                    assert int(cnt.item()) == len(wb)
                    assert np.array_equal(ob.cpu().numpy(), wb) and np.array_equal(op.cpu().numpy(), wp)
                else:
                    ctx.set_variant(-1)
                    tqp.tqp_run_plan(ctx, plan, res, stream)
                    assert ctx.status(stream) == 0
                    compare(dict(gpu_plan_collect(bufs, shape), status=0), want, spec)
            ctx.close()
        except BaseException as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]
