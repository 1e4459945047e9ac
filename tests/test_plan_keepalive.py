"""CPU: a plan keeps the host buffers that its IN and LIKE predicates point to."""
import ctypes as C
import gc
import weakref

import numpy as np

import paper_2203_01877_gb300 as tqp


class Table:  # what make_plan needs of a TableRef
    t = tqp.Table()
    widths = [0, 8]


def test_plan_holds_its_predicates_values(monkeypatch):
    refs = []
    fill = tqp._set_operand

    def spy(table, col, op, v, keep):
        out = fill(table, col, op, v, keep)
        refs.append(weakref.ref(keep[-1]))
        return out

    monkeypatch.setattr(tqp, "_set_operand", spy)
    values = list(range(1000, 1200))
    plan = tqp.make_plan(Table(), [(0, "in", values), (1, "like", "%abc%"), (1, "in", ["xy", "z"])])
    gc.collect()
    noise = [np.full(200, 7, np.int64) for _ in range(50)]
    assert len(refs) == 3 and all(r() is not None for r in refs)
    read = lambda k, n: C.string_at(plan.preds[k].lo, n)  # noqa: E731
    assert np.frombuffer(read(0, 1600), np.int64).tolist() == values
    assert read(1, 5) == b"%abc%" and read(2, 16) == b"xy" + b"\0" * 6 + b"z" + b"\0" * 7
    del plan, noise
    gc.collect()
    assert all(r() is None for r in refs)
