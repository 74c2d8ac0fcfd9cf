"""A Counter that the cyclic collector frees together with its tables, batches
and plans (module globals at the interpreter's end, objects kept by a traceback)
frees each handle once and before its context, whatever the order of the
finalizers.  Host logic, with stand-ins for the library's calls."""
import ctypes
import gc

import numpy as np
import pytest

from paper_2206_05269_gb300 import wc


@pytest.mark.parametrize("order", [0, 1, 2])
def test_objects_in_one_cycle_are_freed_before_their_context(monkeypatch, order):
    log = []
    monkeypatch.setattr(wc, "wc_create", lambda *a: 7)
    monkeypatch.setattr(wc, "wc_plan_create", lambda *a: ctypes.c_void_p(30))
    monkeypatch.setattr(wc, "_stream_handle", lambda s: 0)
    for kind in ("table", "batch", "plan"):
        monkeypatch.setattr(wc, f"wc_{kind}_free", lambda h, kind=kind: log.append((kind, h.value)))
    monkeypatch.setattr(wc, "wc_destroy", lambda c: log.append(("context", c)))
    gc.collect()
    gc.disable()
    try:
        c = wc.Counter()
        objs = [wc.Table(ctypes.c_void_p(11), counter=c), wc.Batch(ctypes.c_void_p(20), 1, counter=c),
                wc.Plan(c, np.zeros(2, np.uint64)), wc.Table(ctypes.c_void_p(12), counter=c)]
        objs.append(wc.Table(ctypes.c_void_p(13), owned=False, owner=objs[1]))
        objs[3].free()
        assert log == [("table", 12)]
        cycle = [c, *objs] if order == 0 else [*objs, c] if order == 1 else [*objs[::-1], c]
        cycle.append(cycle)
        del c, objs, cycle
        gc.collect()
    finally:
        gc.enable()
    assert log[-1] == ("context", 7)
    assert sorted(log) == [("batch", 20), ("context", 7), ("plan", 30), ("table", 11), ("table", 12)]
