"""The memory that a read-out of the exponential-service model keeps with its handle (no GPU: the library is a stand-in that fills
the records)."""
import contextlib
import gc
import sys
import threading
import types
import weakref

import numpy as np
import pytest

from paper_2602_02987_b200 import binding
from qsim_inputs import presets

R = 3


class Library:
    """qsim_ctmc_stats fills every record's event count with the next number."""

    def __init__(self):
        self.reads = 0
        self.filled = lambda k: None

    def qsim_ctmc_stats(self, cfg, ws, nbytes, stream, per):
        self.reads += 1
        k = self.reads
        rec = np.ctypeslib.as_array((np.ctypeslib.ctypes.c_uint8 * (R * binding._CTMC_REP_STATS.itemsize)).from_address(per.value))
        rec = rec.view(binding._CTMC_REP_STATS)
        rec[:] = np.zeros((), binding._CTMC_REP_STATS)
        rec["events"] = k
        self.filled(k)
        return 0


@pytest.fixture
def handle(monkeypatch):
    import torch
    monkeypatch.setattr(torch.cuda, "is_available", lambda: True)
    monkeypatch.setattr(torch.cuda, "device", lambda d: contextlib.nullcontext())
    lib = Library()
    for name in ("qsim_ctmc_workspace_bytes", "qsim_ctmc_init"):
        setattr(lib, name, lambda *a: 0)
    monkeypatch.setattr(binding, "load_library", lambda: lib)
    return binding.QSimCTMC(presets.ctmc_instance(n=4, R=R), device="cpu", stream=types.SimpleNamespace(cuda_stream=0)), lib


def test_a_closed_handle_keeps_no_records(handle, monkeypatch):
    sim, _ = handle
    made = []

    def empty(*a, _empty=np.empty, **kw):
        out = _empty(*a, **kw)
        if out.dtype == binding._CTMC_REP_STATS:
            made.append(weakref.ref(out))
        return out

    monkeypatch.setattr(binding.np, "empty", empty)
    sim.stats()
    sim.stats()
    assert len(made) == 1 and made[0]() is not None          # the second read used the memory of the first
    sim.close()
    gc.collect()
    assert made[0]() is None


def test_two_threads_that_read_at_the_same_time_share_no_records(handle):
    """A second thread's read begins between any two steps of the first one's, and takes its numbers out of the records after the first one's
    records were filled."""
    sim, lib = handle
    code = binding.QSimCTMC.stats.__code__
    main = threading.get_ident()
    step, steps = 0, 1
    while step < steps:
        sim.stats()
        got, filled, begun, first_filled = {}, {}, threading.Event(), threading.Event()

        def on_fill(k):
            filled[threading.get_ident() == main] = k
            if threading.get_ident() == main:
                first_filled.set()
            else:
                begun.set()
                assert first_filled.wait(10)

        other = threading.Thread(target=lambda: got.update(other=sim.stats()["events"]))
        count = 0

        def trace(frame, event, arg):
            nonlocal count
            if frame.f_code is not code:
                return None
            if not frame.f_trace_opcodes:
                frame.f_trace_opcodes = True
                sys.settrace(trace)          # (takes note of it)
            if event == "opcode":
                if count == step:
                    other.start()
                    assert begun.wait(10)
                count += 1
            return trace

        lib.filled = on_fill
        before = sys.gettrace()
        sys.settrace(trace)
        try:
            mine = sim.stats()["events"]
        finally:
            sys.settrace(before)
        if not begun.is_set():          # (the first read had fewer steps this time)
            break
        other.join(10)
        lib.filled = lambda k: None
        assert (mine == filled[True]).all() and (got["other"] == filled[False]).all(), step
        step, steps = step + 1, count
    assert steps > 20
