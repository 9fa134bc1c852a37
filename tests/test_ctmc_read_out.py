"""The memory that a read-out of the exponential-service model keeps with its handle (no GPU: the library is a stand-in that fills
the records)."""
import contextlib
import gc
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
