"""Calendar kernels whose GPU records stay in global memory, and arrival draws of blocks and classes without arrivals."""
import numpy as np
import pytest

from qsim_inputs import presets
from qsim_inputs.spec import PLACE_LEAST_LOADED
from test_gpu_calendar import check, env

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,calls", [
    (lambda: presets.cfg2(N=129, R=2), [150]),
    (lambda: presets.cfg2(N=1025, R=2), [40, 30]),                       # a second row per lane
    (lambda: presets.cfg4(N=257, R=2), [120]),
    (lambda: presets.cfg3(N=200, R=2, block_len=0.3), [420]),            # solo GPUs, decode backlog, role changes
    (lambda: presets.crowded("decode", N=160, R=2, placement=PLACE_LEAST_LOADED), [400]),
    (lambda: presets.paper_instance(n=200, R=2), [300]),                 # uniform placement: the run-time-configured instance
])
def test_records_in_global_memory_against_the_oracle(make, calls):
    with env(QSIM_RECORDS="far"):
        check(make(), calls, "calendar")


def test_records_in_global_memory_resume_and_chunks():
    """A state saved by one of the two kinds of instance is resumed by the other; chunked launches hand replications over."""
    from parity import assert_parity
    from oracle import run_oracle
    from paper_2602_02987_b200 import QSim
    inp = presets.cfg4(N=300, R=40)
    with env(QSIM_RECORDS="far", QSIM_ROUNDS="calendar", QSIM_CHUNKS="3"):
        sim = QSim(inp)
        sim.run(96)
        saved = sim.checkpoint()
        sim.close()
    with env(QSIM_RECORDS="near", QSIM_ROUNDS="calendar"):
        sim = QSim(inp, checkpoint=saved)
        sim.run(40)
        got = sim.stats()
        sim.close()
    assert_parity(got, run_oracle(inp, 136), what="far, then near")


@pytest.mark.parametrize("N", [40, 200])
def test_blocks_and_classes_without_arrivals(N):
    """Draws are divided by the rate of the block in which the next arrival is looked for; empty blocks are skipped."""
    inp = presets.cfg3(N=N, R=3, block_len=0.2)
    rates = np.array(inp.rates, np.float64)
    rates[0:3, 0] = 0.0          # starts in an empty block
    rates[5:9, 1] = 0.0          # a gap
    rates[:, 2] = 0.0            # never arrives
    rates[10:, 3] = 0.0          # ends
    rates[3:5, 3] *= 1e-3        # candidates far past the block's end
    check(inp.with_(rates=rates), [180, 180], "calendar" if N > 128 else "scan")
