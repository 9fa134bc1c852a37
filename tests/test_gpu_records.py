"""Calendar kernels whose GPU records stay in global memory, lists of finish stamps on small clusters, and arrival draws of blocks and
classes without arrivals."""
import numpy as np
import pytest

from qsim_inputs import presets
from qsim_inputs.spec import PLACE_LEAST_LOADED, PLACE_RANDOM, ROUTER_IMMEDIATE, ROUTER_SLI, ROUTER_SLI_GENERAL
from test_gpu_calendar import block_bytes, check, env, light, together

pytestmark = pytest.mark.gpu


def runs_far(inp, **kw):
    """Are the records of this configuration in global memory?  (Less is on chip then than with QSIM_RECORDS=near.)"""
    near, far = (block_bytes(inp, QSIM_ROUNDS="calendar", QSIM_WARPS="1", QSIM_RECORDS=r) for r in ("near", "far"))
    return far < near and block_bytes(inp, **kw) == far


def crowded(N, **kw):
    inp = presets.crowded("decode", N=N, R=2, **kw)
    if kw.get("router") == ROUTER_SLI_GENERAL:
        inp = inp.with_(w_solo=np.array([[0.25, 0.75]]), w_mix=np.array([[0.6, 0.4]]), p_solo=np.array([[0.8, 0.8]]))
    return inp


def trace(N):
    """A trace under the KV slope."""
    inp = presets.trace_replay(n=N, R=1, T=3.0, placement=PLACE_LEAST_LOADED)[0]
    return inp.with_(M=np.array([7 * N // 10], np.uint32))


# (up to 992 GPUs a small batch cap keeps the finish stamps, and with them the records, on chip)
@pytest.mark.parametrize("make,calls,budget", [
    (lambda: presets.cfg2(N=129, R=2), [150], None),
    (lambda: presets.cfg2(N=1025, R=2), [40, 30], None),                 # a second row per lane
    (lambda: presets.cfg4(N=257, R=2), [120], None),
    (lambda: presets.cfg4(N=200, R=2), [60, 60], 40),                    # launches that end on the event budget
    (lambda: presets.cfg3(N=200, R=2, block_len=0.3), [420], None),      # solo GPUs, decode backlog, role changes
    (lambda: presets.cfg4(N=2048, R=1), [30, 10], None),
    (lambda: presets.cfg2(N=4096, R=1), [25], None),                     # the most rows of GPUs and buckets
    (lambda: light(presets.cfg2(N=1200, R=1), 0.2), [60], None),         # short iterations: more ends in a bucket than lanes
    (lambda: crowded(1000, placement=PLACE_LEAST_LOADED), [250], None),
    (lambda: presets.crowded("prefill", N=1100, R=1, placement=PLACE_RANDOM, router=ROUTER_SLI), [200], None),
    # the run-time-configured instance: uniform placement, KV slope, no router, weighted pools, a trace
    (lambda: crowded(1000, placement=PLACE_RANDOM), [150, 50], None),
    (lambda: presets.cfg2(N=1500, R=1, placement=PLACE_RANDOM), [40], None),
    (lambda: presets.cfg2(N=200, R=2).with_(coeffs=presets.COEFFS_PAPER_KV), [150, 100], None),
    (lambda: crowded(1000, placement=PLACE_RANDOM, router=ROUTER_IMMEDIATE), [150], None),
    (lambda: crowded(1000, placement=PLACE_LEAST_LOADED, router=ROUTER_SLI_GENERAL), [100, 50], None),
    (lambda: together(1000), [40, 60], None),                            # all GPUs' ends in a bucket
    (lambda: trace(1000), [120], None),
])
def test_records_in_global_memory_against_the_oracle(make, calls, budget):
    inp = make()
    with env(QSIM_RECORDS="far"):
        assert runs_far(inp, QSIM_ROUNDS="calendar", QSIM_WARPS="1", QSIM_RECORDS="far")
        check(inp, calls, "calendar", budget)


def test_records_in_global_memory_run_time_configured_instance():
    inp = presets.cfg4(N=300, R=2)
    with env(QSIM_RECORDS="far", QSIM_KERNEL="generic"):
        assert runs_far(inp, QSIM_ROUNDS="calendar", QSIM_WARPS="1", QSIM_RECORDS="far")
        check(inp, [60, 30], "calendar")


def test_records_in_global_memory_targets_that_change():
    """Mixed GPUs become solo ones and back between launches, with a backlog in the decode buffer."""
    from oracle import OracleSim
    from paper_2602_02987_b200 import QSim
    from parity import assert_parity
    inp = crowded(1000, placement=PLACE_LEAST_LOADED, router=ROUTER_SLI)
    out = []
    with env(QSIM_RECORDS="far", QSIM_ROUNDS="calendar", QSIM_WARPS="1"):
        assert runs_far(inp, QSIM_RECORDS="far")
        for cls in (QSim, OracleSim):
            sim = cls(inp)
            for M in (500, 250, 500, 1000, 0, 400):
                sim.set_targets(M, inp.xstar[0], inp.n_xstar[0], inp.n_qpstar[0], [0.88, 0.88])
                sim.run(25)
            out.append((sim.stats(), [sim.server_state(r) for r in range(inp.R)]))
            sim.close()
    (got, state), (ref, want) = out
    assert_parity(got, ref, what="targets that change")
    for a, b in zip(state, want):
        for k in a:
            assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("first,second", [("far", "near"), ("near", "far")])
def test_records_in_global_memory_resume_and_chunks(first, second):
    """A state saved by one of the two kinds of instance is resumed by the other; chunked launches hand replications over."""
    from parity import assert_parity
    from oracle import run_oracle
    from paper_2602_02987_b200 import QSim
    inp = presets.cfg4(N=300, R=40)
    assert runs_far(inp, QSIM_ROUNDS="calendar", QSIM_RECORDS="far")
    with env(QSIM_RECORDS=first, QSIM_ROUNDS="calendar", QSIM_CHUNKS="3"):
        sim = QSim(inp)
        sim.run(96)
        saved = sim.checkpoint()
        sim.close()
    with env(QSIM_RECORDS=second, QSIM_ROUNDS="calendar"):
        sim = QSim(inp, checkpoint=saved)
        sim.run(40)
        got = sim.stats()
        sim.close()
    assert_parity(got, run_oracle(inp, 136), what=f"{first}, then {second}")


@pytest.mark.parametrize("N,near", [(1024, 7), (1500, 5), (4096, 2)])
def test_records_in_global_memory_where_few_replications_fit(N, near):
    """By default from fewer than six resident replications on, and when more wait."""
    assert not runs_far(presets.cfg2(N=N, R=near * 148))
    assert runs_far(presets.cfg2(N=N, R=near * 148 + 1)) == (near < 6)


@pytest.mark.parametrize("make,calls", [
    (lambda: presets.cfg2(N=32, R=3).with_(B=1024), [300, 200]),
    (lambda: presets.cfg4(N=31, R=3).with_(B=700), [400]),
    (lambda: presets.cfg2(N=12, R=3).with_(B=4096, coeffs=presets.COEFFS_PAPER_KV), [400]),
    (lambda: presets.single_class(N=30, B=1024, P=20, D=10, lam=400.0, R=2, M=30), [60]),         # many requests finish at once
])
def test_lists_of_stamps_on_clusters_of_up_to_32_gpus(make, calls):
    check(make(), calls, "scan")


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
