"""Injected arrivals, time-based runs and target updates on the CUDA path: hand-worked trajectories and the
online-replanning trace replay, against the oracle and against the hand-computed totals."""
import numpy as np
import pytest

from qsim_inputs import online, presets
from qsim_inputs.spec import PLACE_LEAST_LOADED, PLACE_RANDOM, ROUTER_SLI, ROUTER_SLI_GENERAL

from parity import assert_parity

pytestmark = pytest.mark.gpu


def _both(inp, iters):
    from oracle import OracleSim
    from paper_2602_02987_b200 import QSim
    g = QSim(inp); g.run(iters); gs = g.stats(); gstate = g.server_state(0); g.close()
    o = OracleSim(inp); o.run(iters); os_ = o.stats(); ostate = o.server_state(0); o.close()
    assert_parity(gs, os_, what=inp.name)
    for k in gstate:
        assert np.array_equal(gstate[k], ostate[k]), k
    return gs


def test_hand_trajectory_one_gpu():
    # tests/golden/hand_trace_1gpu.txt: ttft 0.02024 + 0.03958, tpot 0.01017 + 0.00505, 6 iterations, revenue 1032
    inp = presets.single_class(N=1, B=3, C=256, P=512, D=2, M=1, inject=[(0.0, 0, 512, 2), (0.001, 0, 512, 2)])
    st = _both(inp, 20)
    assert abs(st["sum_ttft"][0, 0] - 0.05982) < 1e-12 and abs(st["sum_tpot"][0, 0] - 0.01522) < 1e-12
    assert int(st["iters_mixed"][0]) == 4 and int(st["iters_solo"][0]) == 2
    assert 1.0 * st["tokens_in_completed"].sum() + 2.0 * st["tokens_out_completed"].sum() == 1032.0
    assert abs(st["busy_mixed"][0] - 0.04058) < 1e-12 and abs(st["busy_solo"][0] - 0.0101) < 1e-12


def test_hand_trajectory_two_gpus():
    # tests/golden/hand_trace_2gpu.txt: three requests decode on the solo GPU, one on the mixed GPU, 0.00004 s of buffer wait
    inj = [(0.0, 0, 256, 6), (0.001, 0, 256, 6), (0.002, 0, 256, 6), (0.003, 0, 256, 6)]
    inp = presets.single_class(N=2, B=2, C=256, P=256, D=6, M=1, inject=inj)
    st = _both(inp, 40)
    assert int(st["placed_solo"][0, 0]) == 3 and int(st["placed_mixed"][0, 0]) == 1
    tpot = .005075 + (.05587 - .02024) / 6 + (.06578 - .03036) / 6 + (.07102 - .04053) / 6
    assert abs(st["sum_tpot"][0, 0] - tpot) < 1e-12
    assert abs(st["area_Qd"][0, 0] - 0.00004) < 1e-12
    assert int(st["iters_mixed"][0] + st["iters_solo"][0]) == 21


@pytest.mark.parametrize("placement", [0, 1])
def test_trace_replay_with_online_replanning(placement):
    from oracle import OracleSim
    from paper_2602_02987_b200 import QSim
    inp, Pm, Dm = presets.trace_replay(R=3, T=60.0, placement=placement)
    g = QSim(inp)
    dg = online.run_online(g, inp, Pm, Dm, 60.0)
    gs = g.stats(); g.close()
    o = OracleSim(inp)
    do = online.run_online(o, inp, Pm, Dm, 60.0)
    os_ = o.stats(); o.close()
    assert dg == do and len(dg) == 5
    assert_parity(gs, os_, what=f"trace replay, placement {placement}")
    assert gs["arrivals"][0].sum() == inp.inject_t.shape[0]


def test_run_until_matches_iteration_horizon_on_the_gpu():
    from paper_2602_02987_b200 import QSim
    inp = presets.cfg0(R=4, horizon_iters=800)
    a = QSim(inp); a.run(800); sa = a.stats(); a.close()
    b = QSim(inp); b.run_until(float(sa["T_elapsed"][0]) * 0.4); b.run_until(float(sa["T_elapsed"][0])); sb = b.stats(); b.close()
    for k in sa:
        if sa[k].dtype.kind == "f":
            assert np.allclose(sa[k], sb[k], rtol=1e-12, atol=0), k
        else:
            assert np.array_equal(sa[k], sb[k]), k


@pytest.mark.parametrize("theta", [0.0, 0.2])
@pytest.mark.parametrize("coeffs", [presets.COEFFS_PAPER, presets.COEFFS_PAPER_KV], ids=["no KV slope", "KV slope"])
@pytest.mark.parametrize("placement", [0, 1])
@pytest.mark.parametrize("n", [4, 10, 32, 33])
def test_trace_replay_with_and_without_the_kv_slope(n, placement, coeffs, theta):
    # the KV bookkeeping has memory only where the slope is not zero: every instance that a replay can get, up to and beyond 32 GPUs
    from oracle import OracleSim
    from paper_2602_02987_b200 import QSim
    inp, Pm, Dm = presets.trace_replay(n=n, R=2, T=25.0, placement=placement, coeffs=coeffs)
    inp = inp.with_(theta=np.full(inp.I, theta))
    out = []
    for cls in (QSim, OracleSim):
        sim = cls(inp)
        made = online.run_online(sim, inp, Pm, Dm, 25.0)
        out.append((made, sim.stats(), [sim.server_state(r) for r in range(inp.R)]))
        sim.close()
    (dg, gs, gstate), (do, os_, ostate) = out
    assert dg == do
    assert_parity(gs, os_, what=f"trace replay n={n}, placement {placement}, slope {coeffs[5]}, theta {theta}")
    for a, b in zip(gstate, ostate):
        for k in a:
            assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("placement", [PLACE_LEAST_LOADED, PLACE_RANDOM])
@pytest.mark.parametrize("router", [ROUTER_SLI, ROUTER_SLI_GENERAL])
@pytest.mark.parametrize("N", [12, 140])
def test_smaller_mixed_group_with_a_backlog_in_the_solo_pool(N, router, placement):
    # New targets turn mixed GPUs into solo ones, so the solo pool's backlog finds slots at the next event; when that event ends a
    # prefill whose request goes to the empty mixed pool, the solo pool is still served first (both draw from one sequence)
    from oracle import OracleSim
    from paper_2602_02987_b200 import QSim
    # (few first events after a change are such a prefill: many replications and changes)
    R = 512 if N < 100 else 96
    inp = presets.crowded("decode", N=N, R=R, placement=placement, router=router)
    if router == ROUTER_SLI_GENERAL:
        inp = inp.with_(w_solo=np.array([[0.7, 0.3]]), w_mix=np.array([[0.2, 0.8]]))
    w = (inp.w_solo[0], inp.w_mix[0]) if router == ROUTER_SLI_GENERAL else (None, None)
    out = []
    for cls in (QSim, OracleSim):
        sim = cls(inp)
        for k in range(48):
            M = N // 2 if k % 2 == 0 else N // 4
            sim.set_targets(M, inp.xstar[0], inp.n_xstar[0], inp.n_qpstar[0], [0.88, 0.88], *w)
            sim.run(6)
        out.append((sim.stats(), [sim.server_state(r) for r in range(inp.R)]))
        sim.close()
    (gs, gstate), (os_, ostate) = out
    assert os_["Qd"].sum() > R
    assert_parity(gs, os_, what=f"target change, N={N}, router {router}, placement {placement}")
    for a, b in zip(gstate, ostate):
        for k in a:
            assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("burst", [64, 65, 200])
@pytest.mark.parametrize("N,rounds", [(1, "scan"), (40, "scan"), (140, "scan"), (140, "calendar")])
def test_a_burst_of_arrivals_joins_the_queue_before_the_next_event(N, rounds, burst, monkeypatch):
    # every GPU holds a prefill, which ends 0.7 ms after the burst (less than the shortest iteration, 5 ms): what finds the queue full is
    # lost, although the prefills that end next make room
    monkeypatch.setenv("QSIM_ROUNDS", rounds)
    inj = [(0.0, 0, 512, 40)] * N + [(0.0195, 0, 900, 25)] * burst + [(0.0196, 0, 500, 10)] * 3
    inp = presets.single_class(N=N, B=8, P=900, D=25, lam=0.5, theta=0.0, R=2, M=N, inject=inj).with_(qcap=64 if burst == 64 else burst - 1)
    st = _both(inp, 90)
    assert int(st["overflow"][0, 0]) == (3 if burst == 64 else 4)


@pytest.mark.parametrize("rate", [0.0, 1e-6, 50.0])
@pytest.mark.parametrize("N,gap", [(140, 0.0001), (140, 0.5), (1100, 0.0001), (1100, 0.5)])
def test_rounds_on_large_clusters_follow_the_load_of_the_trace(N, gap, rate):
    # whatever the class rates say: on the calendar (more shared memory than reading all GPUs) when requests come fast, by reading all
    # GPUs, from 32 rows on with two warps, when they come slowly
    from oracle import run_oracle
    from paper_2602_02987_b200 import QSim
    inj = [(gap * (k + 1), 0, 300 + k, 20 + k % 7) for k in range(60)]
    inp = presets.single_class(N=N, B=8, P=900, D=25, lam=0.5, theta=0.0, R=2, M=N // 2, inject=inj).with_(rates=np.array([[rate]]))
    sim = QSim(inp)
    plain = QSim(inp.with_(inject_t=None, inject_job=None, rates=np.array([[1.0 / (gap * N)]])))
    assert sim.layout_info()["warps"] == plain.layout_info()["warps"] == (2 if N > 992 and gap > 0.1 else 1)
    assert sim.layout_info()["smem_bytes"] == plain.layout_info()["smem_bytes"]
    plain.close()
    sim.run(600)
    assert_parity(sim.stats(), run_oracle(inp, 600), what=f"trace of gap {gap}, N={N}, rates {rate}")
    sim.close()
