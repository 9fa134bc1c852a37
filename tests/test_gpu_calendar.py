"""Clusters of more than 128 GPUs on one warp: rounds that work from the calendar of iteration ends and rounds that read all
GPUs, both against the CPU oracle (integer statistics and per-GPU end state exact, fp64 statistics within 1e-9), at the edges
of the calendar's shapes: sizes around its rows and bucket counts, iterations that last a bucket and that are shorter (where small
clusters read all GPUs instead), more iteration ends in a bucket than lanes, light load with empty buckets, a run cut into many
short launches."""
import contextlib
import os

import numpy as np
import pytest

from qsim_inputs import presets
from qsim_inputs.spec import PLACE_LEAST_LOADED, PLACE_RANDOM, ROUTER_SLI

from parity import F64_KEYS, INT_KEYS, assert_parity

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def env(**kw):
    keep = {k: os.environ.get(k) for k in kw}
    os.environ.update(kw)
    try:
        yield
    finally:
        for k, v in keep.items():
            if v is None:
                del os.environ[k]
            else:
                os.environ[k] = v


def check(inp, calls, rounds, budget=None):
    from oracle import OracleSim
    from paper_2602_02987_b200 import QSim
    with env(QSIM_ROUNDS=rounds, QSIM_FAMILY="warp", QSIM_WARPS="1"):
        sim = QSim(inp)
    assert sim.layout_info()["warps"] == 1
    if budget:
        sim.set_event_budget(budget)
    ora = OracleSim(inp)
    for h in calls:
        sim.run(h)
        ora.run(h)
    got, ref = sim.stats(), ora.stats()
    state, want = [sim.server_state(r) for r in range(inp.R)], [ora.server_state(r) for r in range(inp.R)]
    sim.close()
    ora.close()
    assert_parity(got, ref, what=f"{inp.name}, {rounds}")
    for r in range(inp.R):
        for k in state[r]:
            assert np.array_equal(state[r][k], want[r][k]), (inp.name, rounds, r, k)
    return got


def light(inp, share):
    return inp.with_(rates=inp.rates * share)


def short_iterations(N):
    """Iteration times that differ by a factor of three thousand: the shortest is shorter than a bucket of the calendar."""
    return presets.cfg2(N=N, R=2).with_(coeffs=np.array([2e-5, 8e-5, 5e-5, 1e-5, 5e-5, 0.0]))


def one_bucket(N):
    """Iteration times that differ by a factor of 400: the shortest lasts one to two buckets, and no bucket is loaded ahead."""
    return presets.cfg2(N=N, R=2).with_(coeffs=np.array([1.2e-4, 8e-5, 5e-5, 8.3e-5, 5e-5, 0.0]))


def block_bytes(inp, **kw):
    """Shared memory of a replication."""
    from paper_2602_02987_b200 import QSim
    with env(QSIM_FAMILY="warp", **kw):
        sim = QSim(inp)
    info = sim.layout_info()
    sim.close()
    return info["smem_bytes"]


def together(N):
    """One request for every GPU at time zero: all iterations end at the same times, more per bucket than a warp has lanes."""
    return presets.single_class(N=N, B=8, P=900, D=30, lam=0.5, R=2, M=N, inject=[(0.0, 0, 900, 30)] * N + [(0.05, 0, 300, 5)] * 40)


@pytest.mark.parametrize("rounds", ["calendar", "scan"])
@pytest.mark.parametrize("make,calls", [
    (lambda: presets.cfg2(N=129, R=2), [250]),
    (lambda: presets.cfg4(N=255, R=2), [60, 100]),
    (lambda: presets.cfg4(N=257, R=2), [150]),
    (lambda: presets.crowded("decode", N=160, R=2, placement=PLACE_LEAST_LOADED), [600]),
    (lambda: presets.crowded("prefill", N=384, R=2, placement=PLACE_RANDOM, router=ROUTER_SLI), [300]),
    (lambda: presets.cfg3(N=200, R=2, block_len=0.3), [420]),
    (lambda: light(presets.cfg2(N=150, R=2), 0.02), [500]),
    (lambda: light(presets.cfg4(N=300, R=2), 0.0005), [900, 900]),
    (lambda: presets.paper_instance(n=200, R=2), [700]),
    (lambda: short_iterations(140), [200]),
    (lambda: short_iterations(300), [60, 40]),
    (lambda: short_iterations(300).with_(gate=1), [60]),                  # the run-time-configured instance
    (lambda: presets.cfg3(N=220, R=2, block_len=0.2).with_(coeffs=short_iterations(1).coeffs), [150]),
    (lambda: presets.cfg4(N=210, R=2).with_(coeffs=short_iterations(1).coeffs), [60]),
    (lambda: presets.crowded("decode", N=260, R=2, placement=PLACE_RANDOM).with_(coeffs=np.array([2e-5, 8e-4, 5e-5, 1e-5, 5e-5, 0.0])), [6000, 2000]),
    (lambda: one_bucket(140), [200]),
    (lambda: one_bucket(600), [60]),
    (lambda: together(300), [40, 60]),
    (lambda: together(1000), [40, 60]),
    (lambda: light(presets.cfg2(N=700, R=2), 0.3), [70, 30]),             # 30 to 60 ends in a bucket
    (lambda: light(presets.cfg4(N=1025, R=1), 0.1), [90]),
])
def test_calendar_and_scan_against_the_oracle(make, calls, rounds):
    check(make(), calls, rounds)


@pytest.mark.parametrize("make,calendar", [(short_iterations, {200: False, 201: True, 300: True, 2000: True}), (one_bucket, {140: True, 300: True})])
def test_iterations_shorter_than_a_bucket_keep_larger_clusters_on_the_calendar(make, calendar):
    # (the calendar's lists take shared memory, 2 KB where iterations are shorter than a bucket)
    for N, want in calendar.items():
        lists = block_bytes(make(N), QSIM_ROUNDS="calendar", QSIM_WARPS="1") - block_bytes(make(N), QSIM_ROUNDS="scan")
        assert (lists > 0) == want, N
        if make is short_iterations:
            assert lists < 2048 + 4 * N, N


def test_the_kv_slope_takes_little_more_shared_memory():
    """Its longest iteration asks for 512 buckets; their lists stay within 2 KB, next to the 8 bytes per GPU of the token counts."""
    inp = presets.cfg2(N=224, R=2)
    plain = block_bytes(inp, QSIM_ROUNDS="calendar", QSIM_WARPS="1", QSIM_KERNEL="generic")
    slope = block_bytes(inp.with_(coeffs=presets.COEFFS_PAPER_KV), QSIM_ROUNDS="calendar", QSIM_WARPS="1")
    assert 8 * 224 < slope - plain <= 8 * 224 + 2048


@pytest.mark.parametrize("N", [1023, 2049, 4096])
def test_calendar_on_large_clusters_with_many_buckets(N):
    check(presets.cfg2(N=N, R=1), [30, 30], "calendar")


def test_calendar_is_rebuilt_by_every_launch():
    whole = check(presets.cfg4(N=200, R=2), [120], "calendar")
    parts = check(presets.cfg4(N=200, R=2), [1, 2, 3, 5, 8, 13, 21, 34, 33], "calendar", budget=40)
    for k in ("arrivals", "admitted", "done_mixed", "done_solo", "iters_mixed", "iters_solo"):
        assert np.array_equal(whole[k], parts[k]), k


@pytest.mark.parametrize("rounds", ["calendar", "scan"])
@pytest.mark.parametrize("rate,T", [(0.0, 1e15), (1e-10, 4e8)])
def test_long_idle_times_are_skipped(rate, T, rounds):
    # an end time, or a next arrival, more than 2^31 buckets after the last event
    from oracle import OracleSim
    from paper_2602_02987_b200 import QSim
    inp = together(140) if rate == 0.0 else presets.single_class(N=140, B=8, P=900, D=30, lam=rate, R=2, M=140)
    with env(QSIM_ROUNDS=rounds):
        sim = QSim(inp)
    ora = OracleSim(inp)
    for s in (sim, ora):
        s.run_until(T)
    got, ref = sim.stats(), ora.stats()
    assert sim.round_count() < 10000
    sim.close()
    ora.close()
    assert (got["arrivals"] > 0).all()
    for k in INT_KEYS:
        if k in ref:
            assert np.array_equal(got[k], ref[k]), k
    # a time integral is the difference of two sums of at most n times, none after the last event, in any order: each of the n
    # additions of a sum rounds by at most 2^-53 of n times the last event's time
    n, last = float(got["arrivals"].max()), 4e8 if rate > 0.0 else 10.0
    for k in F64_KEYS:
        assert np.allclose(got[k], ref[k], rtol=1e-9, atol=2 * n * n * last * 2.0 ** -53), k


@pytest.mark.parametrize("make,load,warps", [
    (lambda N: presets.cfg2(N=N, R=2), 0.1, {992: 1, 993: 2, 2017: 4, 4096: 16}),
    (lambda N: presets.cfg3(N=N, R=2, block_len=0.3), 0.1, {1100: 2}),
    (lambda N: presets.cfg4(N=N, R=2), 0.1, {1100: 2}),
    (lambda N: presets.cfg2(N=N, R=149), 0.6, {4096: 1}),
    (lambda N: presets.cfg2(N=N, R=2), 1.0, {1100: 1, 4096: 1}),
])
def test_several_warps_on_lightly_loaded_large_clusters(make, load, warps):
    from oracle import run_oracle
    from paper_2602_02987_b200 import QSim
    for N, want in warps.items():
        inp = light(make(N), load)
        sim = QSim(inp)
        assert sim.layout_info()["warps"] == want, N
        if inp.R == 2:
            sim.run(60)
            assert_parity(sim.stats(), run_oracle(inp, 60), what=f"{inp.name}, {want} warps")
        sim.close()


@pytest.mark.parametrize("inp,load,warps", [
    (lambda: presets.cfg2(N=1100, R=2), 0.2, 1),
    (lambda: presets.cfg2(N=2200, R=297), 0.13, 1),
    (lambda: presets.cfg2(N=2200, R=296), 0.13, 4),
    (lambda: presets.cfg2(N=4096, R=148), 0.2, 16),
    (lambda: presets.cfg2(N=4096, R=149), 0.1, 1),
    (lambda: presets.cfg4(N=4096, R=2400).with_(B=16), 1.0, 1),          # (not one thread per replication)
])
def test_the_calendar_runs_medium_loads_and_many_replications_of_large_clusters(inp, load, warps):
    from paper_2602_02987_b200 import QSim
    sim = QSim(light(inp(), load))
    assert sim.layout_info()["warps"] == warps
    sim.close()
