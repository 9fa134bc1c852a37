"""Workloads by which the speed of this library is judged: the calls that its users make, from a handful of replications of
a four-GPU cluster to thousands of replications of large ones, over both simulators (iterations with the state-dependent
iteration time; the exponential-service model) and every option that the benchmark configurations use.

A case names a recipe of `qsim_inputs.presets`, its sizes and how the program calls the library:

  whole   one call from host buffers to host statistics (`simulate_host`): a fresh system, all memory set up in the call
  study   a handle made, run over its whole horizon, read and closed again: one experiment among many
  resume  a handle that is kept and advanced step by step in steady state, as a long run with periodic read-outs does

and what it reads: `stats` (every replication, histograms where they are recorded) or `totals` (sums over replications).
"""
import math

import numpy as np
import torch  # noqa: F401  (device memory and streams of the binding)

from paper_2602_02987_b200 import QSim, QSimCTMC, simulate_host
from qsim_inputs import online, presets
from qsim_inputs.spec import PLACE_LEAST_LOADED, PLACE_RANDOM, ROUTER_SLI, ROUTER_SOLO_FIRST

COUNTERS = ("arrivals", "admitted", "prefill_done", "placed_mixed", "placed_solo", "done_mixed", "done_solo", "abandoned_p",
            "abandoned_d", "overflow", "overflow_d", "tokens_in_prefilled", "tokens_in_completed", "tokens_out_completed",
            "Qp", "X", "Qd", "Ym", "Ys")
SUMS = ("area_Qp", "area_X", "area_Qd", "area_Ym", "area_Ys", "sum_ttft", "sum_tpot")
SCALARS = ("iters_mixed", "iters_solo", "events", "busy_mixed", "busy_solo", "T_elapsed")


def listed():
    return [
        # the smallest call: the paper's kind of toy example, sixteen replications of four GPUs, where launches and set-up count
        dict(name="tiny_whole", recipe="tiny", call="whole", read="stats", N=4, R=16, h=600, placement=PLACE_LEAST_LOADED),
        # the convergence experiment of the paper's appendix: a few dozen seeds of one cluster size, uniform placement
        dict(name="convergence_study", recipe="paper", call="study", read="stats", N=50, R=40, h=1500, placement=PLACE_RANDOM),
        # a controller's what-if replay of one trace: ten GPUs, KV slope, the state read every ten seconds of simulated time
        dict(name="trace_replay", recipe="trace", call="epochs", read="stats", N=10, R=24, T=60.0, placement=PLACE_RANDOM),
        # a medium cluster, priority gate, separate pricing, no abandonment, every replication's statistics read after each step
        dict(name="medium_priority", recipe="cfg1", call="resume", read="stats", N=64, R=1024, h=2000, prewarm=1500),
        # the headline: an overloaded 512-GPU cluster, occupancy gate with abandonment, 4096 replications
        dict(name="overload_512", recipe="cfg2", call="resume", read="totals", N=512, R=4096, h=250, prewarm=500),
        # the same workload on a cluster of an odd size, once from the empty system, from host buffers
        dict(name="overload_whole_333", recipe="cfg2", call="whole", read="totals", N=333, R=1500, h=200),
        # one day of time-varying demand in 24 blocks, latency histograms, percentiles: 1024 GPUs
        dict(name="day_1024", recipe="cfg3", call="study", read="stats", N=1024, R=444, h=360, block_len=0.25),
        # the SLI-aware router with histograms over the sizes of the scaling study
        dict(name="sli_16", recipe="cfg4", call="resume", read="totals", N=16, R=8192, h=1000, prewarm=1000),
        dict(name="sli_256", recipe="cfg4", call="resume", read="totals", N=256, R=4096, h=160, prewarm=400),
        dict(name="sli_4096", recipe="cfg4", call="resume", read="totals", N=4096, R=1712, h=8, prewarm=24),
        # the exponential-service model: a small check and the full wave of replications of a 1000-GPU cluster
        dict(name="markov_small", recipe="ctmc", call="study", read="stats", N=20, R=64, T=6.0, router=ROUTER_SOLO_FIRST),
        dict(name="markov_1000", recipe="ctmc", call="resume", read="stats", N=1000, R=37888, T=3.0, prewarm_T=4.0, router=ROUTER_SLI),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    recipe = rng.choice(("tiny", "paper", "trace", "cfg1", "cfg2", "cfg2", "cfg3", "cfg4", "cfg4", "ctmc"))
    place = rng.choice((PLACE_LEAST_LOADED, PLACE_RANDOM))
    if recipe == "tiny":
        return dict(recipe=recipe, call="whole", read="stats", N=4, R=_log_int(rng, 4, 200), h=_log_int(rng, 200, 2000), placement=place)
    if recipe == "paper":
        return dict(recipe=recipe, call="study", read="stats", N=_log_int(rng, 5, 250), R=rng.randint(5, 60), h=_log_int(rng, 400, 3000), placement=place)
    if recipe == "trace":
        return dict(recipe=recipe, call="epochs", read="stats", N=rng.randint(5, 20), R=_log_int(rng, 1, 60), T=10.0 * rng.randint(3, 8), placement=place)
    if recipe == "cfg1":        # the recipe fixes the cluster of 64 GPUs
        return dict(recipe=recipe, call="resume", read=rng.choice(("stats", "totals")), N=64, R=_log_int(rng, 60, 2500), h=rng.randint(500, 1500), prewarm=1500)
    if recipe == "ctmc":
        N, R = _log_int(rng, 20, 4000), _log_int(rng, 300, 38000)
        T = min(8.0, 1.0e8 / (N * R))
        return dict(recipe=recipe, call="resume", read="stats", N=N, R=R, T=T, prewarm_T=T, router=rng.choice((ROUTER_SOLO_FIRST, ROUTER_SLI)))
    N = _log_int(rng, 16, 1500)
    if recipe == "cfg3":
        return dict(recipe=recipe, call="study", read="stats", N=N, R=max(20, min(1000, _log_int(rng, 5e4, 4e5) // N)), h=360, block_len=0.25)
    R = max(100, min(8192, _log_int(rng, 2e5, 2e6) // N))
    h = max(10, min(1500, int(6e7 / (N * R))))
    if recipe == "cfg2" and rng.random() < 0.5:
        return dict(recipe=recipe, call="whole", read=rng.choice(("stats", "totals")), N=N, R=R, h=h)
    return dict(recipe=recipe, call="resume", read=rng.choice(("stats", "totals", "totals")), N=N, R=R, h=h, prewarm=min(400, 4 * h))


def _inputs(case, seed):
    recipe, N, R = case["recipe"], case["N"], case["R"]
    if recipe == "tiny":
        inp = presets.cfg0(placement=case["placement"], R=R)
    elif recipe == "paper":
        inp = presets.paper_instance(n=N, R=R, placement=case["placement"])
    elif recipe == "trace":
        inp, Pm, Dm = presets.trace_replay(n=N, R=R, T=case["T"], seed=seed, placement=case["placement"])
        lam = np.array([2.4, 1.8])                   # the rates at which the recipe generates its two classes, per GPU
        M, xs, nx, nq, ps = online.replan(lam, Pm, Dm, N, inp.B, inp.C, inp.coeffs, inp.prices, separate=False)
        return inp.with_(M=np.array([M], np.uint32), xstar=xs[None], n_xstar=nx[None], n_qpstar=nq[None], p_solo=ps[None])
    elif recipe == "cfg3":
        inp = presets.cfg3(N=N, R=R, block_len=case["block_len"])
    elif recipe == "ctmc":
        inp = presets.ctmc_instance(n=N, R=R, router=case["router"])
    elif recipe == "cfg1":
        inp = presets.cfg1(R=R)
    else:
        inp = getattr(presets, recipe)(N=N, R=R)
    return inp.with_(seed=seed)


def prepare(case, seed):
    state = dict(case=case, inp=_inputs(case, seed))
    if case["call"] == "resume":
        if case["recipe"] == "ctmc":
            state["sim"], state["T"] = QSimCTMC(state["inp"]), case["prewarm_T"]
            state["sim"].run_until(state["T"])
        else:
            state["sim"] = QSim(state["inp"])
            state["sim"].run(case["prewarm"])
            state["sim"].sync()
    return state


def _of_totals(tot, I):
    out = {n: np.array([getattr(tot.cls[i], n) for i in range(I)], np.int64) for n in COUNTERS}
    out.update({n: np.array([getattr(tot.cls[i], n) for i in range(I)], np.float64) for n in SUMS})
    out.update({n: np.array(getattr(tot, n)) for n in SCALARS})
    return out


def _plain(stats):
    return {k: v.astype(np.int64) if v.dtype.kind == "u" else v for k, v in stats.items() if isinstance(v, np.ndarray)}


def _read(sim, case, I):
    return _plain(sim.stats()) if case["read"] == "stats" else _of_totals(sim.totals()[2], I)


def run(state):
    case, inp = state["case"], state["inp"]
    if case["call"] == "whole":
        got = simulate_host(inp, case["h"], per_rep=case["read"] == "stats")
        return _plain(got if case["read"] == "stats" else got["_totals"])
    if case["recipe"] == "ctmc":
        if case["call"] == "resume":
            state["T"] += case["T"]
            state["sim"].run_until(state["T"])
            return _plain(state["sim"].stats())
        sim = QSimCTMC(inp)
        sim.run_until(case["T"])
        out = _plain(sim.stats())
        sim.close()
        return out
    if case["call"] == "resume":
        state["sim"].run(case["h"])
        return _read(state["sim"], case, inp.I)
    sim = QSim(inp)
    if case["call"] == "epochs":
        seen = []
        for k in range(1, int(round(case["T"] / 10.0)) + 1):
            sim.run_until(10.0 * k)
            got = sim.stats()                      # what a controller reads at each epoch
            seen.append(got["arrivals"].astype(np.int64))
        out = _plain(got)
        out["arrivals_by_epoch"] = np.stack(seen)
    else:
        sim.run(case["h"])
        out = _read(sim, case, inp.I)
        if inp.hist:
            out["p_ttft"], out["p_tpot"] = sim.latency_percentiles([0.5, 0.95, 0.99])
    sim.close()
    return out


def _replication_iterations(case):
    """Server iterations of one replication: iterations are shorter than the one that measures the horizon."""
    if case["recipe"] == "trace":
        return case["N"] * case["T"] / 0.03
    return 1.3 * case["N"] * case["h"]


def work(case):
    """A request's life cycle is an entry of its class queue, the record of its prefill, a decode slot and a buffer entry, each
    written and read once (128 bytes), and 0.2 requests finish per server iteration; a server iteration takes about 20
    double-precision operations (two durations, its end, comparisons).  The exponential-service model keeps its counts on
    chip: its records and results move once, and a jump takes about 60 operations.  Results: 28 numbers per class."""
    I = 4 if case["recipe"] in ("cfg2", "cfg3", "cfg4") else 2
    out = case["R"] * I * 28 * 8 if case["read"] == "stats" else I * 28 * 8
    if case["recipe"] == "ctmc":
        jumps = 4.0 * case["N"] * case["R"] * case["T"]
        return {"bytes": out + 2 * case["R"] * I * 400, "flops": 60 * jumps}
    iters = case["R"] * _replication_iterations(case)
    if case["recipe"] == "cfg3":
        out += case["R"] * I * 2 * 1024 * 8
    return {"bytes": 0.2 * 128 * iters + out, "flops": 20 * iters}


def tolerance(case):
    """Counts are exact.  Clocks are fixed chains of rounded double operations; only sums of them may be taken in another
    order.  The other kernel family and launches in chunks, which add in other orders, differ by up to 1.8e-12 (busy times,
    sums of 1e5 equal-sized terms) in the norm and 2.5e-12 in one value."""
    return {"rel": 1e-11, "max": 1e-11, "differ": 0.0}


# --- the same two models in plain Python, for the cases that take seconds there ---------------------------------------------


def _philox(c, key):
    """Philox4x32-10 (Salmon et al., SC'11)."""
    c0, c1, c2, c3 = c
    k0, k1 = key & 0xffffffff, key >> 32
    for _ in range(10):
        a, b = 0xD2511F53 * c0, 0xCD9E8D57 * c2
        c0, c1, c2, c3 = (b >> 32) ^ c1 ^ k0, b & 0xffffffff, (a >> 32) ^ c3 ^ k1, a & 0xffffffff
        k0, k1 = (k0 + 0x9E3779B9) & 0xffffffff, (k1 + 0xBB67AE85) & 0xffffffff
    return c0, c1, c2, c3


def _uniform(w0, w1):
    return (((w0 << 21) | (w1 >> 11)) + 1) * 2.0 ** -53


def _log(x):
    m, e = math.frexp(x)
    m, e = 2.0 * m, e - 1
    if m > 1.4142135623730951:
        m, e = 0.5 * m, e + 1
    s = (m - 1.0) / (m + 1.0)
    z, acc = s * s, 1.0 / 25.0
    for k in range(11, -1, -1):
        acc = acc * z + 1.0 / (2 * k + 1)
    return e * 0.6931471805599453 + 2.0 * s * acc


class _Draws:
    def __init__(self, seed, rep):
        self.seed, self.rep = seed, rep

    def __call__(self, purpose, cls, index):
        return _philox((index & 0xffffffff, index >> 32, (purpose << 8) | cls, self.rep), self.seed)


class _Area:
    def __init__(self):
        self.parts, self.last = [], 0.0

    def touch(self, n, t):
        self.parts.append(n * (t - self.last))
        self.last = t

    def at(self, n, T):
        return math.fsum(self.parts + [n * (T - self.last)])


def _iterations(inp, T, rep):
    """One replication of the iteration-level model: fixed lengths, occupancy gate, solo-first router, no abandonment."""
    I, N, B, C, M = inp.I, inp.N, inp.B, inp.C, int(inp.M[0])
    a_m, beta, d_m, a_s, d_s = (float(v) for v in inp.coeffs[:5])
    xs, nx, nq = inp.xstar[0].tolist(), inp.n_xstar[0].tolist(), inp.n_qpstar[0].tolist()
    P, D, Lam = inp.P.tolist(), inp.D.tolist(), [float(N) * float(v) for v in inp.rates[0]]
    rnd, order, inf = _Draws(inp.seed, rep), 0, math.inf
    n_draw, ta = [0] * I, [inf] * I

    def next_arrival(i, t0):
        if Lam[i] > 0.0:
            w = rnd(0, i, n_draw[i])
            n_draw[i] += 1
            ta[i] = t0 + -_log(_uniform(w[0], w[1])) / Lam[i]

    for i in range(I):
        next_arrival(i, 0.0)
    cnt = {n: [0] * I for n in COUNTERS}
    area = {n: [_Area() for _ in range(I)] for n in ("Qp", "X", "Qd", "Ym", "Ys")}
    ttft, tpot = [[] for _ in range(I)], [[] for _ in range(I)]
    queue, buffer = [[] for _ in range(I)], []
    it, end, decs, pf = [0] * N, [inf] * N, [[] for _ in range(N)], [None] * N
    cur, busy, n_it, events = [(0, 0.0)] * N, ([], []), [0, 0], 0

    def count(name, i, by, t):
        area[name][i].touch(cnt[name][i], t)
        cnt[name][i] += by

    def choose(ok):
        nonlocal order
        if not ok:
            return None
        if inp.placement == PLACE_LEAST_LOADED:
            return min(ok, key=lambda g: (len(decs[g]), g))
        k = 0
        if len(ok) > 1:
            k = rnd(4, 0, order)[0] * len(ok) >> 32
            order += 1
        return ok[k]

    while True:
        t, src = inf, None
        for i in range(I):
            if ta[i] < t:
                t, src = ta[i], (0, i)
        for g in range(N):
            if end[g] < t:
                t, src = end[g], (1, g)
        if not t <= T:
            break
        events += 1
        if src[0] == 0:
            i = src[1]
            cnt["arrivals"][i] += 1
            count("Qp", i, 1, t)
            queue[i].append(t)
            next_arrival(i, t)
        else:
            g = src[1]
            it[g] += 1
            end[g] = inf
            chunk, tau = cur[g]
            n_it[chunk == 0] += 1
            busy[chunk == 0].append(tau)
            for job in [d for d in decs[g] if d[0] == it[g]]:
                _, i, tpf, mixed = job
                count("Ym" if mixed else "Ys", i, -1, t)
                cnt["done_mixed" if mixed else "done_solo"][i] += 1
                cnt["tokens_in_completed"][i] += P[i]
                cnt["tokens_out_completed"][i] += D[i]
                tpot[i].append((t - tpf) / D[i])
            decs[g] = [d for d in decs[g] if d[0] != it[g]]
            if chunk:
                i, left, arrived = pf[g]
                pf[g] = (i, left - chunk, arrived) if left > chunk else None
                if pf[g] is None:
                    count("X", i, -1, t)
                    cnt["prefill_done"][i] += 1
                    cnt["tokens_in_prefilled"][i] += P[i]
                    ttft[i].append(t - arrived)
                    count("Qd", i, 1, t)
                    buffer.append((i, t))
        while buffer:
            g = choose([g for g in range(M, N) if len(decs[g]) < (B - 1 if pf[g] else B)])
            g = choose([g for g in range(M) if len(decs[g]) < B - 1]) if g is None else g
            if g is None:
                break
            i, tpf = buffer.pop(0)
            count("Qd", i, -1, t)
            count("Ym" if g < M else "Ys", i, 1, t)
            cnt["placed_mixed" if g < M else "placed_solo"][i] += 1
            decs[g].append((it[g] + (end[g] < inf) + D[i], i, tpf, g < M))
        while True:
            wait = [i for i in range(I) if queue[i] and xs[i] > 0.0]
            if not wait:
                break
            i = min(wait, key=lambda i: ((cnt["X"][i] - nx[i]) / xs[i], -(cnt["Qp"][i] - nq[i]), i))
            g = choose([g for g in range(M) if pf[g] is None and len(decs[g]) <= B - 1])
            if g is None:
                break
            pf[g] = (i, P[i], queue[i].pop(0))
            count("Qp", i, -1, t)
            count("X", i, 1, t)
            cnt["admitted"][i] += 1
        for g in range(N):
            if end[g] == inf and (decs[g] or pf[g]):
                chunk = min(C, pf[g][1]) if pf[g] else 0
                tau = a_m + beta * chunk + d_m * len(decs[g]) if chunk else a_s + d_s * len(decs[g])
                cur[g], end[g] = (chunk, tau), t + tau
    out = dict(cnt, sum_ttft=[math.fsum(v) for v in ttft], sum_tpot=[math.fsum(v) for v in tpot], iters_mixed=n_it[0], iters_solo=n_it[1],
               events=events, busy_mixed=math.fsum(busy[0]), busy_solo=math.fsum(busy[1]), T_elapsed=T)
    for n in area:
        out["area_" + n] = [area[n][i].at(cnt[n][i], T) for i in range(I)]
    return out


def _jumps(inp, T, rep):
    """One replication of the exponential-service model: occupancy gate, solo-first or SLI-aware router."""
    I, M, inf, rnd = inp.I, inp.M, math.inf, _Draws(inp.seed, rep)
    cap = {"Ys": (inp.N - M) * inp.B, "Ym": M * (inp.B - 1)}
    runs_on = ["one", "Qp", "Qd0", "Qd1", "X", "Ym", "Ys"]
    rate = [[float(inp.N) * v for v in inp.lam], inp.theta, inp.theta, inp.theta, inp.mu_p, inp.mu_m, inp.mu_s]
    n = {k: [0] * I for k in ("Qp", "X", "Qd0", "Qd1", "Ym", "Ys")}
    n["one"] = [1] * I
    names = ("arrivals", "admitted", "prefill_done", "placed_mixed", "placed_solo", "done_mixed", "done_solo", "abandoned_p", "abandoned_d", "overflow_d")
    cnt = {k: [0] * I for k in names}
    area = {k: [_Area() for _ in range(I)] for k in ("Qp", "X", "Qd", "Ym", "Ys")}
    acc, lvl, last, fire, m = ([[v] * I for _ in range(7)] for v in (0.0, 0.0, 0.0, inf, 0))
    ring, pools, events = ([], []), [0] * I, 0

    def level(k, i):
        w = rnd(k if k < 4 else k + 4, i, m[k][i])
        m[k][i] += 1
        lvl[k][i] = -_log(_uniform(w[0], w[1]))
        return w[2]

    for i in range(I):
        for k in range(7):
            level(k, i)
        if rate[0][i] > 0.0:
            fire[0][i] = 0.0 + lvl[0][i] / rate[0][i]

    def held(c, i):
        return n["Qd0"][i] + n["Qd1"][i] if c[:2] == "Qd" else n[c][i]

    def put(c, i, by, t, fired=None):
        k, v = runs_on.index(c), n[c][i] + by
        if k != fired and rate[k][i] > 0.0:
            acc[k][i] += rate[k][i] * n[c][i] * (t - last[k][i])
            last[k][i] = t
            fire[k][i] = t + max(lvl[k][i] - acc[k][i], 0.0) / (rate[k][i] * v) if v else inf
        area[c[:2] if c[:2] == "Qd" else c][i].touch(held(c, i), t)
        n[c][i] = v

    while True:
        t, k, i = min((fire[k][i], k, i) for k in range(7) for i in range(I))
        if not t <= T:
            break
        events += 1
        c, rank = runs_on[k], level(k, i)
        if k == 0:
            put("Qp", i, 1, t)
        else:
            if c[:2] == "Qd":
                at = [p for p, j in enumerate(ring[k - 2]) if j == i]
                ring[k - 2].pop(at[rank * n[c][i] >> 32])
            put(c, i, -1, t, fired=k)
        cnt[("arrivals", "abandoned_p", "abandoned_d", "abandoned_d", "prefill_done", "done_mixed", "done_solo")[k]][i] += 1
        acc[k][i], last[k][i] = 0.0, t
        fire[k][i] = t + lvl[k][i] / (rate[k][i] * n[c][i]) if n[c][i] else inf
        if k == 4:
            pool = 0
            if inp.router == ROUTER_SLI:
                w = rnd(5, i, pools[i])
                pools[i] += 1
                pool = 0 if _uniform(w[0], w[1]) <= inp.p_solo[i] else 1
            if len(ring[pool]) >= inp.qcap:
                cnt["overflow_d"][i] += 1
            else:
                ring[pool].append(i)
                put("Qd%d" % pool, i, 1, t)
        for pool in (0, 1):
            while ring[pool]:
                open_ = [y for y in ("Ys", "Ym") if sum(n[y]) < cap[y] and (inp.router != ROUTER_SLI or y == ("Ys", "Ym")[pool])]
                if not open_:
                    break
                j = ring[pool].pop(0)
                put("Qd%d" % pool, j, -1, t)
                put(open_[0], j, 1, t)
                cnt["placed_solo" if open_[0] == "Ys" else "placed_mixed"][j] += 1
        while sum(n["X"]) < M:
            wait = [j for j in range(I) if n["Qp"][j] and inp.xstar[j] > 0.0]
            if not wait:
                break
            j = min(wait, key=lambda j: ((n["X"][j] - inp.n_xstar[j]) / inp.xstar[j], -(n["Qp"][j] - inp.n_qpstar[j]), j))
            put("Qp", j, -1, t)
            put("X", j, 1, t)
            cnt["admitted"][j] += 1
    out = dict(cnt, events=events, T_elapsed=T)
    for c in area:
        v = [held("Qd0" if c == "Qd" else c, i) for i in range(I)]
        out[c], out["area_" + c] = v, [area[c][i].at(v[i], T) for i in range(I)]
    done = [a + b for a, b in zip(cnt["done_mixed"], cnt["done_solo"])]
    paid = cnt["prefill_done"] if inp.meta["separate"] else done
    out["_revenue_rate"] = sum(inp.prices[0] * inp.P[i] * paid[i] + inp.prices[1] * inp.D[i] * done[i] for i in range(I)) / (inp.N * T)
    return out


def exact(case, seed):
    if case["recipe"] == "tiny" and case["R"] * case["h"] <= 20_000:
        inp = _inputs(case, seed)
        tau = float(inp.coeffs[3]) + float(inp.coeffs[4]) * inp.B
        reps = [_iterations(inp, float(case["h"]) * tau, r) for r in range(case["R"])]
    elif case["recipe"] == "ctmc" and case["call"] == "study":
        inp = _inputs(case, seed)
        reps = [_jumps(inp, case["T"], r) for r in range(case["R"])]
    else:
        return None
    return {k: np.array([r[k] for r in reps]) for k in reps[0]}
