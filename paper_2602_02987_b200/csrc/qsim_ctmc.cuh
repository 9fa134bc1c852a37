// Exponential-service model of the gate-and-route network (Section 2.3): device kernel and C ABI.
// Included at the end of qsim_lib.cu (it uses that file's error helpers and the Philox / qlog routines of
// qsim_device.cuh).
//
// Requests of a class are exchangeable here, so a replication is a handful of integers per class plus the
// class order of its decode buffers: one THREAD simulates one replication.  Every class has seven unit-rate Poisson
// processes (arrivals, abandonment from the prefill queue, abandonment from each decode buffer, prefill completions,
// mixed and solo decode completions) that run on the integrated intensities of Eq. (7)-(9): a process with intensity
// c n(t) keeps the integral acc of c n since its last jump and the exponential level lvl of its next jump, and its jump
// time is recomputed whenever n changes.  Per event a thread scans its 7 I jump times, applies the jump, lets the policy
// act (decode buffers into free slots, solo group first; then the prefill gate) and then brings the clocks of the counts
// that changed up to date.  All clock arithmetic is single IEEE operations in a fixed order.
// While a launch runs, a replication's clocks and counts sit in shared memory (word w of thread t at w * lanes + t).
//
// Bound: the dependent-instruction latency of each thread's chain and the divergence between jump kinds.  So a jump and the
// policy only change counts (an addition and a bit in a mask); everything a changed count entails - time integral,
// accumulated hazard, the division that gives the next jump time - is done once per changed count by one piece of code at
// the end of the event (commit), where it used to be repeated inline at each of a dozen places (83 KB of code, up to six
// divisions for a finished prefill whose buffer stays empty).  Measured, two-class instance, SLI-aware router, n = 1000: R = 37888,
// 3 s 41.2 -> 27.3 ms (6.6e9 -> 10.0e9 jumps/s), R = 300, 8 s 104 -> 38 ms.  Changes at the same instant add nothing to an
// integral, so the values are those of one update after another.
#pragma once

namespace qsimdev {

enum { CK_ARR = 0, CK_ABP = 1, CK_ABD0 = 2, CK_ABD1 = 3, CK_SP = 4, CK_SDM = 5, CK_SDS = 6, CK_N = 7 };
enum { CC_ARRIVALS = 0, CC_ADMITTED, CC_PREFILL_DONE, CC_PLACED_MIXED, CC_PLACED_SOLO, CC_DONE_MIXED, CC_DONE_SOLO,
       CC_ABANDONED_P, CC_ABANDONED_D, CC_OVERFLOW_D, CC_N };
enum { CA_QP = 0, CA_X, CA_QD, CA_YM, CA_YS, CA_N };

struct CtmcClk { double acc, lvl, t_last, t_fire; unsigned long long m; };

// state of one replication in global memory between launches
struct CtmcRep {
    double T_end;
    unsigned long long events;
    uint32_t head[2], n[2];
    uint32_t err, done;
    CtmcClk clk[CK_N][MAXI];
    uint32_t Qp[MAXI], X[MAXI], Qd[2][MAXI], Ym[MAXI], Ys[MAXI];
    unsigned long long reserved[MAXI];       // (keeps the layout of saved workspaces)
    double area[CA_N][MAXI], area_t[CA_N][MAXI];
    unsigned long long cnt[MAXI][CC_N];
};

struct CtmcClassPar { double lambda, theta, mu_p, mu_m, mu_s, xstar, nx, nq, ps; uint32_t prio, pad; };

struct CtmcParams {
    uint32_t I, N, M, B, R, qcap, gate, router, init, lanes;     // lanes: replications per warp
    unsigned long long seed, rep_offset, event_budget;
    double T_end;
    CtmcClassPar cls[MAXI];
    CtmcRep *reps;          // [R]
    uint8_t *rings;         // [R][2][qcap] class ids of the decode buffers, FCFS
    uint32_t *not_done;
};

// Working copy of one replication in shared memory: 39 I 8-byte words, word w of thread t at [w * lanes + t] (consecutive
// threads hit consecutive banks).  The event counters and the time integrals are only ever added to, so they stay in the
// global record and take fire-and-forget additions (one thread, one address: applied in program order, so the sums are
// deterministic).  A count is stored twice in its word: as it is (low half) and as it was when its clock was last brought up
// to date (high half).  The time of that is also where its integral stands; the two decode buffers share one integral and
// have one more word for it.
enum { CQ_QP = 0, CQ_QD0 = 1, CQ_QD1 = 2, CQ_X = 3, CQ_YM = 4, CQ_YS = 5, CQ_N = 6 };       // the count of process k > 0 is k - 1

struct CtmcSim {
    const CtmcParams &p;
    unsigned long long *const base;   // this thread's word 0
    const uint32_t stride, I, per_class;      // per_class = ceil(2^16 / I): (e per_class) >> 16 = e / I for e < 56
    const double *const coef;         // [7 I] intensity per unit of the count (arrivals: per unit time), shared by the block
    CtmcRep &G;                       // the record in global memory: counters and integrals are added to in place
    uint8_t *const ring;              // [2][qcap]
    const uint32_t rep;
    uint32_t totX, totYm, totYs, err, head0, head1, n0, n1;
    unsigned long long dirty;         // processes whose count changed in this event (bit k I + i)

    __device__ CtmcSim(const CtmcParams &p_, unsigned long long *base_, uint32_t stride_, const double *coef_, CtmcRep &G_, uint32_t rep_)
        : p(p_), base(base_), stride(stride_), I(p_.I), per_class((65536u + p_.I - 1u) / p_.I), coef(coef_), G(G_), ring(p_.rings + (size_t)rep_ * 2 * p_.qcap), rep(rep_),
          totX(0), totYm(0), totYs(0), err(0), head0(0), head1(0), n0(0), n1(0), dirty(0) {}

    __host__ __device__ static uint32_t words(uint32_t I) { return 39u * I; }
    // word numbers; e = k I + i
    __device__ __forceinline__ uint32_t w_fire(uint32_t e) const { return e; }                       // 7 I
    __device__ __forceinline__ uint32_t w_draws(uint32_t e) const { return 7u * I + e; }             // 7 I
    __device__ __forceinline__ uint32_t w_acc(uint32_t e) const { return 13u * I + e; }              // e >= I: 6 I each
    __device__ __forceinline__ uint32_t w_lvl(uint32_t e) const { return 19u * I + e; }
    __device__ __forceinline__ uint32_t w_last(uint32_t e) const { return 25u * I + e; }
    __device__ __forceinline__ uint32_t w_count(uint32_t e) const { return 31u * I + e; }
    __device__ __forceinline__ uint32_t w_qd_last(uint32_t i) const { return 38u * I + i; }          // I
    __device__ __forceinline__ unsigned long long u(uint32_t w) const { return base[w * stride]; }
    __device__ __forceinline__ void su(uint32_t w, unsigned long long v) const { base[w * stride] = v; }
    __device__ __forceinline__ double d(uint32_t w) const { return __longlong_as_double((long long)u(w)); }
    __device__ __forceinline__ void sd(uint32_t w, double v) const { su(w, (unsigned long long)__double_as_longlong(v)); }

    __device__ __forceinline__ uint32_t stream_of(uint32_t k, uint32_t i) const
    {
        const uint32_t purpose = k < CK_SP ? k : k + 4u;      // 0..3 as in the iteration-level simulator, then 8, 9, 10
        return (purpose << 8) | i;
    }
    __device__ __forceinline__ uint4 rnd(uint32_t stream, unsigned long long index) const
    {
        return draw_words(p.seed, (uint32_t)(p.rep_offset + rep), stream, index);
    }
    __device__ __forceinline__ uint32_t cq(uint32_t c, uint32_t i) const { return (uint32_t)u(w_count((c + 1u) * I + i)); }
    __device__ __forceinline__ void bump(uint32_t i, uint32_t c) { atomicAdd(&G.cnt[i][c], 1ull); }
    // count c of class i changes by +1 or -1 (the low half of its word; a count is never negative)
    __device__ __forceinline__ void change(uint32_t c, uint32_t i, int by)
    {
        const uint32_t e = (c + 1u) * I + i, w = w_count(e);
        const unsigned long long v = u(w);
        su(w, (v & 0xffffffff00000000ull) | (uint32_t)((uint32_t)v + (uint32_t)by));
        dirty |= 1ull << e;
    }

    // Bring every changed count's process up to date at time t.  Process `fired` has just jumped: its hazard starts anew.
    __device__ __forceinline__ void commit(double t, uint32_t fired)
    {
#pragma unroll 1
        for (; dirty; dirty &= dirty - 1ull) {
            const uint32_t e = (uint32_t)__ffsll((long long)dirty) - 1u;
            const uint32_t k = (e * per_class) >> 16, i = e - k * I;
            const unsigned long long v = u(w_count(e));
            const uint32_t was = (uint32_t)(v >> 32), now = (uint32_t)v;
            const double dt = __dsub_rn(t, d(w_last(e))), c = coef[e];
            double part = __dmul_rn((double)was, dt);
            uint32_t a = k == CK_ABP ? CA_QP : (k == CK_SP ? CA_X : (k == CK_SDM ? CA_YM : CA_YS));
            if (k == CK_ABD0 || k == CK_ABD1) {
                a = CA_QD;
                const uint32_t both = (uint32_t)(u(w_count(CK_ABD0 * I + i)) >> 32) + (uint32_t)(u(w_count(CK_ABD1 * I + i)) >> 32);
                part = __dmul_rn((double)both, __dsub_rn(t, d(w_qd_last(i))));
                sd(w_qd_last(i), t);
            }
            atomicAdd(&G.area[a][i], part);
            double acc = 0.0;
            if (e != fired) acc = __dadd_rn(d(w_acc(e)), __dmul_rn(__dmul_rn(c, (double)was), dt));
            double tf = dinf();
            if (now > 0 && c > 0.0) {
                double rem = __dsub_rn(d(w_lvl(e)), acc);
                if (rem < 0.0) rem = 0.0;
                tf = __dadd_rn(t, __ddiv_rn(rem, __dmul_rn(c, (double)now)));
            }
            sd(w_acc(e), acc);
            sd(w_last(e), t);
            sd(w_fire(e), tf);
            su(w_count(e), ((unsigned long long)now << 32) | now);
        }
    }

    // Section 4.1 occupancy gate (xi_i = (X_i - n x*_i)/x*_i, ties to the largest Q_p,i - n q*_p,i) or the
    // Section 5.1.1 priority gate (smallest static rank); ties to the lowest class index
    __device__ __forceinline__ uint32_t gate_class() const
    {
        uint32_t best = NONE32;
        double bxi = 0.0, bdq = 0.0;
#pragma unroll 1
        for (uint32_t i = 0; i < I; ++i) {
            const uint32_t Qp = cq(CQ_QP, i);
            if (Qp == 0) continue;
            if (p.gate == 1) {
                if (best == NONE32 || p.cls[i].prio < p.cls[best].prio) best = i;
                continue;
            }
            if (!(p.cls[i].xstar > 0.0)) continue;
            const double xi = __ddiv_rn(__dsub_rn((double)cq(CQ_X, i), p.cls[i].nx), p.cls[i].xstar);
            const double dq = __dsub_rn((double)Qp, p.cls[i].nq);
            if (best == NONE32 || xi < bxi || (xi == bxi && dq > bdq)) { best = i; bxi = xi; bdq = dq; }
        }
        return best;
    }

    // tier that takes the head of the pool's buffer now: 0 solo, 1 mixed, 2 none has a free slot
    __device__ __forceinline__ uint32_t tier_of(uint32_t pool) const
    {
        const bool solo = totYs < (p.N - p.M) * p.B, mix = totYm < p.M * (p.B - 1u);
        if (p.router == 1) return pool ? (mix ? 1u : 2u) : (solo ? 0u : 2u);
        return solo ? 0u : (mix ? 1u : 2u);
    }
    __device__ __forceinline__ void place(uint32_t i, uint32_t tier)
    {
        change(tier ? CQ_YM : CQ_YS, i, 1);
        totYs += tier ? 0u : 1u; totYm += tier ? 1u : 0u;
        bump(i, tier ? CC_PLACED_MIXED : CC_PLACED_SOLO);
    }

    // The policy's turn after every event: buffered requests into free decode slots, then the prefill gate.
    __device__ __forceinline__ void dispatch()
    {
        uint32_t pool = 0;
#pragma unroll 1
        while (n0 | n1) {
            if (pool == 0 && n0 == 0) pool = 1;
            if (pool == 1 && n1 == 0) break;
            const uint32_t tier = tier_of(pool);
            if (tier == 2u) {
                if (pool == 1) break;
                pool = 1;
                continue;
            }
            uint32_t &head = pool ? head1 : head0;
            const uint32_t i = ring[pool * p.qcap + head];
            head = head + 1 == p.qcap ? 0 : head + 1;
            if (pool) --n1; else --n0;
            change(pool ? CQ_QD1 : CQ_QD0, i, -1);
            place(i, tier);
        }
#pragma unroll 1
        while (totX < p.M) {
            const uint32_t i = gate_class();
            if (i == NONE32) break;
            change(CQ_QP, i, -1);
            change(CQ_X, i, 1);
            ++totX;
            bump(i, CC_ADMITTED);
        }
    }

    // empty system at t = 0: every process gets its first level, the arrival processes their first jump time
    __device__ void init()
    {
        for (uint32_t w = 0; w < words(I); ++w) su(w, 0ull);
        for (uint32_t i = 0; i < I; ++i)
            for (uint32_t k = 0; k < CK_N; ++k) {
                const uint32_t e = k * I + i;
                const uint4 w = rnd(stream_of(k, i), 0);
                const double lvl = -qlog(u53(w.x, w.y));
                sd(w_fire(e), (k == CK_ARR && coef[e] > 0.0) ? __dadd_rn(0.0, __ddiv_rn(lvl, coef[e])) : dinf());
                su(w_draws(e), 1ull);
                if (k > 0) sd(w_lvl(e), lvl);
            }
    }

    // events with t <= T_end, at most `budget` of them; returns true when none is left up to T_end
    __device__ bool run(double T_end, unsigned long long budget, unsigned long long &events)
    {
        for (uint32_t i = 0; i < I; ++i) { totX += cq(CQ_X, i); totYm += cq(CQ_YM, i); totYs += cq(CQ_YS, i); }
        const uint32_t n_proc = CK_N * I;
        const unsigned long long tend_bits = (unsigned long long)__double_as_longlong(T_end);
        for (;;) {
            // earliest process; ties by process kind, then class (strict '<' in that scan order; the times are not negative)
            unsigned long long te = 0x7ff0000000000000ull;
            uint32_t e = 0;
#pragma unroll 7
            for (uint32_t q = 0; q < n_proc; ++q) {
                const unsigned long long tf = u(w_fire(q));
                if (tf < te) { te = tf; e = q; }
            }
            if (!(te <= tend_bits) || te == 0x7ff0000000000000ull) return true;
            if (budget == 0) return false;
            --budget;
            const double t = __longlong_as_double((long long)te);
            const uint32_t k = (e * per_class) >> 16, i = e - k * I;
            ++events;
            // the process's next level
            const unsigned long long m = u(w_draws(e));
            su(w_draws(e), m + 1);
            const uint4 w = rnd(stream_of(k, i), m);
            const double lvl = -qlog(u53(w.x, w.y));
            uint32_t c = k - 1u, cc = CC_ABANDONED_D;
            if (k == CK_ARR) {
                c = CQ_QP; cc = CC_ARRIVALS;
                sd(w_fire(e), __dadd_rn(t, __ddiv_rn(lvl, coef[e])));
            } else {
                sd(w_lvl(e), lvl);
                cc = k == CK_ABP ? CC_ABANDONED_P : (k == CK_SP ? CC_PREFILL_DONE : (k == CK_SDM ? CC_DONE_MIXED : (k == CK_SDS ? CC_DONE_SOLO : CC_ABANDONED_D)));
            }
            if (k == CK_ABD0 || k == CK_ABD1) {
                // a uniformly chosen waiting class-i request leaves the pool's buffer; the rest keep their order
                const uint32_t pool = k == CK_ABD1 ? 1u : 0u;
                uint8_t *r = ring + pool * p.qcap;
                uint32_t rank = __umulhi(w.z, cq(c, i)), pos = 0;
                const uint32_t n = pool ? n1 : n0, head = pool ? head1 : head0;
                for (pos = 0; pos < n; ++pos) {
                    uint32_t a = head + pos; if (a >= p.qcap) a -= p.qcap;
                    if (r[a] != i) continue;
                    if (rank == 0) break;
                    --rank;
                }
                if (pos >= n) { err = ERR_INTERNAL; return true; }
                for (uint32_t q = pos; q + 1 < n; ++q) {
                    uint32_t a = head + q, b = head + q + 1;
                    if (a >= p.qcap) a -= p.qcap;
                    if (b >= p.qcap) b -= p.qcap;
                    r[a] = r[b];
                }
                if (pool) --n1; else --n0;
            }
            change(c, i, k == CK_ARR ? 1 : -1);
            bump(i, cc);
            totX -= k == CK_SP ? 1u : 0u; totYm -= k == CK_SDM ? 1u : 0u; totYs -= k == CK_SDS ? 1u : 0u;
            if (k == CK_SP) {
                uint32_t pool = 0;
                if (p.router == 1) {
                    // SLI-aware router: one uniform per finished prefill decides the pool (Section 5.2); its ordinal is the
                    // number of prefills of the class finished before
                    const uint4 z = rnd((STREAM_SLI << 8) | i, m - 1ull);
                    pool = u53(z.x, z.y) <= p.cls[i].ps ? 0u : 1u;
                }
                const uint32_t n = pool ? n1 : n0, tier = n == 0 ? tier_of(pool) : 2u;
                if (tier != 2u) {
                    place(i, tier);          // it passes through its empty buffer at this instant
                } else if (n >= p.qcap) {
                    bump(i, CC_OVERFLOW_D);
                } else {
                    uint32_t pos = (pool ? head1 : head0) + n; if (pos >= p.qcap) pos -= p.qcap;
                    ring[pool * p.qcap + pos] = (uint8_t)i;
                    if (pool) ++n1; else ++n0;
                    change(pool ? CQ_QD1 : CQ_QD0, i, 1);
                }
            }
            dispatch();
            commit(t, k == CK_ARR ? NONE32 : e);
        }
    }

    // the record in global memory <-> the working copy
    __device__ void load(const CtmcRep &S)
    {
        head0 = S.head[0]; head1 = S.head[1]; n0 = S.n[0]; n1 = S.n[1];
        for (uint32_t i = 0; i < I; ++i) {
            const uint32_t cnt[CQ_N] = { S.Qp[i], S.Qd[0][i], S.Qd[1][i], S.X[i], S.Ym[i], S.Ys[i] };
            for (uint32_t k = 0; k < CK_N; ++k) {
                const CtmcClk &q = S.clk[k][i];
                const uint32_t e = k * I + i;
                sd(w_fire(e), q.t_fire);
                su(w_draws(e), q.m);
                if (k == 0) continue;
                // the clock and the integral of a count are brought up to date together, but for a clock of intensity zero that an
                // earlier build saved: that one stood still, so the time is the integral's (the two buffers have w_qd_last for it)
                const double last = k == CK_ABP ? S.area_t[CA_QP][i] : (k == CK_SP ? S.area_t[CA_X][i] : (k == CK_SDM ? S.area_t[CA_YM][i]
                                  : (k == CK_SDS ? S.area_t[CA_YS][i] : q.t_last)));
                sd(w_acc(e), q.acc); sd(w_lvl(e), q.lvl); sd(w_last(e), last);
                su(w_count(e), ((unsigned long long)cnt[k - 1] << 32) | cnt[k - 1]);
            }
            sd(w_qd_last(i), S.area_t[CA_QD][i]);
        }
    }
    __device__ void store(CtmcRep &S) const
    {
        S.head[0] = head0; S.head[1] = head1; S.n[0] = n0; S.n[1] = n1;
        for (uint32_t i = 0; i < I; ++i) {
            for (uint32_t k = 0; k < CK_N; ++k) {
                CtmcClk &q = S.clk[k][i];
                const uint32_t e = k * I + i;
                q.t_fire = d(w_fire(e)); q.m = u(w_draws(e));
                if (k > 0) { q.acc = d(w_acc(e)); q.lvl = d(w_lvl(e)); q.t_last = d(w_last(e)); }
            }
            S.Qp[i] = cq(CQ_QP, i); S.X[i] = cq(CQ_X, i); S.Qd[0][i] = cq(CQ_QD0, i); S.Qd[1][i] = cq(CQ_QD1, i);
            S.Ym[i] = cq(CQ_YM, i); S.Ys[i] = cq(CQ_YS, i);
            S.area_t[CA_QP][i] = d(w_last(CK_ABP * I + i)); S.area_t[CA_X][i] = d(w_last(CK_SP * I + i)); S.area_t[CA_QD][i] = d(w_qd_last(i));
            S.area_t[CA_YM][i] = d(w_last(CK_SDM * I + i)); S.area_t[CA_YS][i] = d(w_last(CK_SDS * I + i));
        }
    }
};

// One thread per replication.  The replication's record lives in global memory between launches; a launch works on a
// copy in shared memory.  init != 0: start from the empty system at t = 0 (no events are processed).
__global__ void __launch_bounds__(32) qsim_ctmc_kernel(CtmcParams p)
{
    extern __shared__ __align__(16) unsigned long long ctmc_sm[];
    const uint32_t lanes = p.lanes, rep = blockIdx.x * lanes + threadIdx.x;
    double *coef = reinterpret_cast<double *>(ctmc_sm);      // [7 I], then the threads' words
    for (uint32_t e = threadIdx.x; e < CK_N * p.I; e += blockDim.x) {
        const uint32_t k = e / p.I, i = e - k * p.I;
        const CtmcClassPar &c = p.cls[i];
        coef[e] = k == CK_ARR ? __dmul_rn((double)p.N, c.lambda) : (k <= CK_ABD1 ? c.theta : (k == CK_SP ? c.mu_p : (k == CK_SDM ? c.mu_m : c.mu_s)));
    }
    __syncwarp();
    if (threadIdx.x >= lanes || rep >= p.R) return;
    CtmcRep &S = p.reps[rep];
    CtmcSim sim(p, ctmc_sm + CK_N * p.I + threadIdx.x, lanes, coef, S, rep);
    if (p.init) {
        uint32_t *w = reinterpret_cast<uint32_t *>(&S);
        for (uint32_t o = 0; o < sizeof(CtmcRep) / 4; ++o) w[o] = 0;
        sim.init();
        sim.store(S);
        S.done = 1;
        return;
    }
    if (S.err || (S.done && S.T_end == p.T_end)) return;
    sim.load(S);
    unsigned long long events = S.events;
    const bool finished = sim.run(p.T_end, p.event_budget, events);
    sim.store(S);
    S.events = events;
    S.T_end = p.T_end;
    S.err = sim.err;
    S.done = finished ? 1u : 0u;
    if (!finished) atomicAdd(p.not_done, 1u);
}

// The public statistics record of every replication, one warp each: counters as they are, time integrals closed at the end
// time (the host's formula, rounded the same).  first_err: lowest replication that stopped on an internal error.
// Memory-bound: about 190 bytes per class in use read and 1.2 KB written per replication.
__global__ void __launch_bounds__(128) qsim_ctmc_stats_kernel(const CtmcRep *reps, uint32_t R, uint32_t I, qsim_ctmc_rep_stats *out, uint32_t *first_err)
{
    const uint32_t r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31u;
    if (r >= R) return;
    const CtmcRep &S = reps[r];
    qsim_ctmc_rep_stats &o = out[r];
    const double T = S.T_end;
    for (uint32_t w = lane; w < MAXI * CC_N; w += 32u) o.cnt[w / CC_N][w % CC_N] = w < I * CC_N ? S.cnt[w / CC_N][w % CC_N] : 0ull;
    for (uint32_t w = lane; w < MAXI * CA_N; w += 32u) {
        const uint32_t i = w / CA_N, a = w % CA_N;
        uint32_t n = 0;
        double area = 0.0;
        if (i < I) {
            n = a == CA_QP ? S.Qp[i] : (a == CA_X ? S.X[i] : (a == CA_QD ? S.Qd[0][i] + S.Qd[1][i] : (a == CA_YM ? S.Ym[i] : S.Ys[i])));
            area = __dadd_rn(S.area[a][i], __dmul_rn((double)n, __dsub_rn(T, S.area_t[a][i])));
        }
        o.state[i][a] = n;
        o.area[i][a] = area;
    }
    if (lane < MAXI) o.reserved[lane] = 0;
    if (lane == 0) {
        o.events = S.events;
        o.T_elapsed = T;
        if (S.err) atomicMin(first_err, r);
    }
}

}  // namespace qsimdev

// ---------------------------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------------------------
namespace {

int ctmc_validate(const qsim_ctmc_config *cfg, const qsim_ctmc_class *cls)
{
    if (!cfg || !cls) return fail(QSIM_EINVAL, "null argument");
    if (cfg->size != sizeof(qsim_ctmc_config)) return fail(QSIM_EINVAL, "qsim_ctmc_config.size does not match this library");
    if (cfg->I < 1 || cfg->I > QSIM_MAXI || cfg->N < 1 || cfg->M > cfg->N || cfg->B < 1 || cfg->R < 1 || cfg->qcap < 1)
        return fail(QSIM_EINVAL, "need 1 <= I <= 8, N >= 1, M <= N, B >= 1, R >= 1, qcap >= 1");
    if ((uint64_t)cfg->N * cfg->B > 0x7fffffffull) return fail(QSIM_EINVAL, "N * B too large");
    if (cfg->gate > QSIM_GATE_PRIORITY || cfg->router > QSIM_ROUTER_SLI)
        return fail(QSIM_EINVAL, "the exponential-service model has the occupancy and priority gates and the solo-first and SLI routers");
    for (uint32_t i = 0; i < cfg->I; ++i) {
        const qsim_ctmc_class &c = cls[i];
        const double v[9] = { c.lambda, c.theta, c.mu_p, c.mu_m, c.mu_s, c.xstar, c.n_xstar, c.n_qpstar, c.p_solo };
        for (double x : v)
            if (!std::isfinite(x) || x < 0.0) return fail(QSIM_EINVAL, "class parameters must be finite and non-negative");
        if (!(c.mu_p > 0.0) || !(c.mu_m > 0.0) || !(c.mu_s > 0.0)) return fail(QSIM_EINVAL, "service rates must be positive");
        if (c.p_solo > 1.0) return fail(QSIM_EINVAL, "p_solo must lie in [0, 1]");
    }
    return QSIM_OK;
}

struct CtmcSections { size_t reps, rings, flag, total; };

CtmcSections ctmc_sections(const qsim_ctmc_config &c)
{
    CtmcSections s;
    size_t o = 0;
    s.reps = o; o = align256(o + (size_t)c.R * sizeof(CtmcRep));
    s.rings = o; o = align256(o + (size_t)c.R * 2 * c.qcap);
    s.flag = o; o = align256(o + 4);
    s.total = o;
    return s;
}

// One warp per block, its first `lanes` threads run a replication each.  A warp executes every path that any of its threads
// takes, so few replications are spread over more warps: the largest power of two that still gives CTMC_WARPS warps (fewer
// replications than that: one per warp).  Measured with the smaller code: n = 1000, R = 300: 104 -> 38 ms (32 -> 1 per warp), n = 50,
// R = 1000: 5.7 -> 2.3 (1), n = 200, R = 3000: 19.2 -> 11.8 (2), n = 1000, R = 8192: 62.6 -> 51.2 (8).
constexpr uint32_t CTMC_WARPS = 888;
int ctmc_launch_shape(const qsim_ctmc_config &c, uint32_t &lanes, size_t &smem)
{
    lanes = 32;
    while (lanes > 1u && c.R / lanes < CTMC_WARPS) lanes >>= 1;
    smem = ((size_t)lanes * CtmcSim::words(c.I) + CK_N * c.I) * 8;
    if (smem > 48u * 1024u)
        CUDA_TRY(cudaFuncSetAttribute(qsim_ctmc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    return QSIM_OK;
}

// The public records from a copy of the device records (3.8 KB each): for few replications, and for a device without room for the
// public records.  Forming them on the device means an allocation and its return, 0.45 ms whatever their number; host / device in ms:
// R = 64 0.12 / 0.53, 256 0.34 / 0.61, 1024 1.09 / 0.95, 4096 4.0 / 1.7.
constexpr uint32_t CTMC_STATS_ON_DEVICE = 768;
int ctmc_stats_on_host(const qsim_ctmc_config &cfg, const char *dev_reps, cudaStream_t st, qsim_ctmc_rep_stats *per_rep)
{
    std::vector<CtmcRep> reps(cfg.R);
    CUDA_TRY(cudaMemcpyAsync(reps.data(), dev_reps, reps.size() * sizeof(CtmcRep), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    for (uint32_t r = 0; r < cfg.R; ++r) {
        const CtmcRep &S = reps[r];
        if (S.err) return fail(QSIM_EOVERFLOW, "replication " + std::to_string(r) + " stopped on an internal error");
        qsim_ctmc_rep_stats &o = per_rep[r];
        std::memset(&o, 0, sizeof o);
        const double T = S.T_end;
        for (uint32_t i = 0; i < cfg.I; ++i) {
            for (int k = 0; k < CC_N; ++k) o.cnt[i][k] = S.cnt[i][k];
            const uint32_t state[5] = { S.Qp[i], S.X[i], S.Qd[0][i] + S.Qd[1][i], S.Ym[i], S.Ys[i] };
            for (int a = 0; a < CA_N; ++a) {
                o.state[i][a] = state[a];
                o.area[i][a] = S.area[a][i] + (double)state[a] * (T - S.area_t[a][i]);     // integral up to the end time
            }
        }
        o.events = S.events;
        o.T_elapsed = T;
    }
    return QSIM_OK;
}

int ctmc_params(const qsim_ctmc_config *cfg, const qsim_ctmc_class *cls, void *ws, size_t bytes, CtmcParams &p)
{
    int rc = ctmc_validate(cfg, cls);
    if (rc != QSIM_OK) return rc;
    const CtmcSections sec = ctmc_sections(*cfg);
    if (!ws) return fail(QSIM_EWORKSPACE, "workspace pointer is null");
    if (bytes < sec.total) return fail(QSIM_EWORKSPACE, "workspace too small: need " + std::to_string(sec.total) + " bytes");
    if ((reinterpret_cast<uintptr_t>(ws) & 255u) != 0) return fail(QSIM_EWORKSPACE, "workspace must be 256-byte aligned");
    std::memset(&p, 0, sizeof p);
    p.I = cfg->I; p.N = cfg->N; p.M = cfg->M; p.B = cfg->B; p.R = cfg->R; p.qcap = cfg->qcap; p.gate = cfg->gate; p.router = cfg->router;
    p.seed = cfg->seed; p.rep_offset = cfg->rep_offset; p.event_budget = 1ull << 26;
    for (uint32_t i = 0; i < cfg->I; ++i) {
        CtmcClassPar &c = p.cls[i];
        c.lambda = cls[i].lambda; c.theta = cls[i].theta; c.mu_p = cls[i].mu_p; c.mu_m = cls[i].mu_m; c.mu_s = cls[i].mu_s;
        c.xstar = cls[i].xstar; c.nx = cls[i].n_xstar; c.nq = cls[i].n_qpstar; c.ps = cls[i].p_solo; c.prio = cls[i].prio_rank;
    }
    char *base = static_cast<char *>(ws);
    p.reps = reinterpret_cast<CtmcRep *>(base + sec.reps);
    p.rings = reinterpret_cast<uint8_t *>(base + sec.rings);
    p.not_done = reinterpret_cast<uint32_t *>(base + sec.flag);
    return QSIM_OK;
}

}  // namespace

extern "C" {

int qsim_ctmc_workspace_bytes(const qsim_ctmc_config *cfg, size_t *bytes)
{
    if (!cfg || !bytes) return fail(QSIM_EINVAL, "null argument");
    if (cfg->size != sizeof(qsim_ctmc_config) || cfg->R < 1 || cfg->qcap < 1) return fail(QSIM_EINVAL, "bad qsim_ctmc_config");
    *bytes = ctmc_sections(*cfg).total;
    return QSIM_OK;
}

int qsim_ctmc_init(const qsim_ctmc_config *cfg, const qsim_ctmc_class *classes, void *dev_workspace, size_t bytes, void *cuda_stream)
{
    CtmcParams p;
    int rc = ctmc_params(cfg, classes, dev_workspace, bytes, p);
    if (rc != QSIM_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    p.init = 1;
    size_t smem = 0;
    rc = ctmc_launch_shape(*cfg, p.lanes, smem);
    if (rc != QSIM_OK) return rc;
    qsim_ctmc_kernel<<<(cfg->R + p.lanes - 1u) / p.lanes, 32, smem, st>>>(p);
    CUDA_TRY(cudaGetLastError());
    return QSIM_OK;
}

int qsim_ctmc_run_until(const qsim_ctmc_config *cfg, const qsim_ctmc_class *classes, void *dev_workspace, size_t bytes,
                        void *cuda_stream, double T_end, uint64_t *launches)
{
    CtmcParams p;
    int rc = ctmc_params(cfg, classes, dev_workspace, bytes, p);
    if (rc != QSIM_OK) return rc;
    if (!(T_end >= 0.0) || !std::isfinite(T_end)) return fail(QSIM_EINVAL, "T_end must be finite and non-negative");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    p.T_end = T_end;
    uint64_t n = 0;
    size_t smem = 0;
    rc = ctmc_launch_shape(*cfg, p.lanes, smem);
    if (rc != QSIM_OK) return rc;
    // a replication that used up its per-launch event budget is continued by further launches
    uint32_t flag = 1;
    for (int guard = 0; guard < 100000 && flag != 0; ++guard) {
        CUDA_TRY(cudaMemsetAsync(p.not_done, 0, 4, st));
        qsim_ctmc_kernel<<<(cfg->R + p.lanes - 1u) / p.lanes, 32, smem, st>>>(p);
        CUDA_TRY(cudaGetLastError());
        ++n;
        CUDA_TRY(cudaMemcpyAsync(&flag, p.not_done, 4, cudaMemcpyDeviceToHost, st));
        CUDA_TRY(cudaStreamSynchronize(st));
    }
    if (launches) *launches = n;
    if (flag != 0) return fail(QSIM_EOVERFLOW, "replications still unfinished after 100000 launches: the end time was not reached");
    return QSIM_OK;
}

int qsim_ctmc_stats(const qsim_ctmc_config *cfg, const void *dev_workspace, size_t bytes, void *cuda_stream, qsim_ctmc_rep_stats *per_rep)
{
    if (!cfg || !per_rep) return fail(QSIM_EINVAL, "null argument");
    if (cfg->size != sizeof(qsim_ctmc_config) || cfg->R < 1 || cfg->qcap < 1 || cfg->I < 1 || cfg->I > QSIM_MAXI) return fail(QSIM_EINVAL, "bad qsim_ctmc_config");
    const CtmcSections sec = ctmc_sections(*cfg);
    if (!dev_workspace || bytes < sec.total) return fail(QSIM_EWORKSPACE, "workspace missing or too small");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (cfg->R < CTMC_STATS_ON_DEVICE) return ctmc_stats_on_host(*cfg, static_cast<const char *>(dev_workspace) + sec.reps, st, per_rep);
    // the public records are formed on the device: a third of the bytes cross to the host, and nothing is left to do there
    const size_t out_bytes = (size_t)cfg->R * sizeof(qsim_ctmc_rep_stats);
    char *scratch = nullptr;
    if (cudaMallocAsync(reinterpret_cast<void **>(&scratch), out_bytes + 4, st) != cudaSuccess) {
        cudaGetLastError();
        return ctmc_stats_on_host(*cfg, static_cast<const char *>(dev_workspace) + sec.reps, st, per_rep);
    }
    uint32_t first_err = NONE32;
    cudaError_t e = cudaMemsetAsync(scratch + out_bytes, 0xff, 4, st);
    if (e == cudaSuccess) {
        qsim_ctmc_stats_kernel<<<(cfg->R + 3u) / 4u, 128, 0, st>>>(reinterpret_cast<const CtmcRep *>(static_cast<const char *>(dev_workspace) + sec.reps),
                                                                  cfg->R, cfg->I, reinterpret_cast<qsim_ctmc_rep_stats *>(scratch),
                                                                  reinterpret_cast<uint32_t *>(scratch + out_bytes));
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&first_err, scratch + out_bytes, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess && first_err == NONE32) e = cudaMemcpyAsync(per_rep, scratch, out_bytes, cudaMemcpyDeviceToHost, st);
    const cudaError_t ef = cudaFreeAsync(scratch, st);
    if (e == cudaSuccess) e = ef;
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return fail(QSIM_ECUDA, std::string("qsim_ctmc_stats: ") + cudaGetErrorString(e));
    if (first_err != NONE32) return fail(QSIM_EOVERFLOW, "replication " + std::to_string(first_err) + " stopped on an internal error");
    return QSIM_OK;
}

int qsim_ctmc_revenue(const qsim_ctmc_config *cfg, const qsim_ctmc_rep_stats *per_rep, const double *P, const double *D,
                      const double *prices, int separate, double *rate)
{
    if (!cfg || !per_rep || !P || !D || !prices || !rate) return fail(QSIM_EINVAL, "null argument");
    if (cfg->size != sizeof(qsim_ctmc_config) || cfg->I < 1 || cfg->I > QSIM_MAXI || cfg->N < 1) return fail(QSIM_EINVAL, "bad qsim_ctmc_config");
    for (uint32_t r = 0; r < cfg->R; ++r) {
        const qsim_ctmc_rep_stats &s = per_rep[r];
        if (!(s.T_elapsed > 0.0)) return fail(QSIM_ESTATE, "no simulated time has elapsed");
        double rev = 0.0;
        for (uint32_t i = 0; i < cfg->I; ++i) {
            const double done = (double)(s.cnt[i][CC_DONE_MIXED] + s.cnt[i][CC_DONE_SOLO]);
            const double paid_in = separate ? (double)s.cnt[i][CC_PREFILL_DONE] : done;       // separate charging credits the prompt at prefill completion
            rev += prices[0] * P[i] * paid_in + prices[1] * D[i] * done;
        }
        rate[r] = rev / ((double)cfg->N * s.T_elapsed);
    }
    return QSIM_OK;
}

}  // extern "C"
