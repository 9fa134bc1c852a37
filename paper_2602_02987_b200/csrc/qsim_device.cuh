// Device side of qsim: one warp simulates one replication.
//
// Look-ahead.  The end of an iteration on a simulated GPU touches nothing outside that GPU unless a request
// finishes its prefill there (it must be routed, and the gate admits the next one) or a decode ends while
// requests wait in a decode buffer (the freed slot must be refilled).  All other iteration ends are
// "local".  A request placed on a running GPU only joins at that GPU's next iteration boundary, and no
// iteration is shorter than tau_min = min(alpha_m, alpha_s).  So in every round the warp finds the next
// non-local event (time T_int) and the earliest running iteration end T_min, and every lane finishes, in
// parallel, the local iteration ends of its own GPUs that come before min(T_int, T_min + tau_min, T_end):
// each GPU has at most one such end, and nothing that happens in that window can change another GPU's
// batch.  Decode completions found on the way are then retired by the whole warp, GPU by GPU, and only
// after that is the non-local event handled by the warp-wide path.  The outcome is event for event that of
// the one-at-a-time order; only the order in which some sums are accumulated differs.
//
// Ownership inside the warp (no two lanes ever write the same word, so the only synchronisation is a
// few __syncwarp per event):
//   * lane i (< I) owns class i: its arrival clock, prefill queue cursor, abandonment clocks, counts,
//     time integrals and statistics (struct ClassState, in shared memory);
//   * lane l owns GPUs l, l+32, l+64, ...: their clocks and batch state (structure-of-arrays in shared
//     memory, staged from / to global memory at kernel entry / exit);
//   * scalars every lane needs (event time, block, buffer cursors, ordinals) are kept replicated in
//     registers and updated identically by all lanes.
// The next event is a warp-wide argmin over every lane's earliest source (three redux.sync on the bit
// pattern of the positive doubles plus the source id, which encodes the tie order).  Up to 128 GPUs a lane looks at all
// of its GPUs (unrolled rows); beyond, iteration ends come from a calendar (Sim::load_bucket) or, where an event comes with
// many local ends, from a scan of all rows.
//
// What bounds these kernels is the chain of dependent instructions of each replication and, with a dozen warps per SM at
// different places of the round loop, instruction fetch: a version of the calendar kernel with 153 KB of code ran 26 % slower
// than the same algorithm without the parts that made it grow (N = 512).  So rare work exists once (one abandonment handler, draws
// out of line, loops not unrolled), and the compiled loops are 55-100 KB where they were 80-240.  Decisions that look
// at all GPUs (least-loaded / k-th eligible GPU) are evaluated by the owners and reduced the same way.
//
// All clock arithmetic is IEEE double, one rounding per operation, never contracted (the file is also
// compiled with --fmad=false).
#pragma once

#include <cstddef>
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

namespace qsimdev {

constexpr int MAXI = 8;
constexpr int LMAX = 8192;
constexpr int NBIN = 1024;
constexpr unsigned FULL = 0xffffffffu;
constexpr uint32_t NONE32 = 0xffffffffu;
constexpr uint32_t CAL_LSH_NEAR = 2, CAL_LSH_FAR = 1;       // lists per bucket of the calendar (by GPU index), binary logarithm; F_FAR: where memory on chip counts
constexpr uint32_t CAL_NONE = 0xffffu;   // end of a list
constexpr uint32_t BATCH_MASK = 0x1fffu, BATCH_MIXED = 0x2000u;   // nact: decodes in the batch (B <= 4096), the iteration processes prompt tokens (CAL)
// Rounds per launch.  Counters of a launch have 32 bits where a lane ends at most four iterations of its own and one more in a round (the
// calendar, unrolled rows); where it ends one for each of up to 128 rows, the iteration counters have 64 (Sim::IterCount).
constexpr unsigned long long BUDGET_MAX = 1ull << 29;
constexpr int ARRIVALS_PER_ROUND = 64;    // arrivals of a class that one round takes (a trace may bring any number at one time)
constexpr uint32_t CAL_FREE = 16;        // free lanes from which the calendar loads another bucket

// Compile-time specialisation of the run kernel.  With F_GENERIC every mode is read from the parameters at
// run time; otherwise the set bits say which features the instance contains and everything else is
// compiled out.  SPL > 0 fixes the number of simulated GPUs per lane (N <= 32 SPL) so the per-GPU loops unroll.
constexpr uint32_t F_GENERIC = 1, F_ABANDON = 2, F_SLI = 4, F_KAPPA = 8, F_HIST = 16, F_BLOCKS = 32, F_RANDOM = 64,
                   F_OCC = 128, F_SLOTS = 256, F_MW = 512, F_FCFS = 1024, F_SLIG = 2048, F_IMM = 4096, F_SCAN = 8192, F_INJECT = 16384, F_FAR = 32768,
                   F_TIGHT = 65536;
// F_SCAN (run-time row count): rounds read all GPUs instead of working from the calendar of iteration ends.
// F_FAR (calendar): the records of the GPUs stay in global memory (L2); on chip are only the calendar and what a choice among
// the GPUs reads.  More replications are resident on an SM, each somewhat slower.
// F_TIGHT (calendar): the shortest iteration is shorter than a bucket.
// F_MW: several warps per replication.  Warp 0 (the master) runs the round loop and every event handler; the
// other warps (helpers) wait at a block barrier for commands and take their share of the per-GPU work of a
// round: rows r = warp, warp + W, ... of the candidate scan and of the local iteration ends / retirements.
enum { MW_SCAN = 1, MW_ENDS = 2, MW_EXIT = 3 };
struct MwCmd { unsigned long long lim_t; uint32_t op, lim_s, buffered, M, force, pad; };
struct MwRes { unsigned long long bt, tmin; uint32_t bs, progressed; };
constexpr int MW_MAX = 16;

// source ids: smaller id wins an exact tie in time
constexpr uint32_t SRC_BLOCK = 0, SRC_ARRIVAL = 1, SRC_ABP = 9, SRC_ABD0 = 17, SRC_ABD1 = 25, SRC_SERVER = 33;

enum { STREAM_ARRIVAL = 0, STREAM_ABANDON_P = 1, STREAM_ABANDON_D0 = 2, STREAM_ABANDON_D1 = 3,
       STREAM_PLACEMENT = 4, STREAM_SLI = 5, STREAM_SELECT0 = 6, STREAM_SELECT1 = 7 };
enum { WANT_SOLO = 1, WANT_MIX = 2, WANT_PREFILL = 4 };
enum { ERR_NONE = 0, ERR_INTERNAL = 1 };

struct AbClock { double acc, lvl, t_last, t_ab; unsigned long long m; };
struct Area { double area, t_last; };

struct ClassState {
    double ta;
    unsigned long long adraw, sli_ord;
    uint32_t ablk, nextP, nextD, pq_head, pq_n, X, Ym, Ys, Qd0, Qd1, pq_tail, pq_pad;   // pq_tail: one-thread-per-replication kernels
    AbClock abp, abd0, abd1;
    Area aQp, aX, aQd;
    double sYm_in, sYm_out, sYs_in, sYs_out;   // sums of (placement / completion time - T_reset): integral of Y = out - in + Y (T - T_reset)
    unsigned long long arrivals, admitted, prefill_done, placed_mixed, placed_solo, done_mixed, done_solo,
        abandoned_p, abandoned_d, overflow, overflow_d, tok_in_pf, tok_in_done, tok_out_done;
    double sum_ttft, sum_tpot;
};

struct RepHeader {
    double T_end, T_reset;
    unsigned long long place_ord, events, H_total, rounds;
    uint32_t blk, done, err, force;    // force: the next event must be followed by a dispatch (targets were replaced)
    double t_now;                      // time of the last event handled (one-thread-per-replication kernels)
    uint32_t seq, chunks_left;         // launches that split the horizon into chunks: hand-over stamp of the last chunk done, chunks not started yet
    uint32_t dq_head0, dq_head1, dq_n0, dq_n1;
    unsigned long long sel_ord0, sel_ord1;   // class selections drawn so far in the solo / mixed pool (general SLI router)
    unsigned long long iters_mixed[32], iters_solo[32];
    double busy_mixed[32], busy_solo[32];
    ClassState cs[MAXI];
};

static_assert(sizeof(ClassState) % 8 == 0 && (sizeof(ClassState) * MAXI) % 16 == 0, "ClassState is copied in 16-byte words");
static_assert(sizeof(RepHeader) % 16 == 0 && offsetof(RepHeader, cs) % 16 == 0, "RepHeader layout");

struct SlotRec { double tpf; uint32_t pk; uint32_t pad; };  // request in a decode slot: prefill end time, packed lengths/class/group
constexpr int STAGE_CAP = 64, ROW_STAGE_CAP = 32;              // finished-request records waiting for their accounting (stamps on chip / in global memory)
// Accounting of finished requests, one block per warp (merged into the class records at kernel exit)
struct WarpClassStats { double sYm_out, sYs_out, sum_tpot; unsigned long long tok_in, tok_out; uint32_t done_mixed, done_solo; };
struct ClassAim { double xstar, nx, nq, ps, theta; };       // LP targets, share of the solo pool and abandonment rate of a class
struct ADraw { double E; uint32_t pk; uint32_t pad; };     // one arrival draw: interarrival time (unit exponential over the rate) and packed lengths
struct QEntry { double t; uint32_t pk; uint32_t cls; };   // 16 bytes: prefill queue (t = arrival) / decode buffer (t = prefill end)

struct ClassPar { double theta; uint32_t P, D, prio, pad; };
struct BlockPar { uint32_t M, pad; double xstar[MAXI], nx[MAXI], nq[MAXI], ps[MAXI], rate[MAXI], ws[MAXI], wm[MAXI]; };

// Shapes and arrays of the one-thread-per-replication family (qsim_lane.cuh); arrays are [R][...]
struct LaneSrv;
struct LanePar {
    uint32_t on;                 // this handle runs that family
    uint32_t nbk;                // calendar buckets (power of two); every pending iteration end lies less than nbk buckets ahead
    uint32_t tlev, toff[6], tsize;   // eligibility trees: internal levels, offset of every level (0 = leaves) and entries per tree
    uint32_t b8, slev, soff[5], ssize;   // slot trees: leaves per GPU, internal levels, offsets of levels 1.. and nodes per GPU
    double inv_w;                // buckets per second
    uint32_t cs_stride, smem_bytes;  // shared memory per lane for the class records (32-bit words) and per block of 1 << lsh lanes (bytes)
    LaneSrv *srv;                // [N] GPU records
    double *tarr;                // [N] arrival time of the request in prefill
    uint16_t *cal_head;          // [nbk] first GPU of every bucket
    uint32_t *cal_bm;            // [nbk/32] non-empty buckets
    uint32_t *tree;              // [3][tsize] solo decode, mixed decode, prefill
    uint32_t *sfin;              // [N][b8] finish iteration per slot (NONE32 = free)
    unsigned long long *snode;   // [N][ssize] minimum of finish << 16 | slot per group of eight
    SlotRec *srec;               // [N][B] request in each slot
    uint16_t *sfree;             // [N][B] entries at and above the GPU's decode count are its free slots
    uint32_t *pql;               // [I][qw] live bits of the prefill-queue positions
    uint32_t qw, lsh;            // words per class in pql (a multiple of four); a warp runs 1 << lsh replications in its first lanes
};

struct Params {
    uint32_t I, N, Npad, R, B, C, nblk, gate, router, placement, length_mode, qcap, hist, advance, any_theta, slots_smem;
    unsigned long long seed, rep_offset, horizon_iters, event_budget;
    double block_len;
    double coef[6];
    ClassPar cls[MAXI];
    const BlockPar *blocks;      // [nblk]
    const uint32_t *lengths;     // [I][2][LMAX] or null
    const double *inject_t;      // injected arrivals (trace replay): times [n_inject], ascending
    const uint32_t *inject_job;  // [n_inject][3] = class, P, D
    uint32_t n_inject, force_dispatch;   // force_dispatch: the policy parameters changed since the last launch
    uint32_t nchunk, launch_tag;         // nchunk > 1: the horizon of this launch is run in that many chunks per replication (see qsim_run_kernel)
    double T_abs;                // advance == 2: absolute end time of this run
    // workspace sections (all arrays are [R][...])
    RepHeader *hdr;
    char *srv;                   // per replication: server structure-of-arrays image, srv_bytes each
    uint32_t *slot_fin;          // [R][N][B]
    SlotRec *slot_rec;           // [R][N][B]
    QEntry *pq;                  // [R][I][qcap]
    QEntry *dq;                  // [R][2][qcap]
    uint32_t *hist_mem;          // [R][I][2][NBIN] or null
    uint32_t *not_done;          // [0] replications that stopped on the event budget, [1] next (chunk, replication) unit to hand out,
                                 // [2] set when a block gave up waiting for the chunk before its own
    uint32_t srv_bytes;
    uint32_t tarr_global;        // pf_tarr lives in tarr_g instead of shared memory
    double *tarr_g;              // [R][N]
    uint32_t *pfjob_g;           // [R][N] packed request in prefill, with tarr_g
    double cal_inv_w;            // calendar of iteration ends (run-time row count, one warp): buckets per second
    uint32_t cal_nbk, cal_K;     // buckets (a power of two); buckets that the shortest iteration lasts at least (0: F_TIGHT)
    uint32_t cal_lsh;            // binary logarithm of the lists per bucket
    LanePar lane;
};

// ---------------------------------------------------------------------------------------------
// random numbers and elementary functions
// ---------------------------------------------------------------------------------------------

// Philox4x32-10 (Salmon et al., SC'11): counter (c0..c3), key (k0,k1).
__device__ __forceinline__ void philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1,
                                       uint32_t &o0, uint32_t &o1, uint32_t &o2, uint32_t &o3)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        c0 = hi1 ^ c1 ^ k0;
        c1 = lo1;
        c2 = hi0 ^ c3 ^ k1;
        c3 = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    o0 = c0; o1 = c1; o2 = c2; o3 = c3;
}

__device__ __forceinline__ void draw(const Params &p, uint32_t rep, uint32_t stream, unsigned long long index,
                                     uint32_t &w0, uint32_t &w1, uint32_t &w2, uint32_t &w3)
{
    const unsigned long long grep = p.rep_offset + rep;
    philox((uint32_t)index, (uint32_t)(index >> 32), stream, (uint32_t)grep, (uint32_t)p.seed,
           (uint32_t)(p.seed >> 32), w0, w1, w2, w3);
}
// The same out of line, for rare draws: the kernels' round loops are about as large as the instruction cache.
__device__ __noinline__ uint4 draw_words(unsigned long long seed, uint32_t global_rep, uint32_t stream, unsigned long long index)
{
    uint4 w;
    philox((uint32_t)index, (uint32_t)(index >> 32), stream, global_rep, (uint32_t)seed, (uint32_t)(seed >> 32), w.x, w.y, w.z, w.w);
    return w;
}
__device__ __forceinline__ void draw_rare(const Params &p, uint32_t rep, uint32_t stream, unsigned long long index,
                                          uint32_t &w0, uint32_t &w1, uint32_t &w2, uint32_t &w3)
{
    const uint4 w = draw_words(p.seed, (uint32_t)(p.rep_offset + rep), stream, index);
    w0 = w.x; w1 = w.y; w2 = w.z; w3 = w.w;
}

// uniform on (0,1]: (top 53 bits of w0:w1, plus one) / 2^53
__device__ __forceinline__ double u53(uint32_t w0, uint32_t w1)
{
    const unsigned long long h = ((unsigned long long)w0 << 21) | (unsigned long long)(w1 >> 11);
    return __dmul_rn((double)(h + 1ull), 1.1102230246251565e-16);   // 2^-53
}

// ln x for x in (0,1] as a fixed chain of rounded operations: x = m 2^e, m in [sqrt(1/2), sqrt(2)),
// s = (m-1)/(m+1), ln m = 2 s sum_{k=0..12} s^(2k)/(2k+1), result = e ln2 + ln m.
__device__ __forceinline__ double qlog(double x)
{
    const long long bits = __double_as_longlong(x);
    int e = (int)((bits >> 52) & 0x7ff) - 1023;
    double m = __longlong_as_double((bits & 0x000fffffffffffffLL) | 0x3ff0000000000000LL);
    if (m > 1.4142135623730951) {
        m = __dmul_rn(m, 0.5);
        e += 1;
    }
    const double s = __ddiv_rn(__dsub_rn(m, 1.0), __dadd_rn(m, 1.0));
    const double z = __dmul_rn(s, s);
    // series coefficients 1/(2k+1): the correctly rounded quotients, formed once at compile time
    constexpr double inv_odd[13] = { 1.0 / 1.0, 1.0 / 3.0, 1.0 / 5.0, 1.0 / 7.0, 1.0 / 9.0, 1.0 / 11.0, 1.0 / 13.0, 1.0 / 15.0,
                                     1.0 / 17.0, 1.0 / 19.0, 1.0 / 21.0, 1.0 / 23.0, 1.0 / 25.0 };
    double acc = inv_odd[12];
#pragma unroll
    for (int k = 11; k >= 0; --k)
        acc = __dadd_rn(__dmul_rn(acc, z), inv_odd[k]);
    const double logm = __dmul_rn(__dmul_rn(2.0, s), acc);
    return __dadd_rn(__dmul_rn((double)e, 0.6931471805599453), logm);
}

// unit exponential from two words, out of line for rare draws
__device__ __noinline__ double unit_exp(uint32_t w0, uint32_t w1) { return -qlog(u53(w0, w1)); }

// iteration time of a batch with pf prefill tokens, d decodes, K resident KV tokens (Eq. (1)-(3))
__device__ __forceinline__ double iter_time(const Params &p, uint32_t pf, uint32_t d, uint32_t K, bool kappa = true)
{
    double t;
    if (pf > 0) {
        t = __dadd_rn(p.coef[0], __dmul_rn(p.coef[1], (double)pf));
        t = __dadd_rn(t, __dmul_rn(p.coef[2], (double)d));
    } else {
        t = __dadd_rn(p.coef[3], __dmul_rn(p.coef[4], (double)d));
    }
    if (kappa && p.coef[5] != 0.0)
        t = __dadd_rn(t, __dmul_rn(p.coef[5], (double)K));
    return t;
}

__device__ __forceinline__ uint32_t hist_bin(double x)
{
    long long b = (long long)((unsigned long long)__double_as_longlong(x) >> 47) - ((long long)(1023 - 20) << 5);
    b = b < 0 ? 0 : (b > NBIN - 1 ? NBIN - 1 : b);
    return (uint32_t)b;
}

__device__ __forceinline__ uint32_t pack_job(uint32_t P, uint32_t D, uint32_t cls, uint32_t flag)
{
    return (P - 1u) | ((D - 1u) << 13) | (cls << 26) | (flag << 31);
}
__device__ __forceinline__ uint32_t job_P(uint32_t pk) { return (pk & 0x1fffu) + 1u; }
__device__ __forceinline__ uint32_t job_D(uint32_t pk) { return ((pk >> 13) & 0x1fffu) + 1u; }
__device__ __forceinline__ uint32_t job_cls(uint32_t pk) { return (pk >> 26) & 7u; }
__device__ __forceinline__ uint32_t job_flag(uint32_t pk) { return pk >> 31; }

__device__ __forceinline__ double dinf() { return __longlong_as_double(0x7ff0000000000000LL); }

__device__ __forceinline__ void area_touch(Area &a, uint32_t count, double t)
{
    a.area = __dadd_rn(a.area, __dmul_rn((double)count, __dsub_rn(t, a.t_last)));
    a.t_last = t;
}

// Abandonment clock of one (class, queue): integrated hazard acc against the exponential level lvl
// (random time change, Eq. (8)-(9)); brought up to date by the owning class lane before the count changes.  The time at
// which the level is reached with the new count costs a division; Sim::settle_queue forms it where it is next asked for.
__device__ __forceinline__ void ab_touch(AbClock &c, double theta, uint32_t Q_old, double t)
{
    c.acc = __dadd_rn(c.acc, __dmul_rn(__dmul_rn(theta, (double)Q_old), __dsub_rn(t, c.t_last)));
    c.t_last = t;
}
// Next abandonment with Q waiting requests, from the state of the clock at its last change.
__device__ __forceinline__ double ab_next(const AbClock &c, double theta, uint32_t Q)
{
    double rem = __dsub_rn(c.lvl, c.acc);
    if (rem < 0.0) rem = 0.0;
    return Q > 0 ? __dadd_rn(c.t_last, __ddiv_rn(rem, __dmul_rn(theta, (double)Q))) : dinf();
}
// The two together, where the next time is wanted at once (one thread per replication).
__device__ __forceinline__ void ab_change(AbClock &c, double theta, uint32_t Q_old, uint32_t Q_new, double t)
{
    if (!(theta > 0.0)) return;
    ab_touch(c, theta, Q_old, t);
    c.t_ab = ab_next(c, theta, Q_new);
}
// Out of line for the warp kernels, where it is rarely asked for (see Sim::next_abandonment).
__device__ __noinline__ double ab_next_call(const AbClock &c, double theta, uint32_t Q) { return ab_next(c, theta, Q); }

// 16-byte asynchronous copy global -> shared (L2 only), and the wait for this thread's copies
__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gsrc)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
// Copies are committed one group per copy, so a thread can wait for an older copy of its own and leave the
// N groups it committed after it in flight.
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N_>
__device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N_) : "memory"); }

// Coarse index of a threshold table: entry b = #{j < LMAX-1 : thr[j] < b 2^24}, b = 0..256 (built by the host when the
// tables are uploaded and stored behind them).  A word w with top byte b has its count between entries b and b+1.
constexpr int LIDX = 260;       // 257 entries, padded

// 1 + #{j < LMAX-1 : thr[j] <= w} by binary search inside the bucket of w's top byte
__device__ __forceinline__ uint32_t table_lookup(const uint32_t *thr, const uint16_t *idx, uint32_t w)
{
    const uint32_t b = w >> 24;
    uint32_t lo = __ldg(idx + b), hi = __ldg(idx + b + 1);          // the count lies in [lo, hi]
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__ldg(thr + mid) <= w) lo = mid + 1; else hi = mid;
    }
    return 1u + lo;
}

// Arrival draw `index` of class i: one Philox block gives the unit exponential and both lengths.
// (Arguments by value: a reference to the kernel parameters would force a local copy of them.)
__device__ __noinline__ ADraw make_draw(unsigned long long seed, unsigned long long global_rep, uint32_t i, uint32_t I,
                                        unsigned long long index, const uint32_t *tables, uint32_t P, uint32_t D, double Lam)
{
    uint32_t w0, w1, w2, w3;
    philox((uint32_t)index, (uint32_t)(index >> 32), (STREAM_ARRIVAL << 8) | i, (uint32_t)global_rep, (uint32_t)seed,
           (uint32_t)(seed >> 32), w0, w1, w2, w3);
    ADraw d;
    d.E = -qlog(u53(w0, w1));
    if (Lam > 0.0) d.E = __ddiv_rn(d.E, Lam);      // one rate for the whole run: the interarrival time itself is stored
    if (tables) {
        const uint16_t *idx = reinterpret_cast<const uint16_t *>(tables + (size_t)I * 2 * LMAX);     // behind the tables
        P = table_lookup(tables + ((size_t)i * 2 + 0) * LMAX, idx + ((size_t)i * 2 + 0) * LIDX, w2);
        D = table_lookup(tables + ((size_t)i * 2 + 1) * LMAX, idx + ((size_t)i * 2 + 1) * LIDX, w3);
    }
    d.pk = pack_job(P, D, i, 0);
    d.pad = 0;
    return d;
}

// ---------------------------------------------------------------------------------------------
// the per-warp simulator
// ---------------------------------------------------------------------------------------------

template <int SPL, uint32_t F>
struct Sim {
    // One warp and a run-time row count: iteration ends come from a calendar (load_bucket) instead of a scan of all GPUs,
    // except in the F_SCAN instances.
    static constexpr bool CAL = SPL == 0 && !(F & (F_MW | F_SCAN));
    static constexpr bool FAR = CAL && (F & F_FAR) != 0;
    static constexpr bool TIGHT = CAL && (F & F_TIGHT) != 0;
    __device__ __forceinline__ uint32_t cal_lsh() const { return (F & (F_GENERIC | F_TIGHT)) ? p.cal_lsh : (FAR ? CAL_LSH_FAR : CAL_LSH_NEAR); }
    __device__ __forceinline__ uint32_t cal_lists() const { return p.cal_nbk << cal_lsh(); }
    static constexpr bool STAGED = !(F & F_MW);      // one warp: finished requests are accounted 32 at a time
    using IterCount = std::conditional_t<SPL == 0 && !CAL, unsigned long long, uint32_t>;      // (see BUDGET_MAX)
    __device__ __forceinline__ bool f_abandon() const { return (F & F_GENERIC) ? p.any_theta != 0 : (F & F_ABANDON) != 0; }
    __device__ __forceinline__ bool f_sli() const { return (F & F_GENERIC) ? (p.router == 1 || p.router == 2) : (F & F_SLI) != 0; }
    __device__ __forceinline__ bool f_slig() const { return (F & F_GENERIC) ? p.router == 2 : false; }
    __device__ __forceinline__ bool f_kappa() const { return (F & F_GENERIC) ? p.coef[5] != 0.0 : (F & F_KAPPA) != 0; }
    __device__ __forceinline__ bool f_hist() const { return (F & F_GENERIC) ? hist != nullptr : (F & F_HIST) != 0; }
    __device__ __forceinline__ bool f_blocks() const { return (F & F_GENERIC) ? p.nblk > 1 : (F & F_BLOCKS) != 0; }
    __device__ __forceinline__ bool f_random() const { return (F & F_GENERIC) ? p.placement == 0 : (F & F_RANDOM) != 0; }
    __device__ __forceinline__ bool f_occ() const { return (F & F_GENERIC) ? p.gate == 0 : (F & F_OCC) != 0; }
    // finish stamps and slot occupancy of every simulated GPU live in shared memory (small N*B only)
    __device__ __forceinline__ bool f_slots() const { return (F & F_GENERIC) ? p.slots_smem != 0 : (F & F_SLOTS) != 0; }
    __device__ __forceinline__ uint32_t n_rows() const { return SPL > 0 ? (uint32_t)SPL : (p.Npad >> 5); }

    const Params &p;
    const int lane;
    const uint32_t rep;
    int warp, nwarps;            // position in the block (F_MW); 0 / 1 otherwise
    MwCmd *cmd;
    MwRes *res;
    WarpClassStats *wcs;         // [nwarps][I]
    // shared memory (lane-owned entries)
    double *tnext, *pf_tarr;               // pf_tarr: arrival time of the request in prefill (shared memory, or global memory on large clusters)
    uint32_t *it, *nfin, *pfjob, *K, *Kpend;
    uint16_t *pfrem;             // prompt tokens still to prefill (0 = no request in prefill; lengths are at most 8192)
    uint16_t *ndec, *nact, *pfcur;
    uint16_t *sfin16;            // [Npad][B]  low 16 bits of each slot's finish iteration (f_slots)
    uint32_t *socc;              // [Npad][ceil(B/32)]  slot occupancy bits; bits past B are set for good
    uint32_t *cal_head;          // [buckets][1 << cal_lsh] first GPU of every list of the calendar (CAL)
    uint16_t *cal_next;          // [GPUs] the GPU after this one in its list (CAL)
    uint16_t *picked;            // [32] GPUs of the bucket being loaded (CAL)
    uint32_t *row_key;           // [3][rows] smallest key of every row of 32 GPUs (CAL, see choose())
    ClassState *cs;
    // global memory of this replication
    uint32_t *s_fin;
    SlotRec *s_rec;
    // shared-memory staging: records of finished requests (copied asynchronously) and queue-head copies
    SlotRec *st_rec;
    double *st_te;
    QEntry *pqh;
    uint32_t n_pend;
    double late_tpf;             // lane 0: record of the request that finished last, on its way from memory (entry n_pend of the staged ones)
    uint32_t late_pk;
    bool has_late;
    uint32_t rec_after;          // per lane: record copies committed since this lane's last queue-head copy
    QEntry *pq, *dq;
    uint32_t *hist;
    // replicated scalars
    double t, T_end, T_blk_next, tau_min;
    const double *T_reset_at;     // (in shared memory, like all that is not read in every round)
    uint32_t blk, M, dq_head0, dq_head1, dq_n0, dq_n1, n_touch, err;
    uint32_t n_idle_pf;          // mixed GPUs whose prefill slot is idle (and that may take a prefill)
    uint32_t idle_hint;          // when n_idle_pf == 1: that GPU if known, else NONE32
    uint32_t need_start;         // per lane: rows of own GPUs touched by the current event
    uint32_t touch_g;            // run-time row count: GPU touched by the current event (lanes below n_touch)
    uint32_t events, rounds;     // of this launch
    unsigned long long place_ord, sel_ord0, sel_ord1;
    bool drain_dirty, gate_dirty, touch_all;
    bool handed;                 // a request has just finished its prefill: class and lengths, pool, its arrival time, and the
    uint32_t d_pk, d_pool, d_gpu;   // GPU it has to decode on (NONE32: the router chooses)
    double d_tarr;
    bool direct;                 // its pool's buffer is empty: it may pass through
    uint32_t stale;              // class lane: abandonment clocks (prefill queue, decode buffers) whose next time is out of date
    uint32_t pools;              // class lane: pools of 32 finished prefills (SLI-aware routers)
    bool pools_due;              // and whether they have to be drawn
    unsigned long long place_base;  // placement draws held by the lanes: ordinal of lane 0's, and the word of this lane's
    uint32_t place_w;
    bool force_nonlocal;         // treat the next event, whatever it is, as non-local (it must end with a dispatch)
    // calendar: last bucket loaded, the pending iteration end that this lane holds (GPU, time)
    unsigned long long cur, held_t;
    uint32_t held_g;
    uint32_t held_na;            // its batch word
    uint32_t held_pk;            // the request whose prefill that end finishes: packed lengths and class, and arrival time
    double held_tarr;
    bool held, crowded;          // crowded: the current bucket holds more ends than lanes
    uint32_t lead;               // no pending event lies more than this many buckets before `cur`
    unsigned long long *left;    // crowded: earliest pending end of the bucket that no lane holds (time, source), in shared memory
    uint32_t dirty_dec, dirty_pf;   // bit k: the keys of row lane + 32 k are out of date (decode / prefill targets)
    // per-lane partial sums
    IterCount it_mixed, it_solo;
    double busy_mixed, busy_solo;
    // pre-generated arrival draws of this lane's class (ring in shared memory) and a pending scheduling request
    double *aring;
    uint32_t *aring_pk;
    uint32_t ring_n, ring_pos;
    bool sched_pending;
    uint32_t ring_blk;           // block whose rate the draws are divided by, and its end
    double ring_end;
    ClassAim *aim;               // [I] parameters of the classes in the current block

    __device__ Sim(const Params &p_, int lane_, uint32_t rep_) : p(p_), lane(lane_), rep(rep_), warp(0), nwarps(1) {}
    __device__ __forceinline__ void block_sync() const { if (F & F_MW) __syncthreads(); else __syncwarp(); }

    __device__ __forceinline__ double block_start(uint32_t b) const { return __dmul_rn((double)b, p.block_len); }

    __device__ __forceinline__ void load_block(uint32_t b)
    {
        blk = b;
        const BlockPar &bp = p.blocks[b];
        M = bp.M;
        dirty_dec = dirty_pf = 0;
        if (CAL)
            for (uint32_t k = 0; ((k << 5) + (uint32_t)lane) < n_rows(); ++k) dirty_dec = dirty_pf |= 1u << k;
        pools_due = f_sli() && lane < (int)p.I;
        if (lane < (int)p.I) {
            ClassAim a;
            a.xstar = bp.xstar[lane]; a.nx = bp.nx[lane]; a.nq = bp.nq[lane]; a.ps = bp.ps[lane]; a.theta = p.cls[lane].theta;
            aim[lane] = a;
        }
        T_blk_next = (f_blocks() && b + 1 < p.nblk) ? block_start(b + 1) : dinf();
    }

    // --- arrivals ------------------------------------------------------------------------------
    // Arrival draws do not depend on the simulation: draw k of class i is one Philox block that gives a unit
    // exponential E_k (words 0,1) and the two lengths (words 2,3).  The warp produces 32 consecutive draws
    // of a class at a time, one per lane, into a ring in shared memory; the class lane consumes them in
    // order.  Draws left in the ring at the end of a launch are given back (adraw is rewound).

    __device__ __forceinline__ void refill(uint32_t i)
    {
        const double t0 = aring[i * 32];                    // (the ring is empty: where the search for the class's next arrival starts)
        const unsigned long long base = cs[i].adraw;        // (only I class records exist: every lane reads record i)
        const uint32_t b = f_blocks() ? cs[i].ablk : 0u;
        // the division E / Lambda is done here, 32 at a time, for the block in which the class's next arrival is looked for
        const double Lam1 = __dmul_rn((double)p.N, p.blocks[b].rate[i]);
        __syncwarp();
        const ADraw d = make_draw(p.seed, p.rep_offset + rep, i, p.I, base + (unsigned long long)lane,
                                  p.length_mode == 1 ? p.lengths : nullptr, p.cls[i].P, p.cls[i].D, Lam1);
        aring[i * 32 + lane] = d.E;
        aring_pk[i * 32 + lane] = d.pk;
        __syncwarp();
        if (lane == (int)i) {
            const bool some = Lam1 > 0.0;       // (a class that never arrives asks for draws once, at the start)
            if (some) cs[i].adraw = base + 32ull;
            ring_pos = 0;
            ring_n = some ? 32u : 0u;
            ring_blk = b;
            ring_end = (f_blocks() && b + 1 < p.nblk) ? block_start(b + 1) : dinf();
            if (sched_pending) { sched_pending = false; schedule_from(t0); }
        }
        __syncwarp();
    }

    // Class lane only: next arrival of this lane's class after t0.  A candidate at or past the end of its
    // block is discarded and drawn again from the boundary under the next block's rate (memorylessness).
    __device__ __forceinline__ void schedule_from(double t0)
    {
        ClassState &c = cs[lane];
        if ((F & (F_GENERIC | F_INJECT)) && p.n_inject > 0) {
            // trace replay: the next entry of this class in the injected list (c.ablk is the read position)
            uint32_t k = c.ablk;
            while (k < p.n_inject && p.inject_job[3 * k] != (uint32_t)lane) ++k;
            if (k < p.n_inject) {
                c.ta = p.inject_t[k]; c.nextP = p.inject_job[3 * k + 1]; c.nextD = p.inject_job[3 * k + 2];
                c.ablk = k + 1;
            } else {
                c.ta = dinf(); c.ablk = k;
            }
            return;
        }
        uint32_t b = f_blocks() ? c.ablk : 0u;
        if (ring_n > 0 && (!f_blocks() || b == ring_blk)) {
            const double cand = __dadd_rn(t0, aring[lane * 32 + ring_pos]);
            const uint32_t pk = aring_pk[lane * 32 + ring_pos];
            ring_pos++; ring_n--;
            if (!f_blocks() || cand < ring_end) {
                c.ta = cand; c.nextP = job_P(pk); c.nextD = job_D(pk);
                return;
            }
            ++b; t0 = ring_end;
        }
        // no draws, or draws divided by the rate of another block: the warp makes new ones at the top of the next round
        if (f_blocks()) { c.adraw -= ring_n; ring_n = 0; }
        bool any = p.blocks[b].rate[lane] > 0.0;
        while (!any && f_blocks() && b + 1 < p.nblk) {
            ++b; t0 = block_start(b);
            any = p.blocks[b].rate[lane] > 0.0;
        }
        c.ablk = b; c.ta = dinf();
        sched_pending = any;
        aring[lane * 32] = t0;
    }

    // Class lane only: the arrival scheduled at c.ta happens; nothing outside the class is touched.
    __device__ __forceinline__ void arrival_local()
    {
        const uint32_t i = (uint32_t)lane;
        ClassState &c = cs[i];
        const double ta = c.ta;
        const uint32_t n = c.pq_n, head = c.pq_head;
        QEntry e; e.t = ta; e.pk = pack_job(c.nextP, c.nextD, i, 0); e.cls = i;
        if (n >= p.qcap) {
            c.overflow++;
        } else {
            if (f_abandon() && aim[lane].theta > 0.0) { ab_touch(c.abp, aim[lane].theta, n, ta); stale |= 1u; }
            area_touch(c.aQp, n, ta);
            c.pq_n = n + 1;
            uint32_t pos = head + n;
            if (pos >= p.qcap) pos -= p.qcap;
            pq[(size_t)i * p.qcap + pos] = e;
            if (n == 0) pqh[i] = e;        // it is the head: keep a copy on chip
        }
        schedule_from(ta);
    }

    // Next abandonment of a clock and levels of new ones where they are rarely asked for: out of line, but for the run-time-configured
    // calendar instances, which spill less with the code in line (SLI-aware router and priority gate, N = 300, R = 6000, 40 iterations of
    // horizon: 206 ms, 226 with the calls; the specialised instance of the occupancy gate spills nothing either way and takes 275 instead of 262).
    __device__ __forceinline__ double next_abandonment(const AbClock &a, uint32_t Q) const
    {
        if constexpr (CAL && (F & F_GENERIC)) return ab_next(a, aim[lane].theta, Q);
        else return ab_next_call(a, aim[lane].theta, Q);
    }
    __device__ __forceinline__ double abandonment_level(uint32_t w0, uint32_t w1) const
    {
        if constexpr (CAL && (F & F_GENERIC)) return -qlog(u53(w0, w1));
        else return unit_exp(w0, w1);
    }

    // Class lane only: next abandonment times of the clocks whose counts changed (the prefill queue's changes in almost every round).
    __device__ __forceinline__ void settle_queue()
    {
        ClassState &c = cs[lane];
        if (stale & 1u) c.abp.t_ab = ab_next(c.abp, aim[lane].theta, c.pq_n);
        stale &= ~1u;
    }
    __device__ __forceinline__ void settle_buffers()
    {
        ClassState &c = cs[lane];
#pragma unroll 1
        for (uint32_t k = 0; k < 2u; ++k) {
            AbClock &a = k ? c.abd1 : c.abd0;
            if (stale & (2u << k)) a.t_ab = next_abandonment(a, k ? c.Qd1 : c.Qd0);
        }
        stale = 0;
    }
    // Class lane only, after local arrivals: may the class's next prefill-queue abandonment come before the source src at time
    // tint?  Mostly not, which a product shows (the margin of a few ulps covers its roundings and those of the quotient).
    __device__ __forceinline__ bool abandons_before(unsigned long long tint, uint32_t src)
    {
        ClassState &c = cs[lane];
        if (stale & 1u) {
            const double ti = __longlong_as_double((long long)tint), dt = __dadd_rn(__dsub_rn(ti, c.abp.t_last), __dmul_rn(ti, 1e-15));
            if (__dsub_rn(c.abp.lvl, c.abp.acc) > __dmul_rn(__dmul_rn(dt, 1.0 + 1e-14), __dmul_rn(aim[lane].theta, (double)c.pq_n))) return false;
            c.abp.t_ab = next_abandonment(c.abp, c.pq_n);
            stale &= ~1u;
        }
        const unsigned long long v = (unsigned long long)__double_as_longlong(c.abp.t_ab);
        return v < tint || (v == tint && SRC_ABP + (uint32_t)lane < src);
    }

    // SLI-aware router: pools of the next 32 finished prefills of class i (bit k: the mixed pool for ordinals k mod 32), drawn together
    __device__ __forceinline__ void refill_pools(uint32_t i)
    {
        const unsigned long long ord = (cs[i].sli_ord & ~31ull) + (unsigned long long)lane;
        const double ps = aim[i].ps;
        uint32_t w0, w1, w2, w3;
        draw_rare(p, rep, (STREAM_SLI << 8) | i, ord, w0, w1, w2, w3);
        const uint32_t m = __ballot_sync(FULL, !(u53(w0, w1) <= ps));
        if (lane == (int)i) { pools = m; pools_due = false; }
    }

    // Top of a round: classes that ran out of arrival draws or pool draws get 32 new ones; clocks whose counts changed get their
    // next abandonment time.
    __device__ __forceinline__ void replenish()
    {
        // (a class whose next candidate lies past the end of its block asks again)
        for (uint32_t need = __ballot_sync(FULL, sched_pending || (f_sli() && pools_due)); need;
             need = f_blocks() ? __ballot_sync(FULL, sched_pending || (f_sli() && pools_due)) : need & (need - 1u)) {
            const uint32_t i = (uint32_t)__ffs((int)need) - 1u;
            if (!f_sli() || __shfl_sync(FULL, (int)sched_pending, (int)i)) refill(i);
            if (f_sli() && __shfl_sync(FULL, (int)pools_due, (int)i)) refill_pools(i);
        }
        if (f_abandon() && lane < (int)p.I) {
            settle_queue();
            if (stale) settle_buffers();
        }
    }

    __device__ uint32_t count_idle_pf()
    {
        // per-lane count over the lane's rows (branch-free), one warp-wide sum
        uint32_t cnt = 0;
#pragma unroll 1
        for (uint32_t k = 0; k < n_rows(); ++k)
            cnt += key_of((k << 5) + (uint32_t)lane, WANT_PREFILL) != NONE32 ? 1u : 0u;
        return __reduce_add_sync(FULL, cnt);
    }

    // --- abandonment ---------------------------------------------------------------------------
    // Remove entry `pos` (offset from head) of a ring of n entries, keeping order: shift the tail down.
    __device__ void ring_remove(QEntry *ring, uint32_t head, uint32_t n, uint32_t pos)
    {
        const uint32_t cap = p.qcap;
#pragma unroll 1
        for (uint32_t k = pos; k + 1 < n; k += 32) {
            const uint32_t j = k + (uint32_t)lane;
            QEntry e;
            const bool act = j + 1 < n;
            if (act) {
                uint32_t src = head + j + 1; if (src >= cap) src -= cap;
                e = ring[src];
            }
            __syncwarp();
            if (act) {
                uint32_t dst = head + j; if (dst >= cap) dst -= cap;
                ring[dst] = e;
            }
            __syncwarp();
        }
    }

    // A class-i request leaves the prefill queue (which = 0) or the decode buffer of pool which - 1.  One body for the three:
    // the size of the round loop is what the instruction cache has to hold.
    __device__ void on_abandon(uint32_t which, uint32_t i)
    {
        const ClassState &ci = cs[i];
        const AbClock &ai = which == 0 ? ci.abp : (which == 1 ? ci.abd0 : ci.abd1);
        const uint32_t Q = which == 0 ? ci.pq_n : (which == 1 ? ci.Qd0 : ci.Qd1);
        const unsigned long long m = ai.m;
        uint32_t w0, w1, w2, w3;
        draw_rare(p, rep, ((STREAM_ABANDON_P + which) << 8) | i, m, w0, w1, w2, w3);
        uint32_t rank = __umulhi(w2, Q), pos = rank;       // uniformly chosen waiting request, in FCFS rank
        QEntry *ring = pq + (size_t)i * p.qcap;
        uint32_t head = ci.pq_head, n = Q;
        if (which == 0) {
            cp_async_wait_all();
        } else {
            // position of the rank-th class-i entry in buffer order
            ring = dq + (size_t)(which - 1u) * p.qcap;
            head = which == 2 ? dq_head1 : dq_head0;
            n = which == 2 ? dq_n1 : dq_n0;
            pos = NONE32;
#pragma unroll 1
            for (uint32_t k = 0; k < n && pos == NONE32; k += 32) {
                const uint32_t j = k + (uint32_t)lane;
                bool mine = false;
                if (j < n) {
                    uint32_t src = head + j; if (src >= p.qcap) src -= p.qcap;
                    mine = ring[src].cls == i;
                }
                const uint32_t b = __ballot_sync(FULL, mine);
                const uint32_t c = (uint32_t)__popc(b);
                // (the lane with `rank` of them before it)
                if (rank < c) pos = k + (uint32_t)__ffs((int)__ballot_sync(FULL, mine && (uint32_t)__popc(b & ((1u << lane) - 1u)) == rank)) - 1u;
                else rank -= c;
            }
            if (pos == NONE32) { err = ERR_INTERNAL; return; }
            if (which == 2) dq_n1--; else dq_n0--;
        }
        __syncwarp();
        ring_remove(ring, head, n, pos);
        if (lane == (int)i) {
            ClassState &c = cs[i];
            AbClock &a = which == 0 ? c.abp : (which == 1 ? c.abd0 : c.abd1);
            if (which == 0) {
                if (Q > 1) pqh[i] = ring[head];     // the head may have changed
                area_touch(c.aQp, Q, t);
                c.pq_n = Q - 1;
                c.abandoned_p++;
            } else {
                area_touch(c.aQd, c.Qd0 + c.Qd1, t);
                if (which == 2) c.Qd1 = Q - 1; else c.Qd0 = Q - 1;
                c.abandoned_d++;
            }
            a.m = m + 1; a.acc = 0.0; a.lvl = abandonment_level(w0, w1); a.t_last = t;
            stale |= 1u << which;
        }
    }

    // --- GPU choice ----------------------------------------------------------------------------
    // --- least-loaded choice on large clusters (CAL) ------------------------------------------------------
    // The smallest key of every row of 32 GPUs is kept, so a choice looks at N / 32 keys (one per lane up to 1024 GPUs) instead
    // of all GPUs; rows in which something changed since are looked up again, a GPU per lane, when a choice needs them.
    __device__ __forceinline__ void decodes_changed(uint32_t g) { if (CAL && lane == (int)((g >> 5) & 31u)) { dirty_dec |= 1u << (g >> 10); dirty_pf |= 1u << (g >> 10); } }
    __device__ __forceinline__ void prefill_changed(uint32_t g)
    {
        // (a solo GPU that still holds a prefill has a slot less for decodes)
        if (CAL && lane == (int)((g >> 5) & 31u)) { dirty_pf |= 1u << (g >> 10); if (g >= M) dirty_dec |= 1u << (g >> 10); }
    }

    // key of GPU g for the wanted tiers: solo GPUs first, then decodes held, then index; NONE32 when it is not eligible
    __device__ __forceinline__ uint32_t key_of(uint32_t g, uint32_t tiers) const
    {
        // g is always inside the padded arrays; every field is read first so that calls over rows overlap
        const uint32_t nd = ndec[g], pf = pfrem[g];
        const bool mix = g < M;
        const uint32_t cap = (mix || pf != 0) ? p.B - 1 : p.B;   // a mixed GPU keeps one slot for prefill
        const bool ok = tiers == WANT_PREFILL ? (mix && pf == 0 && nd <= p.B - 1) : ((tiers & (mix ? WANT_MIX : WANT_SOLO)) != 0 && nd < cap);
        return (ok && g < p.N) ? ((mix ? 0x40000000u : 0u) | (nd << 16) | g) : NONE32;
    }
    // The GPUs of one tier as a range of indices and a bound on the decodes held, without and with a prefill: what key_of tests,
    // with the tier's part of it done once for all rows.
    struct Tier { uint32_t from, to, cap, cap_pf; };
    __device__ __forceinline__ Tier tier_gpus(uint32_t tier) const
    {
        if (tier == WANT_SOLO) return { M, p.N, p.B, p.B - 1u };
        return { 0u, M, tier == WANT_MIX ? p.B - 1u : p.B, tier == WANT_MIX ? p.B - 1u : 0u };
    }
    __device__ __forceinline__ bool in_tier(uint32_t g, const Tier &w) const
    {
        const uint32_t nd = ndec[g], pf = pfrem[g];
        return g >= w.from && g < w.to && nd < (pf != 0 ? w.cap_pf : w.cap);
    }

    // Least loaded (lowest index on ties) or uniformly random among the eligible GPUs of the first tier that has one
    __device__ __forceinline__ uint32_t choose(uint32_t tiers)
    {
        const uint32_t rows = n_rows();
        if (!f_random()) {
            uint32_t best = NONE32;
            if (CAL) {
                // keys of the solo-first router, or of solo GPUs under the SLI-aware ones; of mixed GPUs under those; of prefill targets
                const bool pf = tiers == WANT_PREFILL;
#pragma unroll 1
                for (uint32_t bits = __ballot_sync(FULL, (pf ? dirty_pf : dirty_dec) != 0); bits; bits = __ballot_sync(FULL, (pf ? dirty_pf : dirty_dec) != 0)) {
                    const uint32_t l = (uint32_t)__ffs((int)bits) - 1u;
                    uint32_t row = l;
                    if (rows > 32u) row += ((uint32_t)__ffs((int)__shfl_sync(FULL, pf ? dirty_pf : dirty_dec, (int)l)) - 1u) << 5;
                    const uint32_t g = (row << 5) + (uint32_t)lane;
                    const uint32_t a = __reduce_min_sync(FULL, key_of(g, pf ? WANT_PREFILL : (f_sli() ? WANT_SOLO : (WANT_SOLO | WANT_MIX))));
                    if (f_sli() && !pf) {
                        const uint32_t b = __reduce_min_sync(FULL, key_of(g, WANT_MIX));
                        if (lane == (int)l) row_key[rows + row] = b;
                    }
                    if (lane == (int)l) {
                        row_key[(pf ? 2u * rows : 0u) + row] = a;
                        if (pf) dirty_pf &= dirty_pf - 1u; else dirty_dec &= dirty_dec - 1u;
                    }
                }
                // (a lane reads the rows that it has written)
                const uint32_t *keys = row_key + (pf ? 2u * rows : ((f_sli() && tiers == WANT_MIX) ? rows : 0u));
#pragma unroll 1
                for (uint32_t k = (uint32_t)lane; k < rows; k += 32u) best = min(best, keys[k]);
            } else {
#pragma unroll 4
                for (uint32_t k = 0; k < rows; ++k) best = min(best, key_of((k << 5) + (uint32_t)lane, tiers));
            }
            best = __reduce_min_sync(FULL, best);
            return best == NONE32 ? NONE32 : (best & 0xffffu);
        }
#pragma unroll(SPL > 0 && !(F & F_GENERIC) ? 3 : 1)
        for (uint32_t tier = WANT_SOLO; tier <= WANT_PREFILL; tier <<= 1) {
            if (!(tiers & tier)) continue;
            const Tier w = tier_gpus(tier);
            const uint32_t first = SPL > 0 ? 0u : w.from >> 5, last = SPL > 0 ? rows : (w.to + 31u) >> 5;
            uint32_t cnt = 0;
#pragma unroll(SPL > 0 ? SPL : 4)
            for (uint32_t k = first; k < last; ++k)
                cnt += (uint32_t)__popc(__ballot_sync(FULL, in_tier((k << 5) + (uint32_t)lane, w)));
            if (cnt == 0) continue;
            uint32_t idx = 0;
            if (cnt > 1) idx = __umulhi(placement_word(), cnt);
#pragma unroll(SPL > 0 ? SPL : 4)
            for (uint32_t k = first; k < last; ++k) {
                const bool in = in_tier((k << 5) + (uint32_t)lane, w);
                const uint32_t b = __ballot_sync(FULL, in);
                const uint32_t c = (uint32_t)__popc(b);
                if (idx < c) {
                    // the lane whose GPU has idx eligible ones before it in the row
                    const uint32_t at = __ballot_sync(FULL, in && (uint32_t)__popc(b & ((1u << lane) - 1u)) == idx);
                    return (k << 5) + (uint32_t)__ffs((int)at) - 1u;
                }
                idx -= c;
            }
            err = ERR_INTERNAL;
            return NONE32;
        }
        return NONE32;
    }

    // Word of the next placement draw: the warp makes the draws of 32 consecutive ordinals together, one per lane.
    __device__ __forceinline__ uint32_t placement_word()
    {
        const unsigned long long ord = place_ord++;
        if ((ord & ~31ull) != place_base) {
            uint32_t w1, w2, w3;
            place_base = ord & ~31ull;
            draw_rare(p, rep, STREAM_PLACEMENT << 8, place_base + (unsigned long long)lane, place_w, w1, w2, w3);
        }
        return __shfl_sync(FULL, place_w, (int)(ord & 31ull));
    }

    // GPU g may have to start an iteration at the end of this event: noted in its owner's row mask, or once in a list over the lanes
    __device__ __forceinline__ void touch_server(uint32_t g)
    {
        if (SPL > 0) { if (lane == (int)(g & 31u)) need_start |= 1u << (g >> 5); }
        else if (!__any_sync(FULL, (uint32_t)lane < n_touch && touch_g == g)) {
            if (n_touch == 32u) touch_all = true;
            else { if (lane == (int)n_touch) touch_g = g; n_touch++; }
        }
    }

    // --- decode placement ------------------------------------------------------------------------
    // General SLI-aware router: position (in buffer order) of the request that gets the freed slot of the pool.
    // The class is drawn with probabilities proportional to varpi over the classes that wait in the pool; one
    // waiting class needs no draw, and with no positive weight among them the head of the buffer goes.
    __device__ uint32_t select_in_pool(uint32_t pool)
    {
        const BlockPar &bp = p.blocks[blk];
        uint32_t nonempty = 0, cls = 0;
        double Wsum = 0.0;
        for (uint32_t i = 0; i < p.I; ++i)
            if ((pool ? cs[i].Qd1 : cs[i].Qd0) > 0) { ++nonempty; cls = i; Wsum = __dadd_rn(Wsum, pool ? bp.wm[i] : bp.ws[i]); }
        if (nonempty > 1) {
            if (!(Wsum > 0.0)) return 0;
            uint32_t w0, w1, w2, w3;
            if (pool) draw_rare(p, rep, STREAM_SELECT1 << 8, sel_ord1++, w0, w1, w2, w3);
            else      draw_rare(p, rep, STREAM_SELECT0 << 8, sel_ord0++, w0, w1, w2, w3);
            const double x = __dmul_rn(u53(w0, w1), Wsum);
            double cum = 0.0;
            uint32_t chosen = NONE32, last = NONE32;
            for (uint32_t i = 0; i < p.I && chosen == NONE32; ++i) {
                if ((pool ? cs[i].Qd1 : cs[i].Qd0) == 0) continue;
                const double w = pool ? bp.wm[i] : bp.ws[i];
                cum = __dadd_rn(cum, w);
                if (w > 0.0) { last = i; if (cum >= x) chosen = i; }
            }
            cls = chosen != NONE32 ? chosen : last;
        }
        // oldest request of the class
        const QEntry *ring = dq + (size_t)pool * p.qcap;
        const uint32_t head = pool ? dq_head1 : dq_head0, n = pool ? dq_n1 : dq_n0;
        for (uint32_t k = 0; k < n; k += 32) {
            const uint32_t j = k + (uint32_t)lane;
            bool mine = false;
            if (j < n) {
                uint32_t src = head + j; if (src >= p.qcap) src -= p.qcap;
                mine = ring[src].cls == cls;
            }
            const uint32_t b = __ballot_sync(FULL, mine);
            if (b) return k + (uint32_t)__ffs((int)b) - 1u;
        }
        err = ERR_INTERNAL;
        return 0;
    }

    // Entry pos (0 = head) leaves the pool's buffer to be placed.
    __device__ __forceinline__ QEntry take_buffered(uint32_t pool, uint32_t pos)
    {
        const uint32_t head = pool ? dq_head1 : dq_head0;
        QEntry *ring = dq + (size_t)pool * p.qcap;
        uint32_t src = head + pos; if (src >= p.qcap) src -= p.qcap;
        const QEntry e = ring[src];
        if (!f_slig() || pos == 0) {
            const uint32_t next = (head + 1 == p.qcap) ? 0 : head + 1;
            if (pool) dq_head1 = next; else dq_head0 = next;
        } else {
            __syncwarp();
            ring_remove(ring, head, pool ? dq_n1 : dq_n0, pos);
        }
        if (pool) dq_n1--; else dq_n0--;
        return e;
    }

    // A request leaves for its decode on GPU g.  fresh: it has just finished its prefill (d_pk, arrived at d_tarr) and passes through
    // its pool's empty buffer at this very instant, which leaves the buffer's count, integral and abandonment clock as one
    // touch at time t would, or joins the buffer (g = NONE32); else it is an entry of the pool's buffer.
    // One body for all of that, and its parts - the class lane's and the GPU's - read before they write, so that their reads overlap.
    __device__ __forceinline__ void place(uint32_t pool, uint32_t g, bool fresh)
    {
        const bool placed = g != NONE32, mixed = placed && g < M;
        const uint32_t n_buf = pool ? dq_n1 : dq_n0;
        uint32_t pk = d_pk;
        double tpf = t;
        if (!fresh) {
            const QEntry e = take_buffered(pool, f_slig() ? select_in_pool(pool) : 0u);
            pk = pack_job(job_P(e.pk), job_D(e.pk), e.cls, 0);
            tpf = e.t;
        }
        const bool full = fresh && !placed && n_buf >= p.qcap;
        const uint32_t i = job_cls(pk);
        // the GPU (every lane reads it)
        const uint32_t gg = placed ? g : 0u;
        const uint32_t nd = ndec[gg], it0 = it[gg], nf = nfin[gg];
        const bool running = tnext[gg] < dinf();
        if (lane == (int)i) {
            ClassState &c = cs[i];
            const uint32_t Qd0 = c.Qd0, Qd1 = c.Qd1, Qd = pool ? Qd1 : Qd0;
            if (fresh) {
                const uint32_t X = c.X;
                area_touch(c.aX, X, t);
                c.X = X - 1;
                c.prefill_done++;
                c.tok_in_pf += job_P(pk);                  // separate charging credits the prompt here, Eq. (23)
                const double ttft = __dsub_rn(t, d_tarr);
                c.sum_ttft = __dadd_rn(c.sum_ttft, ttft);
                if (f_hist()) atomicAdd(&hist[((size_t)i * 2 + 0) * NBIN + hist_bin(ttft)], 1u);
                if (f_sli()) {
                    const unsigned long long ord = c.sli_ord + 1ull;
                    c.sli_ord = ord;
                    if ((ord & 31ull) == 0) pools_due = true;
                }
            }
            if (full) {
                c.overflow_d++;
            } else if (fresh && placed) {
                // (nothing accrues on an empty buffer, and its clock starts when it fills)
                if (Qd0 + Qd1 != 0) area_touch(c.aQd, Qd0 + Qd1, t);
            } else {
                const uint32_t Qn = fresh ? Qd + 1u : Qd - 1u;
                if (f_abandon() && aim[lane].theta > 0.0) {
                    ab_touch(pool ? c.abd1 : c.abd0, aim[lane].theta, Qd, t);
                    stale |= pool ? 4u : 2u;
                }
                area_touch(c.aQd, Qd0 + Qd1, t);
                if (pool) c.Qd1 = Qn; else c.Qd0 = Qn;
            }
            if (placed) {
                const double rel = __dsub_rn(t, *T_reset_at);
                if (mixed) { c.sYm_in = __dadd_rn(c.sYm_in, rel); c.Ym++; }
                else       { c.sYs_in = __dadd_rn(c.sYs_in, rel); c.Ys++; }
            }
        }
        if (!placed) {
            if (!full) {
                uint32_t pos = (pool ? dq_head1 : dq_head0) + n_buf;
                if (pos >= p.qcap) pos -= p.qcap;
                if (lane == 0) {
                    QEntry e; e.t = t; e.pk = pk; e.cls = i;
                    dq[(size_t)pool * p.qcap + pos] = e;
                }
                if (pool) dq_n1++; else dq_n0++;
            }
            return;
        }
        const uint32_t P = job_P(pk), D = job_D(pk);
        if (lane == (int)(g & 31u)) {
            // joins the iteration that starts next: a running iteration first finishes as it+1
            const uint32_t fin = it0 + (running ? 1u : 0u) + D;
            size_t o;
            if (f_slots()) {
                // first free slot of the GPU's occupancy words
                const uint32_t bw = (p.B + 31u) >> 5;
                uint32_t slot = 0;
                for (uint32_t w = 0; w < bw; ++w) {
                    const uint32_t word = socc[g * bw + w];
                    if (word != 0xffffffffu) {
                        const uint32_t b = (uint32_t)__ffs((int)~word) - 1u;
                        socc[g * bw + w] = word | (1u << b);
                        slot = (w << 5) + b;
                        break;
                    }
                }
                sfin16[g * p.B + slot] = (uint16_t)fin;
                o = (size_t)g * p.B + slot;
            } else {
                o = (size_t)g * p.B + nd;
                s_fin[o] = fin;
            }
            SlotRec r; r.tpf = tpf; r.pk = pack_job(P, D, i, mixed ? 1u : 0u); r.pad = 0;
            s_rec[o] = r;
            ndec[g] = (uint16_t)(nd + 1);
            nfin[g] = min(nf, fin);
            if (f_kappa()) Kpend[g] += P;
        }
        decodes_changed(g);
        touch_server(g);
    }

    // --- prefill gate ------------------------------------------------------------------------------
    __device__ uint32_t gate_class()
    {
        if ((F & F_GENERIC) && p.gate == 2) {
            // FCFS ablation: the class whose head-of-line request arrived first (heads are mirrored on chip)
            cp_async_wait_all();
            __syncwarp();
            uint32_t best = NONE32;
            double bt = 0.0;
            for (uint32_t i = 0; i < p.I; ++i) {
                if (cs[i].pq_n == 0) continue;
                const double ta = pqh[i].t;
                if (best == NONE32 || ta < bt) { best = i; bt = ta; }
            }
            __syncwarp();
            return best;
        }
        if (!f_occ()) {
            // Prioritize-and-Route: largest D_i/P_i among waiting classes = smallest static rank
            uint32_t key = NONE32;
            if (lane < (int)p.I && cs[lane].pq_n > 0) key = (p.cls[lane].prio << 8) | (uint32_t)lane;
            key = __reduce_min_sync(FULL, key);
            return key == NONE32 ? NONE32 : (key & 0xffu);
        }
        // Occupancy gate: argmin of xi_i = (X_i - n x*_i)/x*_i over the class lanes, ties to the largest Q_p,i - n q*_p,i, then
        // to the lowest class.  Doubles are compared through their bits (order_key), so a minimum is two reductions.
        unsigned long long xi = ~0ull;
        bool ok = false;
        if (lane < (int)p.I) {
            const ClassState &c = cs[lane];
            ok = c.pq_n > 0 && aim[lane].xstar > 0.0;
            if (ok) xi = order_key(__ddiv_rn(__dsub_rn((double)c.X, aim[lane].nx), aim[lane].xstar));
        }
        const uint32_t xh = (uint32_t)(xi >> 32), mh = __reduce_min_sync(FULL, xh);
        const uint32_t ml = __reduce_min_sync(FULL, xh == mh ? (uint32_t)xi : NONE32);
        ok = ok && xh == mh && (uint32_t)xi == ml;
        uint32_t tie = __ballot_sync(FULL, ok);
        if (tie & (tie - 1u)) {
            unsigned long long dq = 0ull;
            if (ok) dq = order_key(__dsub_rn((double)cs[lane].pq_n, aim[lane].nq));
            const uint32_t dh = (uint32_t)(dq >> 32), Mh = __reduce_max_sync(FULL, dh);
            const uint32_t Ml = __reduce_max_sync(FULL, dh == Mh ? (uint32_t)dq : 0u);
            tie = __ballot_sync(FULL, ok && dh == Mh && (uint32_t)dq == Ml);
        }
        return tie ? (uint32_t)__ffs((int)tie) - 1u : NONE32;
    }

    // unsigned integers that order as the doubles do (adding zero makes the two zeros one)
    static __device__ __forceinline__ unsigned long long order_key(double x)
    {
        const long long b = __double_as_longlong(__dadd_rn(x, 0.0));
        return (unsigned long long)b ^ (b < 0 ? ~0ull : 0x8000000000000000ull);
    }

    __device__ void admit(uint32_t i, uint32_t g)
    {
        // the head of the class queue is kept in shared memory (copied there asynchronously after each pop);
        // record copies of finished requests that this lane committed later stay in flight
        if (lane == (int)i) {
            if (rec_after == 1) cp_async_wait_group<1>();
            else if (rec_after == 2) cp_async_wait_group<2>();
            else cp_async_wait_group<0>();
        }
        __syncwarp();
        const QEntry e = pqh[i];
        __syncwarp();
        if (lane == (int)i) {
            ClassState &c = cs[i];
            const uint32_t n = c.pq_n, X = c.X, head = c.pq_head, next = (head + 1 == p.qcap) ? 0 : head + 1;
            if (f_abandon() && aim[lane].theta > 0.0) { ab_touch(c.abp, aim[lane].theta, n, t); stale |= 1u; }
            area_touch(c.aQp, n, t);
            area_touch(c.aX, X, t);
            c.pq_n = n - 1;
            c.pq_head = next;
            c.X = X + 1;
            if (n > 1) { cp_async16(&pqh[i], &pq[(size_t)i * p.qcap + next]); cp_async_commit(); rec_after = 0; }
        }
        n_idle_pf--;
        idle_hint = NONE32;
        if (lane == (int)(g & 31u)) {
            pfjob[g] = e.pk | 0x80000000u;
            pfrem[g] = (uint16_t)job_P(e.pk);
            pf_tarr[g] = e.t;
        }
        prefill_changed(g);
        touch_server(g);
    }

    // Called by the owner: a GPU with work that is between iterations starts one at time ts.  The batch
    // (prefill chunk, decodes) is frozen here for the whole iteration, and with it what its end will bring:
    // bit 14 of nact = some decode emits its last token, bit 15 = the prefill finishes.
    // Straight-line: every field is read first and the stores are predicated on `act`, so that the calls for
    // the rows of one lane overlap.  g is always inside the padded arrays.
    __device__ __forceinline__ void start_at(uint32_t g, double ts, bool act = true)
    {
        const unsigned long long tn = (unsigned long long)__double_as_longlong(tnext[g]);
        const uint32_t nd = ndec[g], rem = pfrem[g], nf = nfin[g], it0 = it[g];
        uint32_t Kg = 0;
        if (f_kappa()) Kg = K[g] + Kpend[g];
        const bool has_pf = rem != 0;
        const uint32_t pc = has_pf ? min(p.C, rem) : 0u;
        uint32_t fl = (nf == it0 + 1u) ? 0x4000u : 0u;
        if (pc > 0 && pc == rem) fl |= 0x8000u;
        if (CAL && pc > 0) fl |= BATCH_MIXED;
        const double tau = iter_time(p, pc, nd, Kg, f_kappa());
        if (act && tn >= 0x7ff0000000000000ull && (nd > 0 || has_pf)) {
            if (f_kappa()) { K[g] = Kg; Kpend[g] = 0; }
            if (!CAL) pfcur[g] = (uint16_t)pc;
            nact[g] = (uint16_t)(nd | fl);
            const double te = __dadd_rn(ts, tau);
            tnext[g] = te;
            if (CAL) file_end(g, te);
        }
    }

    __device__ void dispatch()
    {
        __syncwarp();   // queue entries and GPU state written by the event handler are visible to every lane
        // decode routing: the request that has just finished its prefill, then the buffered ones, FCFS, solo GPUs before mixed ones,
        // or pool by pool
        uint32_t pool = drain_dirty ? 0u : 2u;       // buffer being drained; 2: none left
#pragma unroll 1
        for (;;) {
            uint32_t q = d_pool, g = d_gpu;
            const bool fresh = handed, search = !fresh || (direct && g == NONE32);
            if (!fresh) {
                if (pool == 0 && dq_n0 == 0) pool = f_sli() ? 1u : 2u;
                if (pool == 1 && dq_n1 == 0) pool = 2u;
                if (pool == 2u) break;
                q = pool;
            }
            if (search) g = choose(f_sli() ? (q ? WANT_MIX : WANT_SOLO) : (WANT_SOLO | WANT_MIX));
            if (!fresh && g == NONE32) { pool = (pool == 0 && f_sli()) ? 1u : 2u; continue; }
            if (fresh && search && g == NONE32 && !f_sli()) pool = 2u;       // no GPU has a slot: nothing to drain either
            place(q, g, fresh);
            handed = false;
            __syncwarp();
        }
        // prefill gate on mixed GPUs whose prefill slot is idle; a single idle slot whose GPU is known needs no search (and
        // draws nothing: one candidate)
        if (gate_dirty)
            while (n_idle_pf > 0) {
                const uint32_t cls = gate_class();
                if (cls == NONE32) break;
                const uint32_t g = (n_idle_pf == 1 && idle_hint != NONE32) ? idle_hint : choose(WANT_PREFILL);
                if (g == NONE32) break;
                admit(cls, g);
                __syncwarp();
            }
        drain_dirty = false;
        gate_dirty = false;
        // start the next iteration on every GPU that was touched and is between iterations
        __syncwarp();
        if (SPL > 0) {
            // every owner starts its touched GPUs; different lanes work in parallel
#pragma unroll
            for (uint32_t k = 0; k < (uint32_t)(SPL > 0 ? SPL : 1); ++k)
                start_at((k << 5) + (uint32_t)lane, t, ((need_start >> k) & 1u) != 0);
            need_start = 0;
        } else {
            // one lane per touched GPU, or all GPUs
            const uint32_t n = touch_all ? p.N : n_touch;
#pragma unroll 1
            for (uint32_t k = (uint32_t)lane; k < n; k += 32u) start_at(touch_all ? k : touch_g, t);
        }
        n_touch = 0;
        touch_all = false;
    }

    // Some decode on GPU g emitted its last token in the iteration that ended at te (its it-th): the whole
    // warp scans the GPU's slot list from the tail, accounts every finished request and closes the gaps.
    // Accounting of one finished request (uniform arguments; the class lane does the work).
    __device__ __forceinline__ void account_done(uint32_t pk, double tpf, double te)
    {
        const uint32_t i = job_cls(pk), P = job_P(pk), D = job_D(pk);
        if (lane == (int)i) {
            WarpClassStats &c = wcs[warp * (int)p.I + (int)i];
            const double rel = __dsub_rn(te, *T_reset_at);
            if (job_flag(pk)) { c.sYm_out = __dadd_rn(c.sYm_out, rel); c.done_mixed++; }
            else              { c.sYs_out = __dadd_rn(c.sYs_out, rel); c.done_solo++; }
            c.tok_in += P;       // bundled charging credits the request here, Eq. (21)-(22)
            c.tok_out += D;
            const double tpot = __ddiv_rn(__dsub_rn(te, tpf), (double)D);
            c.sum_tpot = __dadd_rn(c.sum_tpot, tpot);
            if (f_hist()) atomicAdd(&hist[((size_t)i * 2 + 1) * NBIN + hist_bin(tpot)], 1u);
        }
    }

    // Accounting of the finished requests whose records were staged in shared memory: a lane per record forms the latency
    // (the division is the long part: once for 32 records instead of once for each), then the class lanes add theirs up in
    // completion order.
    __device__ void flush_done()
    {
        if (n_pend == 0) return;
        if (f_slots()) cp_async_wait_all();
        __syncwarp();
#pragma unroll 1
        for (uint32_t e = (uint32_t)lane; e < n_pend; e += 32u) {
            const uint32_t pk = st_rec[e].pk;
            const double te = st_te[e], tpot = __ddiv_rn(__dsub_rn(te, st_rec[e].tpf), (double)job_D(pk));
            st_rec[e].tpf = tpot;
            st_te[e] = __dsub_rn(te, *T_reset_at);
            if (f_hist()) atomicAdd(&hist[((size_t)job_cls(pk) * 2 + 1) * NBIN + hist_bin(tpot)], 1u);
        }
        __syncwarp();
        if (lane < (int)p.I) {
            WarpClassStats c = wcs[warp * (int)p.I + lane];
#pragma unroll 1
            for (uint32_t e = 0; e < n_pend; ++e) {
                const uint32_t pk = st_rec[e].pk;
                if (job_cls(pk) != (uint32_t)lane) continue;
                const double rel = st_te[e];
                if (job_flag(pk)) { c.sYm_out = __dadd_rn(c.sYm_out, rel); c.done_mixed++; }
                else              { c.sYs_out = __dadd_rn(c.sYs_out, rel); c.done_solo++; }
                c.tok_in += job_P(pk);       // bundled charging credits the request here, Eq. (21)-(22)
                c.tok_out += job_D(pk);
                c.sum_tpot = __dadd_rn(c.sum_tpot, st_rec[e].tpf);
            }
            wcs[warp * (int)p.I + lane] = c;
        }
        n_pend = 0;
        __syncwarp();
    }

    // retire_decodes when stamps and occupancy are in shared memory: every lane checks one slot per word of
    // occupancy; the lanes that hit fetch their request records at the same time.
    __device__ void retire_slots(uint32_t g, uint32_t itg, uint32_t nd, double te)
    {
        const int owner = (int)(g & 31u);
        const uint32_t bw = (p.B + 31u) >> 5, it16 = itg & 0xffffu;
        uint32_t newmin = NONE32, done = 0, Kdrop = 0;
        for (uint32_t w = 0; w < bw; ++w) {
            const uint32_t occ = socc[g * bw + w];
            const uint32_t j = (w << 5) + (uint32_t)lane;
            const bool live = ((occ >> lane) & 1u) != 0 && j < p.B;
            const uint32_t dist = live ? (((uint32_t)sfin16[g * p.B + j] - it16) & 0xffffu) : NONE32;
            const bool hit = live && dist == 0;
            if (live && !hit) newmin = min(newmin, dist);
            uint32_t hits = __ballot_sync(FULL, hit);
            if (hits) {
                if (lane == owner) socc[g * bw + w] = occ & ~hits;
                done += (uint32_t)__popc(hits);
                if (!f_kappa()) {
                    // the records only feed statistics: copy them on chip asynchronously, account later
                    if (n_pend + 32u > (uint32_t)STAGE_CAP) flush_done();
                    if (hit) {
                        const uint32_t pos = n_pend + (uint32_t)__popc(hits & ((1u << lane) - 1u));
                        cp_async16(&st_rec[pos], &s_rec[(size_t)g * p.B + j]);
                        cp_async_commit();
                        rec_after++;
                        st_te[pos] = te;
                    }
                    n_pend += (uint32_t)__popc(hits);
                } else {
                    SlotRec r; r.tpf = 0.0; r.pk = 0;
                    if (hit) r = s_rec[(size_t)g * p.B + j];
                    while (hits) {
                        const int hl = __ffs((int)hits) - 1;
                        hits &= hits - 1;
                        const uint32_t pkh = __shfl_sync(FULL, r.pk, hl);
                        const double tpfh = __shfl_sync(FULL, r.tpf, hl);
                        account_done(pkh, tpfh, te);
                        Kdrop += job_P(pkh) + job_D(pkh);
                    }
                }
            }
        }
        newmin = __reduce_min_sync(FULL, newmin);
        if (lane == owner) {
            ndec[g] = (uint16_t)(nd - done);
            nfin[g] = newmin == NONE32 ? NONE32 : itg + newmin;
            if (f_kappa()) K[g] -= Kdrop;
        }
        decodes_changed(g);
        __syncwarp();
    }

    __device__ void retire_decodes(uint32_t g, uint32_t itg, uint32_t nd, double te)
    {
        if (f_slots()) { retire_slots(g, itg, nd, te); return; }
        const int owner = (int)(g & 31u);
        uint32_t n = nd, newmin = NONE32, Kdrop = 0;
        uint32_t *fin = s_fin + (size_t)g * p.B;
        SlotRec *rec = s_rec + (size_t)g * p.B;
        if constexpr (SPL == 1) {
            // Up to 32 GPUs: the finished request's record and the tail entry that takes its place are read together, after the stamps, a
            // second round trip, but less code, from which the run-time-configured instance gains most (priority gate with blocks, N = 20,
            // R = 4000, 24 blocks of 0.5 s: 9.5 ms, 10.5 the other way).
#pragma unroll 1
            for (int k0 = (int)((nd - 1u) & ~127u); k0 >= 0; k0 -= 128) {
                uint32_t f[4], hit[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t j = (uint32_t)(k0 + 32 * q + lane);
                    f[q] = j < nd ? fin[j] : NONE32;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (f[q] != itg) newmin = min(newmin, f[q]);
                    hit[q] = __ballot_sync(FULL, f[q] == itg);
                }
#pragma unroll 1
                for (;;) {          // from the tail of the list down
                    const int q = hit[3] ? 3 : (hit[2] ? 2 : (hit[1] ? 1 : 0));
                    const uint32_t hits = hit[3] ? hit[3] : (hit[2] ? hit[2] : (hit[1] ? hit[1] : hit[0]));
                    if (!hits) break;
                    const int hl = 31 - __clz((int)hits);
#pragma unroll
                    for (int j = 0; j < 4; ++j) hit[j] &= j == q ? ~(1u << hl) : ~0u;
                    const uint32_t h = (uint32_t)(k0 + 32 * q + hl), last = n - 1u;
                    const SlotRec rh = rec[h], rl = rec[last];
                    const uint32_t fl = fin[last];
                    if (n_pend == (uint32_t)ROW_STAGE_CAP) flush_done();
                    if (lane == 0) { st_rec[n_pend] = rh; st_te[n_pend] = te; }
                    n_pend++;
                    Kdrop += job_P(rh.pk) + job_D(rh.pk);
                    __syncwarp();
                    if (lane == 0 && h != last) { fin[h] = fl; rec[h] = rl; }
                    __syncwarp();
                    n = last;
                }
            }
        } else {
            // The stamps of 128 slots are fetched together, four neighbours per lane, and with them the tail entry that will close the
            // gap of the first finished request: one memory round trip.  The finished request's own record only feeds the
            // statistics: with one warp it stays on its way until the next one (`late`).
            SlotRec rl; rl.tpf = 0.0; rl.pk = 0; rl.pad = 0;
            uint32_t fl = 0;
            if (lane == 0) { rl = rec[nd - 1]; fl = fin[nd - 1]; }
#pragma unroll 1
            for (int k0 = (int)((nd - 1u) & ~127u); k0 >= 0; k0 -= 128) {
                uint32_t f[4], mine = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t j = (uint32_t)(k0 + 4 * lane + q);
                    f[q] = j < nd ? fin[j] : NONE32;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (f[q] == itg) mine |= 1u << q;
                    else newmin = min(newmin, f[q]);
                }
#pragma unroll 1
                for (uint32_t any = __ballot_sync(FULL, mine != 0); any; any = __ballot_sync(FULL, mine != 0)) {      // from the tail of the list down
                    const int hl = 31 - __clz((int)any);
                    const int q = 31 - __clz((int)__shfl_sync(FULL, mine, hl));
                    if (lane == hl) mine &= ~(1u << q);
                    const uint32_t h = (uint32_t)(k0 + 4 * hl + q), last = n - 1u;
                    if (STAGED && !f_kappa()) {
                        stage_late();
                        if (n_pend == (uint32_t)ROW_STAGE_CAP) flush_done();
                        has_late = true;
                        if (lane == 0) { const SlotRec r = rec[h]; late_tpf = r.tpf; late_pk = r.pk; st_te[n_pend] = te; }
                    } else {
                        const SlotRec rh = rec[h];
                        if (STAGED) {
                            if (n_pend == (uint32_t)ROW_STAGE_CAP) flush_done();
                            if (lane == 0) { st_rec[n_pend] = rh; st_te[n_pend] = te; }
                            n_pend++;
                        } else {
                            account_done(rh.pk, rh.tpf, te);
                        }
                        Kdrop += job_P(rh.pk) + job_D(rh.pk);
                        __syncwarp();
                    }
                    if (lane == 0) {
                        if (h != last) { fin[h] = fl; rec[h] = rl; }
                        if (last > 0) { rl = rec[last - 1]; fl = fin[last - 1]; }      // for the next one, if there is one
                    }
                    n = last;
                }
            }
        }
        newmin = __reduce_min_sync(FULL, newmin);
        if (lane == owner) {
            ndec[g] = (uint16_t)n;
            nfin[g] = newmin;
            if (f_kappa()) K[g] -= Kdrop;
        }
        decodes_changed(g);
        __syncwarp();
    }

    // The record that was on its way joins the staged ones.
    __device__ __forceinline__ void stage_late()
    {
        if (!has_late) return;
        if (lane == 0) { SlotRec r; r.tpf = late_tpf; r.pk = late_pk; r.pad = 0; st_rec[n_pend] = r; }
        n_pend++;
        has_late = false;
    }

    // --- end of an iteration on GPU g (warp-wide path: the end is not local) ----------------------
    // nd_before: decodes that g held before this event's retirements (one warp: the round's passes have ended the iteration)
    // na_ev: its batch word; pk_ev, tarr_ev: the request whose prefill has ended (CAL: it was read when the end was loaded)
    __device__ __forceinline__ void on_server(uint32_t g, uint32_t nd_before, uint32_t na_ev, uint32_t pk_ev, double tarr_ev)
    {
        const int owner = (int)(g & 31u);
        uint32_t flags = 0, itg = 0, nd = 0;
        if (SPL > 0 || CAL) {      // (one warp, unrolled rows or calendar)
            // the round's passes have ended the iteration and retired its finished decodes; the frozen batch
            // flags say what the end brought
            flags = na_ev >> 14;
            nd = nd_before;
        } else {
            if (lane == owner) {
                itg = it[g] + 1;
                it[g] = itg;
                const uint32_t na = nact[g] & BATCH_MASK, pc = pfcur[g], Kg = f_kappa() ? K[g] : 0u;
                const double tau = iter_time(p, pc, na, Kg, f_kappa());     // duration of the iteration that ends (the chain of its start)
                if (pc > 0) { it_mixed++; busy_mixed = __dadd_rn(busy_mixed, tau); }
                else        { it_solo++;  busy_solo = __dadd_rn(busy_solo, tau); }
                if (f_kappa()) K[g] = Kg + na;
                tnext[g] = dinf();
                nd = ndec[g];
                if (nfin[g] == itg) flags |= 1u;
                if (pc > 0) {
                    const uint32_t rem = pfrem[g] - pc;
                    pfrem[g] = (uint16_t)rem;
                    if (rem == 0) flags |= 2u;
                }
                pfcur[g] = 0;
            }
            flags = __shfl_sync(FULL, flags, owner);
            if (flags & 1u) {
                itg = __shfl_sync(FULL, itg, owner);
                nd = __shfl_sync(FULL, nd, owner);
                retire_decodes(g, itg, nd, t);
            }
        }
        if (flags & 1u) {
            drain_dirty = true;
            gate_dirty = true;   // a promoted GPU at the cap may now take a prefill
            if (!(flags & 2u) && g < M && pfrem[g] == 0 && nd > p.B - 1 && ndec[g] <= p.B - 1) {
                // Only g changed: its idle prefill slot counts again once its decodes fit under the mixed cap (a prefill
                // that finishes in this event is counted below, with the decode count after the retirement).
                n_idle_pf++;
                idle_hint = (n_idle_pf == 1) ? g : NONE32;
            }
        }
        if (flags & 2u) {
            // prefill finished: the request goes to the decode stage (place())
            const uint32_t pk = CAL ? pk_ev : pfjob[g], i = job_cls(pk);
            d_tarr = CAL ? tarr_ev : pf_tarr[g];
            const uint32_t nd_now = ndec[g];
            uint32_t pool = 0;
            // SLI-aware router: one uniform per finished prefill decides the pool
            if (f_sli()) pool = (__shfl_sync(FULL, pools, (int)i) >> ((uint32_t)cs[i].sli_ord & 31u)) & 1u;
            __syncwarp();   // every lane has read the finished job before its owner clears it
            if (lane == owner) pfjob[g] = 0;
            prefill_changed(g);
            // No router (immediate same-slot decoding, an ablation of the paper's EC): the request goes on decoding on
            // g, in the slot it holds; it passes through the empty buffer at this instant.
            const bool immediate = (F & F_GENERIC) && p.router == 3;
            // the prefill slot of g is idle again
            if (g < M && nd_now + (immediate ? 1u : 0u) <= p.B - 1) {
                n_idle_pf++;
                idle_hint = (n_idle_pf == 1) ? g : NONE32;
            }
            // Decode stage.  With an empty buffer the request is its head at once and the dispatch places it if a slot is free.
            d_pool = pool;
            d_pk = pk & 0x7fffffffu;
            d_gpu = immediate ? g : NONE32;
            handed = true;
            // (The solo pool is served first; under random placement both pools draw from one sequence, so a request of the
            // mixed pool waits its turn behind a backlog of the solo pool, which new targets may have made room for.)
            direct = immediate || ((pool ? dq_n1 : dq_n0) == 0 && !(f_random() && pool == 1u && dq_n0 != 0));
            drain_dirty = true;
            gate_dirty = true;
        }
        touch_server(g);
    }

    // --- local end of an iteration (owner lane only) ----------------------------------------------------
    // The iteration of GPU g ends at te and nothing outside g depends on it.  Returns true when a decode
    // finished: the GPU then waits for retire_decodes before it starts its next iteration.
    // evt: the end is the round's non-local event; the GPU is then not restarted here (the event's handler and
    // the dispatch that follows may change its batch first).
    __device__ __forceinline__ bool local_end(uint32_t g, double te, bool act = true, bool evt = false)
    {
        // straight-line: all fields are read first and the stores are predicated on `act` (see start_at)
        const uint32_t it0 = it[g], na_raw = nact[g], nd = ndec[g], pr = pfrem[g], nf = nfin[g];
        const uint32_t pc = CAL ? ((na_raw & BATCH_MIXED) ? min(p.C, pr) : 0u) : (uint32_t)pfcur[g];
        uint32_t K0 = 0, Kp = 0;
        if (f_kappa()) { K0 = K[g]; Kp = Kpend[g]; }
        const double tau = iter_time(p, pc, na_raw & BATCH_MASK, K0, f_kappa());   // duration of the iteration that ends (the chain of its start)
        const uint32_t itg = it0 + 1u;
        const uint32_t rem = pr - pc;                       // prompt tokens left after this iteration's chunk
        const bool retire = (na_raw & 0x4000u) != 0;        // a decode finished: the GPU waits for retire_decodes
        const bool has_pf = rem != 0;                       // (the end of a prefill is never local: rem > 0 while one runs)
        const bool restart = !retire && !evt && (nd != 0 || has_pf);
        // restart at te with what the GPU holds now (requests placed meanwhile join here)
        const uint32_t Kend = K0 + (na_raw & BATCH_MASK);
        const uint32_t Kg = Kend + Kp;
        const uint32_t pc2 = has_pf ? min(p.C, rem) : 0u;
        uint32_t fl = (nf == itg + 1u) ? 0x4000u : 0u;
        if (pc2 > 0 && pc2 == rem) fl |= 0x8000u;
        if (CAL && pc2 > 0) fl |= BATCH_MIXED;
        const double tau2 = iter_time(p, pc2, nd, Kg, f_kappa());
        if (act) {
            it[g] = itg;
            if (pc > 0) { it_mixed++; busy_mixed = __dadd_rn(busy_mixed, tau); pfrem[g] = (uint16_t)rem; }
            else        { it_solo++;  busy_solo = __dadd_rn(busy_solo, tau); }
            if (f_kappa()) { K[g] = restart ? Kg : Kend; if (restart) Kpend[g] = 0; }
            if (!CAL) pfcur[g] = restart ? (uint16_t)pc2 : (uint16_t)0;
            if (restart) nact[g] = (uint16_t)(nd | fl);
            const double tn = __dadd_rn(te, tau2);
            tnext[g] = restart ? tn : dinf();
            if (CAL && restart) file_end(g, tn);
        }
        return act && retire;
    }

    // Counters that follow from others while a launch runs are kept as their difference from those: every request that arrived is
    // in the queue or was admitted, left or was turned away; one that was admitted is in prefill or has finished it; one that was
    // placed decodes or is done.  (Class lanes; `back` at the end of the launch.)
    __device__ __forceinline__ void derived_counters(bool back)
    {
        ClassState &c = cs[lane];
        const unsigned long long in_prefill = c.X + c.prefill_done, m = c.Ym + c.done_mixed, so = c.Ys + c.done_solo;
        const unsigned long long admitted = back ? c.admitted + in_prefill : c.admitted;
        const unsigned long long arrived = c.pq_n + admitted + c.abandoned_p + c.overflow;
        c.admitted += back ? in_prefill : 0ull - in_prefill;
        c.arrivals += back ? arrived : 0ull - arrived;
        c.placed_mixed += back ? m : 0ull - m;
        c.placed_solo += back ? so : 0ull - so;
    }

    // Class lanes of the master: add every warp's accounting of finished requests to the class records.
    __device__ void merge_warp_stats()
    {
        if (warp == 0 && lane < (int)p.I) {
            ClassState &c = cs[lane];
            for (int w = 0; w < nwarps; ++w) {
                const WarpClassStats &a = wcs[w * (int)p.I + lane];
                c.sYm_out = __dadd_rn(c.sYm_out, a.sYm_out);
                c.sYs_out = __dadd_rn(c.sYs_out, a.sYs_out);
                c.sum_tpot = __dadd_rn(c.sum_tpot, a.sum_tpot);
                c.tok_in_done += a.tok_in; c.tok_out_done += a.tok_out;
                c.done_mixed += a.done_mixed; c.done_solo += a.done_solo;
                c.Ym -= a.done_mixed; c.Ys -= a.done_solo;
            }
        }
    }

    // This warp's share (rows warp, warp + nwarps, ...) of the candidate scan; run-time row count.
    __device__ void scan_share(bool buffered, unsigned long long &bt, uint32_t &bs, unsigned long long &tmin)
    {
        const unsigned long long INF = 0x7ff0000000000000ull;
#pragma unroll 4
        for (uint32_t k = (uint32_t)warp; k < n_rows(); k += (uint32_t)nwarps) {
            // straight-line (INF is the identity of the minimum; padded GPUs never run)
            const uint32_t g = (k << 5) + (uint32_t)lane;
            const unsigned long long v = (unsigned long long)__double_as_longlong(tnext[g]);
            const uint32_t na = nact[g], nd = ndec[g];
            const bool nl = force_nonlocal || (na & 0x8000u) != 0 ||
                            ((na & 0x4000u) != 0 && (buffered || (g < M && nd > p.B - 1)));
            tmin = min(tmin, v);
            if (v < INF && nl && v < bt) { bt = v; bs = SRC_SERVER + g; }
        }
    }

    // This warp's share of the local iteration ends below the limit key, with their retirements.
    __device__ bool ends_share(unsigned long long lim_t, uint32_t lim_s, bool buffered)
    {
        bool progressed = false;
        for (uint32_t k = (uint32_t)warp; k < n_rows(); k += (uint32_t)nwarps) {
            const uint32_t g = (k << 5) + (uint32_t)lane;
            const unsigned long long v = (unsigned long long)__double_as_longlong(tnext[g]);
            bool retire = false;
            if ((v < lim_t || (v == lim_t && SRC_SERVER + g < lim_s)) && is_local(g, buffered)) {     // (the limit is finite)
                retire = local_end(g, __longlong_as_double((long long)v));
                progressed = true;
            }
            uint32_t need = __ballot_sync(FULL, retire);
            __syncwarp();   // the owners' updates of it / n_dec are visible to the whole warp
            while (need) {
                const int l = __ffs((int)need) - 1;
                need &= need - 1;
                const uint32_t gg = (k << 5) + (uint32_t)l;
                const double te = __longlong_as_double((long long)__shfl_sync(FULL, v, l));
                retire_decodes(gg, it[gg], (uint32_t)ndec[gg], te);
                if (lane == l) start_at(gg, te);
            }
        }
        return progressed;
    }

    // warp-level argmin of (time bits, source) and min of times
    __device__ __forceinline__ void warp_keys(unsigned long long bt, uint32_t bs, unsigned long long tmin,
                                              unsigned long long &tint, uint32_t &src, unsigned long long &tmin_all) const
    {
        const uint32_t hi = (uint32_t)(bt >> 32), lo = (uint32_t)bt;
        const uint32_t mhi = __reduce_min_sync(FULL, hi);
        const uint32_t mlo = __reduce_min_sync(FULL, hi == mhi ? lo : NONE32);
        src = __reduce_min_sync(FULL, (hi == mhi && lo == mlo) ? bs : NONE32);
        tint = ((unsigned long long)mhi << 32) | mlo;
        const uint32_t th = (uint32_t)(tmin >> 32);
        const uint32_t tmh = __reduce_min_sync(FULL, th);
        const uint32_t tml = __reduce_min_sync(FULL, th == tmh ? (uint32_t)tmin : NONE32);
        tmin_all = ((unsigned long long)tmh << 32) | tml;
    }

    // Helper warps (F_MW): serve the master's commands until it says stop.  Every command is bracketed by two
    // block barriers; the master executes the same two.
    __device__ void helper_loop()
    {
        const unsigned long long INF = 0x7ff0000000000000ull;
        for (;;) {
            __syncthreads();
            const uint32_t op = cmd->op;
            if (op == MW_EXIT) return;
            const bool buffered = cmd->buffered != 0;
            M = cmd->M;
            force_nonlocal = cmd->force != 0;
            if (op == MW_SCAN) {
                unsigned long long bt = INF, tmin = INF, tint, tall;
                uint32_t bs = NONE32, src;
                scan_share(buffered, bt, bs, tmin);
                warp_keys(bt, bs, tmin, tint, src, tall);
                if (lane == 0) { MwRes r; r.bt = tint; r.bs = src; r.tmin = tall; r.progressed = 0; res[warp] = r; }
            } else {
                const bool pr = ends_share(cmd->lim_t, cmd->lim_s, buffered);
                const uint32_t any = __ballot_sync(FULL, pr);
                if (lane == 0) res[warp].progressed = any != 0;
            }
            __syncthreads();
        }
    }

    // --- calendar of iteration ends (CAL) ---------------------------------------------------------------
    // Time is cut into buckets of equal width.  The GPUs whose iterations end in a bucket form a few linked lists (a new end is
    // put at the front with one atomic exchange; a lane follows each list), and no iteration is longer than cal_nbk - 2
    // buckets, so a list holds the ends of one bucket only.  The warp works through the buckets in order: load_bucket gives
    // the GPUs of a bucket to lanes that hold none; rounds then look at the lanes only.  The next bucket is loaded as soon as
    // enough lanes are free, so that the next event that is not local is usually among the held ends.  Invariant: every pending
    // event lies in bucket cur - lead or later, so an iteration that starts now ends cal_K = floor(tau_min / width) >= 1
    // buckets after that one or later, and the bucket after `cur` may be loaded while lead + 1 < cal_K.
    // F_TIGHT (cal_K = 0): one bucket at a time; every round loads what was filed in it meanwhile and ends before T_min + tau_min.
    __device__ __forceinline__ unsigned long long bucket_abs(double x) const { return __double2ull_rd(__dmul_rn(x, p.cal_inv_w)); }
    __device__ __forceinline__ void file_end(uint32_t g, double te)
    {
        const uint32_t b = (uint32_t)bucket_abs(te) & (p.cal_nbk - 1u);
        cal_next[g] = (uint16_t)atomicExch(&cal_head[(b << cal_lsh()) + (g & ((1u << cal_lsh()) - 1u))], g);
    }

    // Give the GPUs whose ends lie in bucket b to the free lanes (mine: this lane's, or NONE32); returns how many there are (nothing
    // is taken when there are more than free lanes).
    __device__ __forceinline__ uint32_t load_bucket(unsigned long long b, uint32_t free_lanes, uint32_t &mine)
    {
        const uint32_t below = (1u << lane) - 1u;
        uint32_t *head = cal_head + (((uint32_t)b & (p.cal_nbk - 1u)) << cal_lsh()) + (uint32_t)lane;
        uint32_t n = 0, g = ((uint32_t)lane >> cal_lsh()) == 0 ? *head : CAL_NONE;
#pragma unroll 1
        for (uint32_t k = __ballot_sync(FULL, g != CAL_NONE); k && n <= 32u; k = __ballot_sync(FULL, g != CAL_NONE)) {
            const uint32_t pos = n + (uint32_t)__popc(k & below);
            n += (uint32_t)__popc(k);
            if (g != CAL_NONE) {
                if (pos < 32u) picked[pos] = (uint16_t)g;
                g = cal_next[g];
            }
        }
        if (n == 0 || n > (uint32_t)__popc(free_lanes)) return n;
        if (((uint32_t)lane >> cal_lsh()) == 0) *head = CAL_NONE;
        __syncwarp();
        const uint32_t rank = (uint32_t)__popc(free_lanes & below);
        if (!held && rank < n) mine = (uint32_t)picked[rank];
        __syncwarp();
        return n;
    }
    // This lane holds GPU g's pending end.  The request whose prefill it finishes is read now, rounds before it is needed (N = 512,
    // R = 4096: 569 -> 553 ms).  Asking for the stamps of the finishing decodes as well costs more than it saves (553 against 536).
    __device__ __forceinline__ void hold(uint32_t g)
    {
        held = true; held_g = g;
        held_t = (unsigned long long)__double_as_longlong(tnext[g]);
        const uint32_t na = nact[g];
        held_na = na;
        if (na & 0x8000u) { held_pk = pfjob[g]; held_tarr = pf_tarr[g]; }
    }

    // More ends in bucket `cur` than lanes (short iterations of lightly loaded GPUs, GPUs that started together): the lists are dealt out to the
    // lanes, 32 GPUs at a time; each lane keeps its earliest end and files the others again, and the earliest of those limits
    // the round.  (Looking at all GPUs instead: half the load of cfg2, 32 and 20 iterations of horizon: N = 512, R = 2000 66 ms
    // against 47, N = 4096, R = 592 1093 against 142.)
    __device__ __forceinline__ uint32_t load_crowded()
    {
        const unsigned long long INF = 0x7ff0000000000000ull;
        const uint32_t below = (1u << lane) - 1u;
        if (held) file_end(held_g, __longlong_as_double((long long)held_t));
        __syncwarp();
        uint32_t g = CAL_NONE;
        if (((uint32_t)lane >> cal_lsh()) == 0) {
            uint32_t *head = cal_head + (((uint32_t)cur & (p.cal_nbk - 1u)) << cal_lsh()) + (uint32_t)lane;
            g = *head;
            *head = CAL_NONE;
        }
        unsigned long long first = INF, left_t = INF;
        uint32_t mine = NONE32, left_s = NONE32;
        held = false; held_t = INF; held_g = 0;
#pragma unroll 1
        for (uint32_t k = __ballot_sync(FULL, g != CAL_NONE); k;) {
            uint32_t n = 0;
#pragma unroll 1
            for (; k && n + (uint32_t)__popc(k) <= 32u; k = __ballot_sync(FULL, g != CAL_NONE)) {
                if (g != CAL_NONE) {
                    picked[n + (uint32_t)__popc(k & below)] = (uint16_t)g;
                    g = cal_next[g];
                }
                n += (uint32_t)__popc(k);
            }
            __syncwarp();       // (what the lanes read from the lists is read before any of it is filed again)
            if ((uint32_t)lane < n) {
                uint32_t c = (uint32_t)picked[lane];
                unsigned long long v = (unsigned long long)__double_as_longlong(tnext[c]);
                if (v < first || (v == first && c < mine)) {
                    const unsigned long long w = first;
                    const uint32_t m = mine;
                    first = v; mine = c;
                    v = w; c = m;
                }
                if (c != NONE32) {
                    file_end(c, __longlong_as_double((long long)v));
                    if (v < left_t || (v == left_t && SRC_SERVER + c < left_s)) { left_t = v; left_s = SRC_SERVER + c; }
                }
            }
            __syncwarp();
        }
        crowded = __any_sync(FULL, left_t < INF);
        const uint32_t hi = (uint32_t)(left_t >> 32), lo = (uint32_t)left_t;
        const uint32_t mhi = __reduce_min_sync(FULL, hi), mlo = __reduce_min_sync(FULL, hi == mhi ? lo : NONE32);
        left_s = __reduce_min_sync(FULL, (hi == mhi && lo == mlo) ? left_s : NONE32);
        if (lane == 0) { left[0] = ((unsigned long long)mhi << 32) | mlo; left[1] = left_s; }
        __syncwarp();
        return mine;
    }

    // Buckets from `cur` to the next one with a pending iteration end (a large number when no GPU runs).
    __device__ __forceinline__ uint32_t next_bucket() const
    {
        uint32_t best = 0x7fffffffu;
#pragma unroll 1
        for (uint32_t c = (uint32_t)lane; c < cal_lists(); c += 32u)
            if (cal_head[c] != CAL_NONE) best = min(best, ((c >> cal_lsh()) - (uint32_t)cur) & (p.cal_nbk - 1u));
        return __reduce_min_sync(FULL, best);
    }

    // Calendar from the GPU records, at kernel entry.
    __device__ __forceinline__ void calendar_build()
    {
        unsigned long long first = 0x7ff0000000000000ull;
#pragma unroll 1
        for (uint32_t c = (uint32_t)lane; c < cal_lists(); c += 32u) cal_head[c] = CAL_NONE;
#pragma unroll 1
        for (uint32_t g = (uint32_t)lane; g < p.N; g += 32u) first = min(first, (unsigned long long)__double_as_longlong(tnext[g]));
        if (lane < (int)p.I) first = min(first, class_first());
        if (f_blocks() && lane == 0) first = min(first, (unsigned long long)__double_as_longlong(T_blk_next));
        const uint32_t hi = (uint32_t)(first >> 32), mhi = __reduce_min_sync(FULL, hi);
        const uint32_t mlo = __reduce_min_sync(FULL, hi == mhi ? (uint32_t)first : NONE32);
        cur = mhi >= 0x7ff00000u ? bucket_abs(T_end) : bucket_abs(__longlong_as_double((long long)(((unsigned long long)mhi << 32) | mlo)));
        lead = 0;
        held = false; held_t = 0x7ff0000000000000ull; held_g = 0; held_na = 0; held_pk = 0; held_tarr = 0.0;
        crowded = true;      // the first round deals out this bucket
        __syncwarp();
#pragma unroll 1
        for (uint32_t g = (uint32_t)lane; g < p.N; g += 32u) {
            const double x = tnext[g];
            if (x < dinf()) file_end(g, x);
        }
        __syncwarp();
    }
    // earliest clock of this lane's class
    __device__ __forceinline__ unsigned long long class_first() const
    {
        const ClassState &c = cs[lane];
        unsigned long long v = (unsigned long long)__double_as_longlong(c.ta);
        if (f_abandon()) {
            v = min(v, (unsigned long long)__double_as_longlong(c.abp.t_ab));
            v = min(v, (unsigned long long)__double_as_longlong(c.abd0.t_ab));
            v = min(v, (unsigned long long)__double_as_longlong(c.abd1.t_ab));
        }
        return v;
    }

    // The round loop on the calendar: as run(), with the lanes' held ends in the place of all GPUs.
    // Bound: the chain of dependent instructions of each replication, about 1500 a round, and fetching them.  Measured at N = 512,
    // R = 4096, 250 iterations of horizon: 955 ms reading all rows in every round, 594 with a byte per GPU that names its bucket
    // and is searched for every bucket, 556 with lists per bucket (four; with two 2-3 % more) and one memory round trip per retirement.  The
    // instance of the occupancy gate spills no registers (8 bytes spilled in the loop cost 20 %: the L1 next to 200 KB of shared memory is too
    // small for them), and any change of the loop moves its time by 1 to 10 % through the layout of the code.
    // N = 4096, R = 1712: 702 -> 351 ms, 155 with the records in global memory.
    __device__ bool run_calendar()
    {
        const uint32_t budget = (uint32_t)min(p.event_budget, BUDGET_MAX);
        const unsigned long long INF = 0x7ff0000000000000ull;
        const unsigned long long tend_bits = (unsigned long long)__double_as_longlong(T_end);
        uint32_t want = CAL_FREE;        // free lanes to load another bucket
        calendar_build();
        for (;;) {
            const unsigned long long cur0 = cur;
            __syncwarp();
            replenish();
            unsigned long long bt = INF;
            uint32_t bs = NONE32;
            bool arrival_due = false;        // an arrival that only joins its queue is pending up to T_end
            if (f_blocks() && lane == 0 && T_blk_next < dinf()) { bt = (unsigned long long)__double_as_longlong(T_blk_next); bs = SRC_BLOCK; }
            if (lane < (int)p.I) {
                const ClassState &c = cs[lane];
                unsigned long long v = (unsigned long long)__double_as_longlong(c.ta);
                arrival_due = v <= tend_bits;
                if ((n_idle_pf > 0 || force_nonlocal) && v < bt) { bt = v; bs = SRC_ARRIVAL + lane; }
                if (f_abandon()) {
                    v = (unsigned long long)__double_as_longlong(c.abp.t_ab);
                    if (v < bt) { bt = v; bs = SRC_ABP + lane; }
                    v = (unsigned long long)__double_as_longlong(c.abd0.t_ab);
                    if (v < bt) { bt = v; bs = SRC_ABD0 + lane; }
                    v = (unsigned long long)__double_as_longlong(c.abd1.t_ab);
                    if (v < bt) { bt = v; bs = SRC_ABD1 + lane; }
                }
            }
            // Load buckets (one copy of the code for every reason to): the current one again when it is crowded; the next one that
            // holds an event when no lane holds an end any more; the following one when enough lanes are free.
            bool look = crowded, again = TIGHT && !crowded;
            uint32_t turn = 0, d = 0;
#pragma unroll 1
            for (;;) {
                const uint32_t free_lanes = ~__ballot_sync(FULL, held);
                uint32_t ahead = 0, mine = NONE32, n = 0;
                const bool all = look;
                look = false;
                if (all) {
                    mine = load_crowded();
                } else if (TIGHT && again) {
                    again = false;       // (ends that were filed in the current bucket meanwhile)
                } else if (free_lanes == FULL && !crowded) {
                    if (turn == 0) {
                        // buckets to the first class event or block end
                        unsigned long long first = bt;
                        if (lane < (int)p.I) first = min(first, (unsigned long long)__double_as_longlong(cs[lane].ta));
                        d = 0x7fffffffu;
                        if (first < INF) {
                            const unsigned long long b = bucket_abs(__longlong_as_double((long long)first));
                            d = b <= cur ? 0u : (uint32_t)min(b - cur, 0x7fffffffull);
                        }
                        d = __reduce_min_sync(FULL, d);
                        if (d == 0) break;
                        ++cur; --d;
                    } else {
                        if (d == 0) break;
                        const uint32_t skip = min(next_bucket(), d);
                        if (skip >= 0x7ffffffeu) {
                            // no GPU runs and d is at its cap: go to the first class event or block end, however far it is
                            unsigned long long first = bt;
                            if (lane < (int)p.I) first = min(first, (unsigned long long)__double_as_longlong(cs[lane].ta));
                            const uint32_t hi = (uint32_t)(first >> 32), mhi = __reduce_min_sync(FULL, hi);
                            const uint32_t mlo = __reduce_min_sync(FULL, hi == mhi ? (uint32_t)first : NONE32);
                            first = ((unsigned long long)mhi << 32) | mlo;
                            if (first > tend_bits) return true;
                            cur = bucket_abs(__longlong_as_double((long long)first));
                        } else {
                            if (cur + skip > bucket_abs(T_end)) return true;      // nothing left up to T_end
                            if (skip == 0) break;
                            cur += skip;
                        }
                        d = 0;
                    }
                    lead = 0;
                    want = CAL_FREE;
                    ++turn;
                } else {
                    if (turn || crowded || (uint32_t)__popc(free_lanes) < want || lead + 1u >= p.cal_K) break;
                    ahead = 1;
                }
                if (!all) n = load_bucket(cur + ahead, free_lanes, mine);
                if (mine != NONE32) hold(mine);
                if (ahead) {
                    if (n <= (uint32_t)__popc(free_lanes)) { ++cur; ++lead; want = CAL_FREE; }
                    else want = min(n, 32u);            // (more than 32: it has to wait until no lane holds anything)
                    break;
                }
                look = n > (TIGHT ? (uint32_t)__popc(free_lanes) : 32u);
            }
            const bool buffered = (dq_n0 | dq_n1) != 0;
            const uint32_t na = held_na, nd0 = ndec[held_g];
            const bool nl = force_nonlocal || (na & 0x8000u) != 0 || ((na & 0x4000u) != 0 && (buffered || (held_g < M && nd0 > p.B - 1)));
            if (held && nl && held_t < bt) { bt = held_t; bs = SRC_SERVER + held_g; }
            unsigned long long tint;
            uint32_t src;
            {
                const uint32_t hi = (uint32_t)(bt >> 32), lo = (uint32_t)bt;
                const uint32_t mhi = __reduce_min_sync(FULL, hi);
                const uint32_t mlo = __reduce_min_sync(FULL, hi == mhi ? lo : NONE32);
                src = __reduce_min_sync(FULL, (hi == mhi && lo == mlo) ? bs : NONE32);
                tint = ((unsigned long long)mhi << 32) | mlo;
            }
            const unsigned long long left_t = crowded ? left[0] : INF;
            if (tint > tend_bits && left_t > tend_bits && cur >= bucket_abs(T_end) && !__any_sync(FULL, arrival_due || held_t <= tend_bits)) return true;
            if (rounds == budget) return false;
            ++rounds;
            // a class event further ahead waits until its bucket is the current one
            const bool here = tint < INF && (src >= SRC_SERVER || bucket_abs(__longlong_as_double((long long)tint)) <= cur);
            unsigned long long lim_t = here ? tint : INF;
            uint32_t lim_s = here ? src : NONE32;
            if (crowded) {
                const uint32_t left_s = (uint32_t)left[1];
                if (left_t < lim_t || (left_t == lim_t && left_s < lim_s)) { lim_t = left_t; lim_s = left_s; }
            }
            if (TIGHT) {
                // no iteration that starts in this round can end before T_min + tau_min
                unsigned long long tmin = held_t;
                if (lane < (int)p.I) tmin = min(tmin, (unsigned long long)__double_as_longlong(cs[lane].ta));
                const uint32_t hi = (uint32_t)(tmin >> 32), mhi = __reduce_min_sync(FULL, hi);
                const uint32_t mlo = __reduce_min_sync(FULL, hi == mhi ? (uint32_t)tmin : NONE32);
                if (mhi < 0x7ff00000u) {
                    const unsigned long long wt = (unsigned long long)__double_as_longlong(__dadd_rn(__hiloint2double((int)mhi, (int)mlo), tau_min));
                    if (wt <= lim_t) { lim_t = wt; lim_s = 0; }
                }
            }
            const bool first_is_event = here && lim_t == tint && lim_s == src;      // nothing that is not held or could still start comes before it
            if (tend_bits < lim_t) { lim_t = tend_bits; lim_s = NONE32; }
            bool progressed = false;
            const bool first_here = first_is_event && tint <= tend_bits, arrival_now = first_here && src >= SRC_ARRIVAL && src < SRC_ABP;
            const bool local = n_idle_pf == 0 && !force_nonlocal;
            bool redo = false;
            if ((local || arrival_now) && lane < (int)p.I) {
                // local arrivals of this lane's class, or the arrival that is the round's event (see run())
                const ClassState &c = cs[lane];
#pragma unroll 1
                for (int guard = 0;; ++guard) {
                    const unsigned long long v = (unsigned long long)__double_as_longlong(c.ta);
                    if (local) {
                        if (!(v < lim_t || (v == lim_t && SRC_ARRIVAL + (uint32_t)lane < lim_s))) break;
                        if (f_abandon()) {
                            if (stale & 1u) { cs[lane].abp.t_ab = next_abandonment(cs[lane].abp, cs[lane].pq_n); stale &= ~1u; }
                            if (v > (unsigned long long)__double_as_longlong(c.abp.t_ab)) break;
                        }
                        if (bucket_abs(__longlong_as_double((long long)v)) > cur) break;
                    } else if (!(arrival_now && src == SRC_ARRIVAL + (uint32_t)lane && guard == 0)) break;
                    if (guard == ARRIVALS_PER_ROUND) { redo = true; break; }
                    arrival_local();
                    progressed = true;
                }
            }
            redo = redo || (sched_pending && !arrival_now);
            if (f_abandon() && lane < (int)p.I) redo = redo || abandons_before(tint, src);
            const bool any_redo = __any_sync(FULL, redo);
            const bool do_event = !any_redo && first_here;
            // the held ends below the limit and, if it happens now, the event's end
            const unsigned long long v = held_t;
            const uint32_t g = held_g;
            const bool evt = do_event && held && SRC_SERVER + g == src;
            const bool act = evt || (held && !nl && (v < lim_t || (v == lim_t && SRC_SERVER + g < lim_s)));
            const uint32_t ev_lane = __ballot_sync(FULL, evt);       // the lane that holds the event's end, if it is one
            const bool retire = local_end(g, __longlong_as_double((long long)v), act, evt);
            if (act) { held = false; held_t = INF; progressed = true; }
            uint32_t need = __ballot_sync(FULL, retire);
            if (need) {
                __syncwarp();   // the lanes' updates of it / n_dec are visible to the whole warp
                do {
                    const int l = __ffs((int)need) - 1;
                    need &= need - 1;
                    const uint32_t gg = __shfl_sync(FULL, g, l);
                    const double te = __longlong_as_double((long long)__shfl_sync(FULL, v, l));
                    retire_decodes(gg, it[gg], (uint32_t)ndec[gg], te);
                } while (need);
                start_at(g, __longlong_as_double((long long)v), retire && !evt);
            }
            if (do_event) {
                t = __longlong_as_double((long long)tint);
                lead = min(lead, (uint32_t)(cur - min(cur, bucket_abs(t))));
                if (src >= SRC_SERVER) {
                    const int l = __ffs((int)ev_lane) - 1;
                    on_server(src - SRC_SERVER, __shfl_sync(FULL, nd0, l), __shfl_sync(FULL, na, l), __shfl_sync(FULL, held_pk, l), __shfl_sync(FULL, held_tarr, l));
                } else {
                    if (f_abandon() && src >= SRC_ABP) on_abandon((src - SRC_ABP) >> 3, (src - SRC_ABP) & 7u);
                    else if (src >= SRC_ARRIVAL) gate_dirty = true;
                    else { ++events; load_block(blk + 1); drain_dirty = true; gate_dirty = true; n_idle_pf = count_idle_pf(); idle_hint = NONE32; }
                }
                if (err) return true;
                dispatch();
                force_nonlocal = false;
            } else if (!any_redo && cur == cur0 && !__any_sync(FULL, progressed)) {
                err = ERR_INTERNAL;     // a round that brought nothing: never spin
                return true;
            }
        }
    }

    // --- round loop ----------------------------------------------------------------------------------
    __device__ bool run()
    {
        const uint32_t budget = (uint32_t)min(p.event_budget, BUDGET_MAX);
        const uint32_t rows = n_rows();
        const unsigned long long INF = 0x7ff0000000000000ull;
        const unsigned long long tend_bits = (unsigned long long)__double_as_longlong(T_end);
        for (;;) {
            __syncwarp();
            replenish();
            // next non-local event of this lane (sources scanned in id order with '<' keep the tie order);
            // an arrival is local while no prefill slot is idle: it only joins its class queue
            unsigned long long bt = INF, tmin = INF;
            uint32_t bs = NONE32;
            if (f_blocks() && lane == 0 && T_blk_next < dinf()) { bt = (unsigned long long)__double_as_longlong(T_blk_next); bs = SRC_BLOCK; }
            if (lane < (int)p.I) {
                const ClassState &c = cs[lane];
                unsigned long long v = (unsigned long long)__double_as_longlong(c.ta);
                tmin = v;
                if ((n_idle_pf > 0 || force_nonlocal) && v < bt) { bt = v; bs = SRC_ARRIVAL + lane; }
                if (f_abandon()) {
                    v = (unsigned long long)__double_as_longlong(c.abp.t_ab);
                    if (v < bt) { bt = v; bs = SRC_ABP + lane; }
                    v = (unsigned long long)__double_as_longlong(c.abd0.t_ab);
                    if (v < bt) { bt = v; bs = SRC_ABD0 + lane; }
                    v = (unsigned long long)__double_as_longlong(c.abd1.t_ab);
                    if (v < bt) { bt = v; bs = SRC_ABD1 + lane; }
                }
            }
            const bool buffered = (dq_n0 | dq_n1) != 0;
            constexpr int NC = SPL > 0 ? SPL : 1;       // per-row values kept in registers when the rows unroll
            unsigned long long vrow[NC];
            bool lrow[NC];
            unsigned long long tint, tmin_all;
            uint32_t src;
            if (F & F_MW) {
                // every warp scans its rows; the partial results meet in shared memory
                if (lane == 0) { cmd->op = MW_SCAN; cmd->buffered = buffered; cmd->M = M; cmd->force = force_nonlocal; }
                __syncthreads();
                scan_share(buffered, bt, bs, tmin);
                warp_keys(bt, bs, tmin, tint, src, tmin_all);
                if (lane == 0) { MwRes r; r.bt = tint; r.bs = src; r.tmin = tmin_all; r.progressed = 0; res[0] = r; }
                __syncthreads();
                bt = INF; bs = NONE32; tmin = INF;
                if (lane < nwarps) { bt = res[lane].bt; bs = res[lane].bs; tmin = res[lane].tmin; }
                warp_keys(bt, bs, tmin, tint, src, tmin_all);
            } else {
#pragma unroll
                for (uint32_t k = 0; k < rows; ++k) {
                    // straight-line (INF is the identity of the minimum; padded GPUs never run)
                    const uint32_t g = (k << 5) + (uint32_t)lane;
                    const unsigned long long v = (unsigned long long)__double_as_longlong(tnext[g]);
                    const uint32_t na = nact[g], nd = ndec[g];
                    const bool nl = force_nonlocal || (na & 0x8000u) != 0 ||
                                    ((na & 0x4000u) != 0 && (buffered || (g < M && nd > p.B - 1)));
                    const bool loc = v < INF && !nl;
                    if (SPL > 0) { vrow[k] = v; lrow[k] = loc; }
                    tmin = min(tmin, v);
                    if (v < INF && nl && v < bt) { bt = v; bs = SRC_SERVER + g; }
                }
                // warp argmin of (time bits, source id) over non-local events; warp min over all pending times
                warp_keys(bt, bs, tmin, tint, src, tmin_all);
            }
            if (tint > tend_bits && tmin_all > tend_bits) return true;     // nothing left up to T_end
            if (rounds == budget) return false;
            ++rounds;
            // no iteration that starts in this round can end before T_min + tau_min
            unsigned long long wt = INF;
            if (tmin_all < INF)
                wt = (unsigned long long)__double_as_longlong(__dadd_rn(__longlong_as_double((long long)tmin_all), tau_min));
            // local ends strictly before the limit key min{(T_int, src), (W, 0), (T_end, max)}
            unsigned long long lim_t = tint;
            uint32_t lim_s = src;
            if (wt <= lim_t) { lim_t = wt; lim_s = 0; }
            if (tend_bits < lim_t) { lim_t = tend_bits; lim_s = NONE32; }
            bool progressed = false;
            const bool first_here = tint < wt && tint <= tend_bits, arrival_now = first_here && src >= SRC_ARRIVAL && src < SRC_ABP;
            if (F & F_MW) {
                if (lane == 0) { cmd->op = MW_ENDS; cmd->lim_t = lim_t; cmd->lim_s = lim_s; cmd->buffered = buffered; cmd->M = M; cmd->force = force_nonlocal; }
                __syncthreads();
            }
            const bool local = n_idle_pf == 0 && !force_nonlocal;
            bool redo = false;
            if ((local || arrival_now) && lane < (int)p.I) {
                // local arrivals of this lane's class, in time order, up to the limit and up to the class's own
                // next abandonment (which each arrival moves); or the one arrival that is the round's event (it is not local,
                // so none is): nothing in the rest of the round depends on whether it joins its queue here or at the end
                const ClassState &c = cs[lane];
#pragma unroll 1
                for (int guard = 0;; ++guard) {
                    const unsigned long long v = (unsigned long long)__double_as_longlong(c.ta);
                    if (local) {
                        if (!(v < lim_t || (v == lim_t && SRC_ARRIVAL + (uint32_t)lane < lim_s))) break;
                        if (f_abandon()) {
                            if (stale & 1u) { cs[lane].abp.t_ab = next_abandonment(cs[lane].abp, cs[lane].pq_n); stale &= ~1u; }
                            if (v > (unsigned long long)__double_as_longlong(c.abp.t_ab)) break;
                        }
                    } else if (!(arrival_now && src == SRC_ARRIVAL + (uint32_t)lane && guard == 0)) break;
                    if (guard == ARRIVALS_PER_ROUND) { redo = true; break; }
                    arrival_local();
                    progressed = true;
                }
            }
            // a class that ran out of draws has an unknown next arrival, possibly before T_int, one that stopped at the bound of
            // the loop has a known one, and a local arrival may have pulled its class's next abandonment before T_int: then T_int
            // is not next after all
            redo = redo || (sched_pending && !arrival_now);
            if (f_abandon() && lane < (int)p.I) redo = redo || abandons_before(tint, src);
            // the non-local event happens in this round if it comes before anything a new iteration could bring
            const bool any_redo = __any_sync(FULL, redo);
            const bool do_event = !any_redo && first_here;
            // with unrolled rows the event GPU's iteration ends in pass 1 and its decodes retire in pass 2
            const uint32_t ev_g = (SPL > 0 && do_event && src >= SRC_SERVER) ? src - SRC_SERVER : NONE32;
            const uint32_t nd_ev = ev_g != NONE32 ? (uint32_t)ndec[ev_g] : 0u;
            // pass 1: every lane ends the local iterations of its own GPUs (straight-line over the rows)
            uint32_t retire_rows = 0;
            if (SPL == 0) {
                // run-time row count (and, with helpers, only this warp's rows): ends and retirements row by row
                if (ends_share(lim_t, lim_s, buffered)) progressed = true;
                if (F & F_MW) {
                    const uint32_t mine = __ballot_sync(FULL, progressed);
                    if (lane == 0) res[0].progressed = mine != 0;
                    __syncthreads();
                    if (lane < nwarps && res[lane].progressed) progressed = true;
                }
            }
            if (SPL > 0) {
#pragma unroll
                for (uint32_t k = 0; k < rows; ++k) {
                    const uint32_t g = (k << 5) + (uint32_t)lane;
                    const unsigned long long v = vrow[k];
                    const bool evt = g == ev_g;
                    const bool act = evt || (lrow[k] && (v < lim_t || (v == lim_t && SRC_SERVER + g < lim_s)));
                    if (local_end(g, __longlong_as_double((long long)v), act, evt)) retire_rows |= 1u << k;
                    progressed = progressed || act;
                }
            }
            if (SPL > 0) {
                // pass 2: decode completions found in pass 1, retired by the whole warp, GPU by GPU
                if (__ballot_sync(FULL, retire_rows != 0)) {
                    __syncwarp();   // the owners' updates of it / n_dec are visible to the whole warp
#pragma unroll(SPL <= 2 && (F & F_SLOTS) ? 2 : 1)
                    for (uint32_t k = 0; k < rows; ++k) {
                        uint32_t need = __ballot_sync(FULL, (retire_rows >> k) & 1u);
                        unsigned long long v = vrow[0];
#pragma unroll
                        for (uint32_t j = 1; j < (uint32_t)NC; ++j) v = j == k ? vrow[j] : v;
                        while (need) {
                            const int l = __ffs((int)need) - 1;
                            need &= need - 1;
                            const uint32_t gg = (k << 5) + (uint32_t)l;
                            const double te = __longlong_as_double((long long)__shfl_sync(FULL, v, l));
                            retire_decodes(gg, it[gg], (uint32_t)ndec[gg], te);
                        }
                    }
                    // the retired GPUs restart where their iteration ended (straight-line over the rows)
#pragma unroll
                    for (uint32_t k = 0; k < rows; ++k)
                        start_at((k << 5) + (uint32_t)lane, __longlong_as_double((long long)vrow[k]),
                                 ((retire_rows >> k) & 1u) != 0 && (k << 5) + (uint32_t)lane != ev_g);
                }
            }
            if (do_event) {
                t = __longlong_as_double((long long)tint);
                if (src >= SRC_SERVER) {
                    on_server(src - SRC_SERVER, nd_ev, SPL > 0 ? (uint32_t)nact[src - SRC_SERVER] : 0u, 0u, 0.0);
                } else {
                    if (f_abandon() && src >= SRC_ABP) on_abandon((src - SRC_ABP) >> 3, (src - SRC_ABP) & 7u);
                    else if (src >= SRC_ARRIVAL) gate_dirty = true;
                    else { ++events; load_block(blk + 1); drain_dirty = true; gate_dirty = true; n_idle_pf = count_idle_pf(); idle_hint = NONE32; }
                }
                if (err) return true;
                dispatch();
                force_nonlocal = false;
            } else if (!any_redo && !__any_sync(FULL, progressed)) {
                err = ERR_INTERNAL;     // a round that neither ended an iteration nor handled an event: never spin
                return true;
            }
        }
    }

    // Is the end of the running iteration of GPU g local?  Not when its prefill finishes, nor when a decode
    // finishes while requests wait in a decode buffer or while the GPU (moved into the mixed group by a block
    // switch) holds a full solo batch and could take a prefill afterwards.
    __device__ __forceinline__ bool is_local(uint32_t g, bool buffered) const
    {
        if (force_nonlocal) return false;
        const uint32_t na = nact[g];
        if (na & 0x8000u) return false;
        if ((na & 0x4000u) && (buffered || (g < M && ndec[g] > p.B - 1))) return false;
        return true;
    }
};

// shared-memory carve-up for one replication (one warp per block)
struct SmemLayout {
    uint32_t off_tnext, off_tarr, off_it, off_nfin, off_pfrem, off_pfjob, off_K, off_Kpend, off_ndec, off_nact,
        off_pfcur, off_sfin16, off_socc, img_ndec, img_nact, img_pfcur, img_pfrem, img_sfin16, img_socc, srv_bytes, off_head, off_next, off_picked, off_rows, off_left, off_cs, off_ring, off_ringpk, off_strec, off_stte, off_pqh, off_aim, off_wcs, off_cmd, off_res, total;
};

// tarr_global: the arrival times and the job words of the requests in prefill (read once per finished prefill) live in
// global memory (large clusters: shared memory is what limits the resident replications there); I: classes (sizes the
// class records and the ring of arrival draws)
__host__ __device__ inline SmemLayout smem_layout(uint32_t N, uint32_t Npad, uint32_t B, uint32_t slots_smem, uint32_t nwarps, bool kappa,
                                                  bool tarr_global, uint32_t I, uint32_t cal_lists, bool far)
{
    SmemLayout L;
    uint32_t o = 0;
    L.off_tnext = o; o += 8 * Npad;
    L.off_tarr = o; if (!tarr_global) o += 8 * Npad;
    L.off_it = o; o += 4 * Npad;
    L.off_nfin = o; o += 4 * Npad;
    L.off_pfjob = o; if (!tarr_global) o += 4 * Npad;
    L.off_K = o; if (kappa) o += 4 * Npad;        // KV-token counts exist only when the KV slope is on
    L.off_Kpend = o; if (kappa) o += 4 * Npad;
    L.off_ndec = L.img_ndec = o; o += 2 * Npad;
    L.off_nact = L.img_nact = o; o += 2 * Npad;
    // (with the calendar the chunk of the running iteration follows from its batch word: the image has it, the chip does not)
    const bool cal = cal_lists > 0;
    L.off_pfcur = L.img_pfcur = o;
    L.img_pfrem = o + 2 * Npad;
    L.off_pfrem = cal ? o : L.img_pfrem;
    o = (o + 4 * Npad + 15u) & ~15u;
    // the slot arrays of the image cover the padded GPUs; on chip only the N real ones have any (N = 16, B = 256: 16 KB of shared
    // memory instead of 24, which is 12 resident replications per SM instead of 9)
    const uint32_t words = (B + 31u) >> 5;
    L.img_sfin16 = o;
    if (far) { L.off_ndec = 0; L.off_pfrem = 2 * Npad; }       // (the other arrays are used where they are in the image)
    if (cal) o = (L.off_pfrem + 2 * Npad + 15u) & ~15u;
    L.img_socc = (L.img_sfin16 + (slots_smem ? 2 * Npad * B : 0u) + 15u) & ~15u;
    L.srv_bytes = (L.img_socc + (slots_smem ? 4 * Npad * words : 0u) + 15u) & ~15u;
    L.off_sfin16 = o; if (slots_smem) o += 2 * N * B;
    o = (o + 15u) & ~15u;
    L.off_socc = o; if (slots_smem) o += 4 * N * words;
    o = (o + 15u) & ~15u;
    L.off_head = o; o += 4 * cal_lists;       // calendar of iteration ends
    L.off_next = o; if (cal) o += 2 * Npad;
    L.off_picked = o; if (cal) o += 2 * 32;
    L.off_rows = o; if (cal) o += 3 * 4 * (Npad >> 5);
    o = (o + 15u) & ~15u;
    L.off_left = o; if (cal) o += 16;
    L.off_cs = o; o += (uint32_t)sizeof(ClassState) * I;
    o = (o + 15u) & ~15u;
    L.off_ring = o; o += 8 * 32 * I;
    L.off_ringpk = o; o += 4 * 32 * I;
    const uint32_t stage = slots_smem ? STAGE_CAP : (nwarps == 1 ? ROW_STAGE_CAP : 0);
    L.off_strec = o; o += (uint32_t)sizeof(SlotRec) * stage;
    L.off_stte = o; o += 8 * stage;
    L.off_pqh = o; o += (uint32_t)sizeof(QEntry) * I;
    L.off_aim = o; o += (uint32_t)sizeof(ClassAim) * I;
    L.off_wcs = o; o += (uint32_t)sizeof(WarpClassStats) * I * nwarps;
    o = (o + 15u) & ~15u;
    L.off_cmd = o; if (nwarps > 1) o += (uint32_t)sizeof(MwCmd);        // master and helpers only
    o = (o + 15u) & ~15u;
    L.off_res = o; if (nwarps > 1) o += (uint32_t)sizeof(MwRes) * MW_MAX;
    L.total = (o + 15u) & ~15u;
    return L;
}

template <int SPL, uint32_t F>
__device__ __forceinline__ void bind_pointers(Sim<SPL, F> &s, char *sm, const SmemLayout &L)
{
    char *const rec = Sim<SPL, F>::FAR ? s.p.srv + (size_t)s.rep * s.p.srv_bytes : sm;
    s.tnext = reinterpret_cast<double *>(rec + L.off_tnext);
    s.pf_tarr = s.p.tarr_global ? s.p.tarr_g + (size_t)s.rep * s.p.N : reinterpret_cast<double *>(sm + L.off_tarr);
    s.it = reinterpret_cast<uint32_t *>(rec + L.off_it);
    s.nfin = reinterpret_cast<uint32_t *>(rec + L.off_nfin);
    s.pfrem = reinterpret_cast<uint16_t *>(sm + L.off_pfrem);
    s.pfjob = s.p.tarr_global ? s.p.pfjob_g + (size_t)s.rep * s.p.N : reinterpret_cast<uint32_t *>(sm + L.off_pfjob);
    s.K = reinterpret_cast<uint32_t *>(rec + L.off_K);
    s.Kpend = reinterpret_cast<uint32_t *>(rec + L.off_Kpend);
    s.ndec = reinterpret_cast<uint16_t *>(sm + L.off_ndec);
    s.nact = reinterpret_cast<uint16_t *>(rec + L.off_nact);
    s.pfcur = reinterpret_cast<uint16_t *>(sm + L.off_pfcur);
    s.sfin16 = reinterpret_cast<uint16_t *>(sm + L.off_sfin16);
    s.socc = reinterpret_cast<uint32_t *>(sm + L.off_socc);
    s.cal_head = reinterpret_cast<uint32_t *>(sm + L.off_head);
    s.cal_next = reinterpret_cast<uint16_t *>(sm + L.off_next);
    s.picked = reinterpret_cast<uint16_t *>(sm + L.off_picked);
    s.row_key = reinterpret_cast<uint32_t *>(sm + L.off_rows);
    s.left = reinterpret_cast<unsigned long long *>(sm + L.off_left);
    s.cs = reinterpret_cast<ClassState *>(sm + L.off_cs);
    s.aring = reinterpret_cast<double *>(sm + L.off_ring);
    s.aring_pk = reinterpret_cast<uint32_t *>(sm + L.off_ringpk);
    s.st_rec = reinterpret_cast<SlotRec *>(sm + L.off_strec);
    s.st_te = reinterpret_cast<double *>(sm + L.off_stte);
    s.pqh = reinterpret_cast<QEntry *>(sm + L.off_pqh);
    s.aim = reinterpret_cast<ClassAim *>(sm + L.off_aim);
    s.wcs = reinterpret_cast<WarpClassStats *>(sm + L.off_wcs);
    s.cmd = reinterpret_cast<MwCmd *>(sm + L.off_cmd);
    s.res = reinterpret_cast<MwRes *>(sm + L.off_res);
    s.n_pend = 0; s.has_late = false;
    s.late_tpf = 0.0; s.late_pk = 0;
    s.rec_after = 0;
    s.ring_n = 0; s.ring_pos = 0; s.sched_pending = false;
    s.ring_blk = NONE32; s.ring_end = dinf();
    s.stale = 0; s.pools = 0; s.pools_due = false;
    s.place_base = ~0ull; s.place_w = 0;
    const Params &p = s.p;
    const size_t r = s.rep;
    s.s_fin = p.slot_fin + r * (size_t)p.N * p.B;
    s.s_rec = p.slot_rec + r * (size_t)p.N * p.B;
    s.pq = p.pq + r * (size_t)p.I * p.qcap;
    s.dq = p.dq + r * (size_t)2 * p.qcap;
    s.hist = p.hist_mem ? p.hist_mem + r * (size_t)p.I * 2 * NBIN : nullptr;
}

// Empty system at t = 0: idle GPUs, first arrival of every class scheduled, abandonment levels drawn.
__global__ void __launch_bounds__(32, 1) qsim_init_kernel(Params p)
{
    constexpr int SPLT = 0;
    constexpr uint32_t FT = F_GENERIC;
    extern __shared__ __align__(16) char sm[];
    const int lane = threadIdx.x;
    for (uint32_t rep = blockIdx.x; rep < p.R; rep += gridDim.x) {
        const SmemLayout L = smem_layout(p.Npad, p.Npad, p.B, p.slots_smem, 1, p.coef[5] != 0.0, p.tarr_global != 0, p.I, 0, false);       // (laid out as the image)
        Sim<SPLT, FT> s(p, lane, rep);
        bind_pointers(s, sm, L);
        __syncwarp();
        for (uint32_t o = lane * 4; o < L.total; o += 128) *reinterpret_cast<uint32_t *>(sm + o) = 0;
        __syncwarp();
        for (uint32_t g = lane; g < p.Npad; g += 32) { s.tnext[g] = dinf(); s.nfin[g] = NONE32; }
        if (p.slots_smem && (p.B & 31u)) {
            const uint32_t bw = (p.B + 31u) >> 5;
            for (uint32_t g = lane; g < p.Npad; g += 32) s.socc[g * bw + bw - 1] = ~0u << (p.B & 31u);
        }
        if (p.tarr_global)
            for (uint32_t g = lane; g < p.N; g += 32) { s.pf_tarr[g] = 0.0; s.pfjob[g] = 0; }
        if (lane < (int)p.I) {
            ClassState &c = s.cs[lane];
            c.ta = dinf();
            AbClock *clk[3] = { &c.abp, &c.abd0, &c.abd1 };
            const uint32_t streams[3] = { STREAM_ABANDON_P, STREAM_ABANDON_D0, STREAM_ABANDON_D1 };
            for (int k = 0; k < 3; ++k) {
                uint32_t w0, w1, w2, w3;
                draw(p, rep, (streams[k] << 8) | (uint32_t)lane, 0, w0, w1, w2, w3);
                clk[k]->acc = 0.0; clk[k]->lvl = -qlog(u53(w0, w1)); clk[k]->t_last = 0.0; clk[k]->t_ab = dinf();
                clk[k]->m = 1;
            }
        }
        __syncwarp();
        // first arrival of every class: ask for draws, let the warp fill the rings, give the unused draws back
        s.sched_pending = lane < (int)p.I && p.n_inject == 0;
        if (lane < (int)p.I) s.aring[lane * 32] = 0.0;
        __syncwarp();
        if (p.n_inject > 0 && lane < (int)p.I) s.schedule_from(0.0);
#pragma unroll 1
        for (uint32_t i = 0; i < p.I; ++i)
#pragma unroll 1
            for (uint32_t guard = 0; guard <= p.nblk && __shfl_sync(FULL, (int)s.sched_pending, (int)i) != 0; ++guard) s.refill(i);
        if (lane < (int)p.I) s.cs[lane].adraw -= s.ring_n;
        __syncwarp();
        // write everything out
        RepHeader &h = p.hdr[rep];
        for (uint32_t o = lane * 4; o < sizeof(RepHeader); o += 128)
            *reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(&h) + o) = 0;
        __syncwarp();
        if (lane < (int)p.I) h.cs[lane] = s.cs[lane];
        char *img = p.srv + (size_t)rep * p.srv_bytes;
        for (uint32_t o = lane * 16; o < L.srv_bytes; o += 512)
            *reinterpret_cast<uint4 *>(img + o) = *reinterpret_cast<const uint4 *>(sm + o);
        if (p.hist_mem)
            for (uint32_t o = lane; o < p.I * 2 * NBIN; o += 32) s.hist[o] = 0;
        __syncwarp();
    }
}

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t *a)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_u32(uint32_t *a, uint32_t v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" :: "l"(a), "r"(v) : "memory");
}
// A block waits this many times about a microsecond (minutes in all) for the chunk before its own before it gives up.
// Another block is running that chunk, so the wait lasts one chunk at most.
constexpr uint32_t CHUNK_SPIN_LIMIT = 1u << 28;

// The per-GPU image of a replication between global memory and its place on chip, in 16-byte words (IN: to shared memory).
template <bool IN>
__device__ __forceinline__ void copy16(char *sm, char *img, uint32_t bytes, uint32_t tid, uint32_t nthr)
{
    for (uint32_t o = tid * 16; o < bytes; o += nthr * 16) {
        if (IN) *reinterpret_cast<uint4 *>(sm + o) = *reinterpret_cast<const uint4 *>(img + o);
        else    *reinterpret_cast<uint4 *>(img + o) = *reinterpret_cast<const uint4 *>(sm + o);
    }
}
template <bool IN, bool CAL, bool FAR>
__device__ __forceinline__ void stage_image(char *sm, char *img, const SmemLayout &L, const Params &p, uint32_t tid, uint32_t nthr)
{
    if (!FAR) copy16<IN>(sm, img, CAL ? L.img_pfcur : L.img_sfin16, tid, nthr);
    else copy16<IN>(sm + L.off_ndec, img + L.img_ndec, 2 * p.Npad, tid, nthr);
    if (CAL) {
        // the prompt remainders, and the chunk in progress from or to the batch word
        __syncwarp();
        uint16_t *na = reinterpret_cast<uint16_t *>((FAR ? img : sm) + L.off_nact), *rem = reinterpret_cast<uint16_t *>(sm + L.off_pfrem);
        uint16_t *cur = reinterpret_cast<uint16_t *>(img + L.img_pfcur), *irem = reinterpret_cast<uint16_t *>(img + L.img_pfrem);
        uint16_t *ina = reinterpret_cast<uint16_t *>(img + L.img_nact);
        const double *tn = reinterpret_cast<const double *>((FAR ? img : sm) + L.off_tnext);
#pragma unroll 1
        for (uint32_t g = tid; g < p.Npad; g += nthr) {
            if (IN) {
                rem[g] = irem[g];
                if (cur[g] != 0) na[g] |= (uint16_t)BATCH_MIXED;
            } else {
                const uint32_t w = na[g];
                irem[g] = rem[g];
                cur[g] = tn[g] < dinf() && (w & BATCH_MIXED) ? (uint16_t)min(p.C, (uint32_t)rem[g]) : (uint16_t)0;
                ina[g] = (uint16_t)(w & ~BATCH_MIXED);
            }
        }
    }
    if (p.slots_smem) {
        copy16<IN>(sm + L.off_sfin16, img + L.img_sfin16, 2 * p.N * p.B, tid, nthr);
        copy16<IN>(sm + L.off_socc, img + L.img_socc, 4 * p.N * ((p.B + 31u) >> 5), tid, nthr);
    }
}

// Advance replications to their new end time (or until the per-launch event budget runs out).
template <int SPLT, uint32_t FT>
// One-warp instances whose slot records live in global memory need little shared memory, so registers decide how many
// replications are resident on an SM: they are compiled for at least 12 blocks per SM (at most 168 registers; the specialised
// instances spill nothing or 4 to 28 bytes, 44 in the SLI-aware one with the records in global memory, the run-time-configured ones 40 to 108; +16-24 % at
// N = 64 with thousands of replications).  Instances with the finish stamps on chip are
// limited by shared memory and keep all the registers they want (the cap cost them 13 %), but for those of up to 32 GPUs, whose
// stamps take little (N = 16, R = 8192: 133 -> 98 ms).
#ifndef QSIM_MIN_BLOCKS
#define QSIM_MIN_BLOCKS 12
#endif
#ifndef QSIM_SLOT_BLOCKS
#define QSIM_SLOT_BLOCKS 12
#endif
__global__ void __launch_bounds__((FT & F_MW) ? 32 * MW_MAX : 32, (FT & F_MW) ? 1 : ((FT & F_SLOTS) ? (SPLT == 1 ? QSIM_SLOT_BLOCKS : 1) : QSIM_MIN_BLOCKS)) qsim_run_kernel(Params p)
{
    extern __shared__ __align__(16) char sm[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t nthr = blockDim.x;
    // With nchunk = K > 1 the grid is one block per resident slot and the work is R x K units (chunk c of replication r is
    // unit c R + r), handed out in that order through a counter: replications outnumbering the slots then finish together
    // instead of leaving a last, nearly empty wave.  Chunk c of a replication starts when chunk c - 1 has published its
    // stamp; that unit was handed out earlier, so the block it waits for is running.  The chunks end at the times at
    // which K successive launches would end, so the result is theirs: that of one launch, up to the order in which the
    // fp64 sums of finished requests are added to the totals.
    __shared__ uint32_t sh_unit[2];
    __shared__ double sh_T_reset;
    const uint32_t K = p.nchunk > 1 ? p.nchunk : 1u;
    const uint32_t n_units = p.R * K;
    for (uint32_t unit = blockIdx.x;; unit += gridDim.x) {
        if (K > 1) {
            if (tid == 0) sh_unit[0] = atomicAdd(p.not_done + 1, 1u);
            if (FT & F_MW) __syncthreads(); else __syncwarp();
            unit = sh_unit[0];
            if (FT & F_MW) __syncthreads(); else __syncwarp();
        }
        if (unit >= n_units) break;
        const uint32_t rep = unit % p.R, chunk = unit / p.R;
        RepHeader &h = p.hdr[rep];
        uint32_t advance = p.advance, chunks_left = 0;
        unsigned long long horizon_iters = p.horizon_iters;
        if (K > 1) {
            if (tid == 0) {
                uint32_t ok = 1;
                if (chunk > 0) {
                    const uint32_t want = p.launch_tag + chunk;
                    for (uint32_t spins = 0; ld_acquire_u32(&h.seq) != want; ++spins) {
                        if (spins > CHUNK_SPIN_LIMIT || ld_acquire_u32(p.not_done + 2) != 0) { ok = 0; break; }
                        __nanosleep(1000);
                    }
                }
                sh_unit[1] = ok;
            }
            if (FT & F_MW) __syncthreads(); else __syncwarp();
            const uint32_t ok = sh_unit[1];
            __threadfence();
            if (FT & F_MW) __syncthreads(); else __syncwarp();
            if (!ok) {      // the chunk before this one did not finish in time: report, start nothing
                if (tid == 0) { atomicExch(p.not_done + 2, 1u); atomicAdd(p.not_done, 1u); }
                continue;
            }
            const bool first = chunk == 0 && p.advance == 1;
            chunks_left = first ? K : h.chunks_left;
            bool idle = false;
            if (!first && !h.done) advance = 0;                 // stopped on the event budget: go on to the same end time
            else if (chunks_left > 0) {
                const unsigned long long j = K - chunks_left;
                horizon_iters = p.horizon_iters * (j + 1) / K - p.horizon_iters * j / K;
                advance = 1;
                --chunks_left;
            } else idle = true;
            if (idle) {
                if (FT & F_MW) __syncthreads(); else __syncwarp();
                if (tid == 0) st_release_u32(&h.seq, p.launch_tag + chunk + 1u);
                continue;
            }
        } else if (!p.advance && h.done) continue;
        Sim<SPLT, FT> s(p, lane, rep);
        const SmemLayout L = smem_layout(p.N, p.Npad, p.B, p.slots_smem, nthr >> 5, p.coef[5] != 0.0, p.tarr_global != 0, p.I, Sim<SPLT, FT>::CAL ? s.cal_lists() : 0u, Sim<SPLT, FT>::FAR);
        s.warp = warp;
        s.nwarps = (int)(nthr >> 5);
        bind_pointers(s, sm, L);
        s.block_sync();
        // stage state: per-GPU arrays (coalesced 16-byte copies) and the class records; clear the per-warp accounting
        char *const img = p.srv + (size_t)rep * p.srv_bytes;
        stage_image<true, Sim<SPLT, FT>::CAL, Sim<SPLT, FT>::FAR>(sm, img, L, p, (uint32_t)tid, nthr);
        {
            const uint4 *src = reinterpret_cast<const uint4 *>(h.cs);
            uint4 *dst = reinterpret_cast<uint4 *>(s.cs);
            for (uint32_t o = tid; o < sizeof(ClassState) * p.I / 16; o += nthr) dst[o] = src[o];
            uint32_t *w = reinterpret_cast<uint32_t *>(s.wcs);
            for (uint32_t o = tid; o < sizeof(WarpClassStats) * p.I * (nthr >> 5) / 4; o += nthr) w[o] = 0;
        }
        s.block_sync();
        // the end time is one rounded product of the cumulative horizon: run(a); run(b) ends where run(a+b) ends
        double T_end = h.T_end;
        const unsigned long long H_total = h.H_total + (advance == 1 ? horizon_iters : 0ull);
        if (advance == 1) T_end = __dmul_rn((double)H_total, iter_time(p, 0, p.B, 0));
        if (advance == 2) T_end = p.T_abs;
        s.T_end = T_end;
        s.block_sync();       // (every thread has read the old times)
        if (tid == 0) { h.T_end = T_end; h.H_total = H_total; }
        if (tid == 0) sh_T_reset = h.T_reset;
        s.T_reset_at = &sh_T_reset;
        s.tau_min = fmin(p.coef[0], p.coef[3]);
        s.t = 0.0;
        s.load_block(h.blk);
        s.dq_head0 = h.dq_head0; s.dq_head1 = h.dq_head1; s.dq_n0 = h.dq_n0; s.dq_n1 = s.f_sli() ? h.dq_n1 : 0u;
        s.place_ord = h.place_ord; s.events = 0; s.rounds = 0; s.touch_g = 0; s.sel_ord0 = h.sel_ord0; s.sel_ord1 = h.sel_ord1;
        s.n_touch = 0; s.touch_all = false; s.need_start = 0; s.err = h.err; s.direct = false; s.handed = false;
        s.drain_dirty = true; s.gate_dirty = true;
        s.force_nonlocal = (p.force_dispatch != 0 && chunk == 0) || h.force != 0;
        s.n_idle_pf = 0;
        s.idle_hint = NONE32;
        s.it_mixed = 0; s.it_solo = 0; s.busy_mixed = 0.0; s.busy_solo = 0.0;
        bool finished = true;
        if (warp == 0) {
            if (lane < (int)p.I) s.derived_counters(false);
            s.n_idle_pf = s.count_idle_pf();
            if (lane < (int)p.I && s.cs[lane].pq_n > 0) s.pqh[lane] = s.pq[(size_t)lane * p.qcap + s.cs[lane].pq_head];
            __syncwarp();
            s.busy_mixed = h.busy_mixed[lane]; s.busy_solo = h.busy_solo[lane];
            if constexpr (Sim<SPLT, FT>::CAL) {
                finished = s.err ? true : s.run_calendar();
            } else {
                finished = s.err ? true : s.run();
            }
            s.stage_late();
            s.flush_done();
            if (FT & F_MW) {
                if (lane == 0) s.cmd->op = MW_EXIT;
                __syncthreads();
            }
        } else {
            s.helper_loop();
        }
        s.block_sync();
        s.merge_warp_stats();
        if (warp == 0 && lane < (int)p.I) s.derived_counters(true);
        if (warp == 0 && lane < (int)p.I) s.cs[lane].adraw -= s.ring_n;     // unused arrival draws are produced again next time
        s.block_sync();
        // stage back
        stage_image<false, Sim<SPLT, FT>::CAL, Sim<SPLT, FT>::FAR>(sm, img, L, p, (uint32_t)tid, nthr);
        {
            uint4 *dst = reinterpret_cast<uint4 *>(h.cs);
            const uint4 *src = reinterpret_cast<const uint4 *>(s.cs);
            for (uint32_t o = tid; o < sizeof(ClassState) * p.I / 16; o += nthr) dst[o] = src[o];
        }
        // per-thread partial sums go to the 32 lane slots, warp after warp (a fixed order)
        for (int w = 0; w < s.nwarps; ++w) {
            if (warp == w) {
                if (w == 0) {
                    h.iters_mixed[lane] += s.it_mixed; h.iters_solo[lane] += s.it_solo;
                    h.busy_mixed[lane] = s.busy_mixed; h.busy_solo[lane] = s.busy_solo;
                } else {
                    h.iters_mixed[lane] += s.it_mixed; h.iters_solo[lane] += s.it_solo;
                    h.busy_mixed[lane] = __dadd_rn(h.busy_mixed[lane], s.busy_mixed);
                    h.busy_solo[lane] = __dadd_rn(h.busy_solo[lane], s.busy_solo);
                }
            }
            if (FT & F_MW) { __threadfence_block(); __syncthreads(); }
        }
        if (tid == 0) {
            if (s.f_blocks()) h.blk = s.blk;
            // (what an instance does not change is not written: it would be carried in registers through the whole run)
            h.dq_head0 = s.dq_head0; h.dq_n0 = s.dq_n0;
            if (s.f_sli()) { h.dq_head1 = s.dq_head1; h.dq_n1 = s.dq_n1; }
            if (s.f_random()) h.place_ord = s.place_ord;
            h.events += s.events; h.rounds += s.rounds; h.err = s.err;
            if (s.f_slig()) { h.sel_ord0 = s.sel_ord0; h.sel_ord1 = s.sel_ord1; }
            h.done = finished ? 1u : 0u;
            h.force = s.force_nonlocal ? 1u : 0u;
            if (K > 1) {
                h.chunks_left = chunks_left;
                if (chunk == K - 1u && (!finished || chunks_left > 0)) atomicAdd(p.not_done, 1u);
            } else if (!finished) atomicAdd(p.not_done, 1u);
        }
        if (K > 1) {        // hand the replication over to the unit of its next chunk
            __threadfence();
            s.block_sync();
            if (tid == 0) st_release_u32(&h.seq, p.launch_tag + chunk + 1u);
        }
        s.block_sync();
    }
}

// Zero the statistics of every replication, keep the simulated state.
__global__ void qsim_reset_kernel(Params p)
{
    const uint32_t rep = blockIdx.x * blockDim.x + threadIdx.x;
    if (rep >= p.R) return;
    RepHeader &h = p.hdr[rep];
    const double T = h.T_end;
    h.T_reset = T;
    h.events = 0;
    h.rounds = 0;
    for (int l = 0; l < 32; ++l) { h.iters_mixed[l] = 0; h.iters_solo[l] = 0; h.busy_mixed[l] = 0.0; h.busy_solo[l] = 0.0; }
    for (uint32_t i = 0; i < MAXI; ++i) {
        ClassState &c = h.cs[i];
        Area *as[3] = { &c.aQp, &c.aX, &c.aQd };
        for (int k = 0; k < 3; ++k) { as[k]->area = 0.0; as[k]->t_last = T; }
        c.sYm_in = c.sYm_out = c.sYs_in = c.sYs_out = 0.0;
        c.arrivals = c.admitted = c.prefill_done = c.placed_mixed = c.placed_solo = c.done_mixed = c.done_solo = 0;
        c.abandoned_p = c.abandoned_d = c.overflow = c.overflow_d = c.tok_in_pf = c.tok_in_done = c.tok_out_done = 0;
        c.sum_ttft = 0.0; c.sum_tpot = 0.0;
    }
    if (p.hist_mem) {
        uint32_t *hm = p.hist_mem + (size_t)rep * p.I * 2 * NBIN;
        for (uint32_t o = 0; o < p.I * 2 * NBIN; ++o) hm[o] = 0;
    }
}

}  // namespace qsimdev
