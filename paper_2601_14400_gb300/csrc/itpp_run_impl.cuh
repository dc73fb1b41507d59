// itpp_run_impl.cuh -- a run of gates in one launch.
//
// Below a few million terms a gate is a few microseconds of work, and a gate
// made of launches (scatter, merge, check, post, the select's passes: 25 of
// them, each a few microseconds even when it returns at once) spent nearly
// all of its time between them: 160 us per gate at 2^13 terms as at 2^18.
// k_run keeps a team of CTAs resident over all gates of a layer (one
// propagation: the whole grid; a batch: every instance its own team, over all
// layers) and goes from phase to phase over a barrier in global memory:
//
//   scatter   (a window's first gate) the state into the window's partitions
//   merge     the gate over every partition, in place (itpp_inplace.cuh)
//   select    the team's first CTA, once all have arrived: statistics, the next
//             normaliser, the top-M threshold from the candidates the merge
//             listed, published for the next gate
//
// so inside a window a gate costs one arrival of every CTA and one word that
// all of them wait for.  The rest is rare and decided
// on the device: a threshold outside the listed range takes radix passes over
// the state by the whole team; a merge that left children out which the bound
// then needed, or that ran out of a partition's stride, is done again from its
// unchanged input into a contiguous run.  Between launches the state is that
// contiguous run with the select applied, as every other entry point reads it.
//
// Every wait is bounded; a team that gives up stores the error and leaves.
#pragma once

#include <cstring>

#include "itpp_common.cuh"
#include "itpp_gate_body.cuh"
#include "itpp_launch.h"
#include "itpp_run.cuh"
#include "itpp_stage.cuh"
#include "itpp_team.cuh"
#include "itpp_inplace.cuh"

namespace itpp {

namespace {

constexpr uint32_t kPushBuf = 512;                // candidates a CTA lists in shared memory
constexpr int kRangeShift = 45;                   // first candidate range: T +- about 1/128 of T

// What the first CTA of a team publishes after a gate.
struct Pub {
    unsigned long long T;        // pending select: kept at or above this pattern (0: none)
    uint64_t tk[4];              // ... and at it up to this key
    unsigned long long lo, hi;   // candidate range of the next gate (hi == 0: none)
    unsigned long long thr;      // children at or below this pattern are left out
    unsigned long long n;        // logical terms
    unsigned long long base, range, rank;   // a select by the team: values pattern - base
    double rnorm;
    int all_ties, stop, full, rescatter, redo, pad;
};

// Written by every CTA during a gate; one set per gate parity, one for the
// merge that is done again.
struct Acc {
    unsigned long long kept, out_max, alloc, pad;
    unsigned int cand_n, over, n_long, scatter_over;
};

}  // namespace

struct RunShared {
    TeamHead head;
    Pub pub;
    Acc acc[2][2];
    unsigned int sel_n;          // select by the team: entries gathered
    unsigned int pad;
    unsigned int hist[3][kBins];
};

namespace {

using Team = TeamOf<RunShared>;

// Publish a block prepared in shared memory (the first CTA's first warp, whose
// thread 0 wrote it, calls it).
__device__ __forceinline__ void publish(const Team& t, const Pub* s_next) {
    constexpr int N = sizeof(Pub) / 8;
    __syncwarp();
    if (threadIdx.x < N)
        __stcg(reinterpret_cast<unsigned long long*>(&t.rs->pub) + threadIdx.x,
               reinterpret_cast<const unsigned long long*>(s_next)[threadIdx.x]);
    __syncwarp();
    if (threadIdx.x == 0)
        asm volatile("st.release.gpu.global.u32 [%0], %1;" :: "l"(&t.rs->head.seq), "r"(t.seq + 1u) : "memory");
}

// Wait for the next publication and copy it (every thread calls it).
__device__ __forceinline__ bool take_pub(Team& t, DevCtl* ctl, Pub* s_pub) {
    static_assert(sizeof(Pub) % 8 == 0 && sizeof(Pub) <= 256, "one load per lane");
    constexpr int N = sizeof(Pub) / 8;
    __shared__ int s_ok;
    t.seq += 1u;
    __syncthreads();   // the last one's readers are done
    if (threadIdx.x < 32) {
        int ok = 0;
        if (threadIdx.x == 0) {
            ok = wait_for(&t.rs->head.seq, t.seq, &t.rs->head, ctl);
            s_ok = ok;
        }
        __syncwarp();
        if (threadIdx.x < N)
            reinterpret_cast<unsigned long long*>(s_pub)[threadIdx.x] =
                __ldcg(reinterpret_cast<const unsigned long long*>(&t.rs->pub) + threadIdx.x);
    }
    __syncthreads();
    return s_ok != 0;
}

// ---------------------------------------------------------------------------
// Candidates of a merge: a shared list per CTA, then the global one.
// ---------------------------------------------------------------------------
struct PushList {
    unsigned long long* v;   // shared [kPushBuf]
    uint32_t* idx;
    uint32_t* n;             // shared: claims (past kPushBuf: the list is full)
    uint32_t* staged;        // shared: entries in the list
    unsigned long long* gv;  // the team's list
    uint32_t* gidx;
    unsigned int* gn;        // its length (claims; past the end: the list overflowed)
    uint64_t cap;
};

__device__ __forceinline__ void push_cand(const PushList& p, bool hit, unsigned long long v,
                                          uint64_t idx) {
    const unsigned int m = __ballot_sync(0xffffffffu, hit);
    if (!m) return;
    const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
    const uint32_t nb = __popc(m), r = __popc(m & ((1u << lane) - 1u));
    uint32_t q = 0;
    if (lane == leader) q = atomicAdd(p.n, nb);
    q = __shfl_sync(0xffffffffu, q, leader);
    if (q + nb <= kPushBuf) {
        if (hit) {
            p.v[q + r] = v;
            p.idx[q + r] = (uint32_t)idx;
        }
        if (lane == leader) atomicAdd(p.staged, nb);
        return;
    }
    // no room: straight to the global list.  No later claim fits either (the
    // count only grows), so the staged entries are a prefix of the list.
    if (lane == leader) q = atomicAdd(p.gn, nb);
    q = __shfl_sync(0xffffffffu, q, leader);
    if (hit && (uint64_t)q + r < p.cap) {
        p.gv[q + r] = v;
        p.gidx[q + r] = (uint32_t)idx;
    }
}

// ---------------------------------------------------------------------------
// The run
// ---------------------------------------------------------------------------
// The prediction's state between gates (kept by the first CTA's thread 0, in
// the control block between launches).
struct Predict {
    unsigned long long tprev;
    int shift, reason;
    unsigned long long cands, range, full;   // statistics
};

// The candidate range around the threshold predicted for the next gate: C +-
// 2^s in pattern units, narrower when the list ran long, wider when the
// threshold fell outside.  C is this threshold moved by what the next gate's
// moved in the last layer (dn), or, without that, carried into the next gate's
// scale.
__device__ __forceinline__ void next_range(Predict* q, uint64_t cand_hi, long long* drift_now,
                                           long long dn, unsigned long long T, double rnorm,
                                           uint32_t cn, unsigned long long dbits, Pub* p) {
    if (drift_now) *drift_now = q->tprev ? (long long)(T - q->tprev) : 0LL;
    q->tprev = T;
    q->cands += cn;
    int sft = q->shift ? q->shift : kRangeShift;
    switch (q->reason) {
        case 0: if (cn > cand_hi) sft -= 1; break;
        case 1: sft = kRangeShift; break;
        case 2: sft -= 2; break;
        default: sft += 1; break;
    }
    sft = sft < 8 ? 8 : (sft > kRangeShiftMax ? kRangeShiftMax : sft);
    q->shift = sft;
    unsigned long long C;
    if (dn != 0LL) {
        const long long c = (long long)T + dn;
        C = c > 0 ? (unsigned long long)c : 0ULL;
    } else {
        C = abs_pattern(__dmul_rn(__longlong_as_double((long long)T), rnorm));
    }
    const SelRange r = sel_range(C, sft, dbits);
    p->thr = r.thr;
    p->lo = r.thr + 1ULL;
    p->hi = r.hi;
}

template <int W>
__device__ __forceinline__ GateArg<W> gate_arg_of(const RunGate<W>& r, int maxw) {
    GateArg<W> g;
#pragma unroll
    for (int w = 0; w < W; ++w) { g.qx[w] = r.qx[w]; g.qz[w] = r.qz[w]; }
    g.ch = r.ch;
    g.msh = r.msh;
    g.qyy = 0;   // the sign here comes from commute_sign
    g.maxw = maxw;
    return g;
}

// The partition function of the window of level `lv` that starts at a gate,
// or of its pair key (lv < 0).
template <int W>
__device__ __forceinline__ PartFn<W> part_fn_of(const RunGate<W>& r, int lv) {
    PartFn<W> f;
    bool found = false;
#pragma unroll
    for (int w = 0; w < 2 * W; ++w) {
        const uint64_t m = w < W ? r.qx[w] : r.qz[w - W];
        const uint64_t bit = (!found && m) ? (m & (~m + 1)) : 0ULL;
        if (w < W) f.px[w] = bit; else f.pz[w - W] = bit;
        found = found || m;
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const uint64_t win = lv < 0 ? 0ULL : (lv ? r.win[1][w] : r.win[0][w]);
        f.kx[w] = ~win;
        f.kz[w] = ~win;
    }
    f.pair = lv < 0;
    f.sites = lv < 0 ? 0 : (lv ? r.sites[1] : r.sites[0]);
    return f;
}

// Cursors lie a line apart: a scatter makes an atomic per term, and those on
// one line follow one another (20 us against 5 us for 2^18 terms into 608
// partitions with packed cursors).
constexpr uint32_t kPad = kRunPad;

// The instance's arrays (by compare-select: a dynamic index into an array of
// pointers would put it in local memory).
template <int W>
struct Arrays {
    PKey<W>*k0, *k1, *kp;
    double *c0, *c1, *cp;
    unsigned int* n0;   // three cursor arrays of `pm` entries, kPad apart
    uint32_t pm;
    int a;              // the contiguous state's buffer at the start
    __device__ __forceinline__ PKey<W>* run_keys(int b) const { return b ? k1 : k0; }
    __device__ __forceinline__ double* run_coef(int b) const { return b ? c1 : c0; }
    __device__ __forceinline__ PKey<W>* home(int h) const { return h ? run_keys(a ^ 1) : kp; }
    __device__ __forceinline__ double* coef(int x) const { return x ? run_coef(a ^ 1) : cp; }
    __device__ __forceinline__ unsigned int* cnt(int p) const { return n0 + (uint64_t)p * pm * kPad; }
};

// Which window a scatter at this gate prepares: the long one (level 0) while
// the groups, the strings with one pattern outside it, are small (as the
// separate scatter decides it), else the three-site one (level 1), whose
// groups of at most 64 strings balance over partitions whatever the state,
// if there are a few groups to a partition; else the gate's pair key (-1).  A
// single partition holds any window.
template <int W>
__device__ __forceinline__ int window_level(const RunGate<W>& r, int n_sites, uint64_t n,
                                            uint64_t parts) {
    if (r.len[0] > 0 && (parts == 1 || window_fits(n_sites, r.sites[0], n))) return 0;
    if (r.len[1] > 0) {
        const int free_bits = 2 * (n_sites - r.sites[1]);
        if (free_bits >= 40 || (1ULL << (free_bits < 0 ? 0 : free_bits)) >= 4ULL * parts)
            return 1;
    }
    return -1;
}

// Run gates [0, n_gates) n_layers times on one instance.  Returns false when
// a wait ran out.
template <int W>
__device__ bool run_instance(const RunArgs<W>& a, const RunGate<W>* gates, int n_gates, int inst,
                             Team& team) {
    using A = InPass<W>;
    constexpr uint32_t C = A::C;
    __shared__ Pub s_pub, s_next;
    // raw storage: a shared variable gets no constructor, and GateArg has a
    // default member initialiser
    __shared__ __align__(16) unsigned char s_g_raw[sizeof(GateArg<W>)];
    GateArg<W>& s_g = *reinterpret_cast<GateArg<W>*>(s_g_raw);
    __shared__ PartFn<W> s_f;
    __shared__ unsigned long long s_cv[kPushBuf];
    __shared__ uint32_t s_ci[kPushBuf];
    __shared__ uint32_t s_cn, s_cs, s_app, s_rare, s_n, s_try;
    __shared__ int s_over;
    __shared__ unsigned long long s_at;
    __shared__ uint32_t s_red[kBlock / 32], s_kept[kBlock / 32], s_w[kBlock / 32];
    // first CTA: statistics of the run, counters of the gate
    __shared__ unsigned long long s_stat[8];
    __shared__ Acc s_acc;
    __shared__ double s_norm, s_rnorm;
    __shared__ int s_status;
    __shared__ long long s_dn;
    __shared__ Predict s_pred;
    __shared__ PickOut s_pick;
    __shared__ unsigned int s_long;

    DevCtl* ctl = a.ctl + inst;
    RunShared* rs = team.rs;
    const bool leader = team.rank == 0;
    Arrays<W> arr;
    arr.k0 = a.k[0] + (uint64_t)inst * a.buf_stride;
    arr.k1 = a.k[1] + (uint64_t)inst * a.buf_stride;
    arr.kp = a.kp + (uint64_t)inst * a.part_stride;
    arr.c0 = a.c[0] + (uint64_t)inst * a.buf_stride;
    arr.c1 = a.c[1] + (uint64_t)inst * a.buf_stride;
    arr.cp = a.cp + (uint64_t)inst * a.part_stride;
    arr.n0 = a.cnt + (uint64_t)inst * 3 * a.part_max * kPad;
    arr.pm = a.part_max;
    arr.a = ctl->cur;
    // candidates and ties share the merge table's memory
    char* scr = static_cast<char*>(a.scratch) + (uint64_t)inst * a.scratch_stride;
    unsigned long long* cand_v = reinterpret_cast<unsigned long long*>(scr);
    uint32_t* cand_i = reinterpret_cast<uint32_t*>(scr + a.cand_cap * 8);
    PKey<W>* ties = reinterpret_cast<PKey<W>*>(scr + a.tie_off);
    long long* drift = a.drift + (uint64_t)inst * (a.drift_stride);
    const int n_drift = a.gates ? n_gates : a.drift_gates;
    const int sites = a.n ? a.n[inst] : a.one_n;

    const PushList pl{s_cv, s_ci, &s_cn, &s_cs, cand_v, cand_i, nullptr, a.cand_cap};

    // start: the published state from the control block, the cursor arrays
    // zero, no chain head of an earlier use
    if (threadIdx.x < 8) s_stat[threadIdx.x] = 0ULL;
    if (threadIdx.x == 0) g_delta = a.delta_bits;
    inplace_init<W, kBlock, 12>();
    for (uint32_t i = team.rank * kBlock + threadIdx.x; i < 3u * a.part_max; i += team.size * kBlock)
        arr.n0[(uint64_t)i * kPad] = 0u;
    if (leader && threadIdx.x == 0) {
        Pub& first = s_next;
        memset(rs->acc, 0, sizeof rs->acc);
        memset(&first, 0, sizeof first);
        first.all_ties = 1;
        first.lo = ctl->sp_lo;
        first.hi = ctl->sp_hi;
        first.thr = ctl->sp_thr > a.delta_bits ? ctl->sp_thr : a.delta_bits;
        s_pred.tprev = ctl->sp_tprev;
        s_pred.shift = ctl->sp_shift;
        s_pred.reason = 1;
        s_pred.cands = s_pred.range = s_pred.full = 0ULL;
        first.n = live_count(ctl, arr.a);
        first.rnorm = ctl->rnorm[arr.a];
        first.stop = ctl->status != 0;
        first.rescatter = 1;
    }
    if (leader)
        for (int b = threadIdx.x; b < 3 * kBins; b += kBlock) rs->hist[0][b] = 0u;
    team_arrive(team);
    if (leader) {
        if (!team_wait(team, ctl)) return false;
        if (threadIdx.x < 32) publish(team, &s_next);
    }
    if (!take_pub(team, ctl, &s_pub)) return false;

    uint32_t tag = 0, pass = 0;
    int layout = 0, hb = 0, cx = 0, ci = 0, run_buf = arr.a;
    bool any = false;                   // a gate ran
    uint64_t run_n = s_pub.n;           // terms stored in the contiguous run
    uint32_t P = 0;
    uint64_t R = 0, n_scat = 0;         // stride; terms at the last scatter
    int win_end = 0;                    // the partitions hold for the gates before this one
    const int total = n_gates * a.n_layers;
    for (int gi = 0; gi < total; ++gi) {
        const int k = gi % n_gates;
        const int np_ = gi & 1;         // parity of this gate's counters
        if (s_pub.stop) break;          // uniform over the team
        if (threadIdx.x == 0) {
            s_g = gate_arg_of<W>(gates[k], a.maxw);
            s_cn = s_cs = s_app = s_rare = s_try = 0u;
            s_over = 0;
        }
        const GateArg<W>& g = s_g;
        const uint64_t n_in = s_pub.n;
        PKey<W> tk;
#pragma unroll
        for (int w = 0; w < W; ++w) { tk.x[w] = s_pub.tk[w]; tk.z[w] = s_pub.tk[W + w]; }
        __syncthreads();
        Acc* acc = &rs->acc[np_][0];
        // ---- scatter ----------------------------------------------------
        if (layout == 0 || gi >= win_end || s_pub.rescatter) {
            // at least a partition for every CTA of the team, of no fewer
            // than min_part terms, so that a small state uses the chip
            uint64_t want = (n_in + a.target - 1) / a.target;
            const uint64_t most = (n_in + a.min_part - 1) / a.min_part;
            const uint64_t wide = most < team.size ? most : team.size;
            if (want < wide) want = wide;
            // ... and whole rounds of the team: a round lasts as long for one
            // partition as for one each (1,498 partitions of 700 strings went
            // in 3.3 rounds of 456; four of 575: a two-layer Strang run of 2^20
            // terms 43.5 -> 41.1 ms)
            want = (want + team.size - 1) / team.size * team.size;
            if (want < 1) want = 1;
            if (want > most && want > wide) want = most > wide ? most : wide;
            if (want > a.part_max) want = a.part_max;
            // by the window, then by the pair key, then into half as many
            // partitions (of twice the stride), at last into one, which holds any
            // state; a try whose stride ran out leaves its number behind
            for (int lv = window_level<W>(gates[k], sites, n_in, want);; lv = -1) {
                if (threadIdx.x == 0) {
                    s_f = part_fn_of<W>(gates[k], lv);
                    s_try += 1u;
                }
                __syncthreads();
                PartFn<W> f = s_f;
                uint64_t np = want;
                if (lv >= 0) {   // a stride holds a whole group (up to 4^sites strings)
                    const uint64_t gmax = 1ULL << (2 * f.sites);
                    if (a.home_cap / np < gmax) np = a.home_cap / gmax > 0 ? a.home_cap / gmax : 1;
                }
                const uint32_t oldP = P;
                const uint64_t oldR = R;
                PartPlan plan;
                plan.P = (uint32_t)np;
                plan.R = a.home_cap / np;
                Pending<W> pd;
                pd.on = s_pub.T != 0ULL;
                pd.all_ties = s_pub.all_ties != 0;
                pd.T = s_pub.T;
                pd.tk = tk;
                const int dh = layout == 0 ? 0 : hb ^ 1, dx = layout == 0 ? 0 : cx ^ 1;
                const int dc = next3(ci);
                auto over = [&] { *(volatile unsigned int*)&acc->scatter_over = s_try; };
                if (layout == 0) {
                    scatter_run<W>(arr.run_keys(run_buf), arr.run_coef(run_buf), run_n,
                                   (uint64_t)team.rank * kBlock, (uint64_t)team.size * kBlock, pd,
                                   ctl, arr.home(dh), arr.coef(dx), arr.cnt(dc), plan, g, f, over, kPad);
                } else {
                    for (uint32_t p = team.rank; p < oldP; p += team.size) {
                        const uint64_t c = __ldcg(arr.cnt(ci) + (uint64_t)p * kPad);
                        scatter_run<W>(arr.home(hb) + p * oldR, arr.coef(cx) + p * oldR, c, 0,
                                       kBlock, pd, ctl, arr.home(dh), arr.coef(dx), arr.cnt(dc),
                                       plan, g, f, over, kPad);
                    }
                }
                if (!team_barrier(team, ctl)) return false;
                if (leader && threadIdx.x == 0) s_stat[4] += 1;
                const bool full = __ldcg(&acc->scatter_over) == s_try;
                if (full && plan.P == 1u && threadIdx.x == 0) set_status(ctl, ST_CAPACITY, 40);
                if (!full || plan.P == 1u) {
                    hb = dh;
                    cx = dx;
                    ci = dc;
                    layout = 1;
                    P = plan.P;
                    R = plan.R;
                    n_scat = n_in;
                    win_end = gi + (lv < 0 ? 1 : (lv ? gates[k].len[1] : gates[k].len[0]));
                    break;
                }
                if (lv < 0) want = plan.P / 2u;
                for (uint32_t i = team.rank * kBlock + threadIdx.x; i < a.part_max;
                     i += team.size * kBlock)
                    arr.cnt(dc)[(uint64_t)i * kPad] = 0u;
                if (!team_barrier(team, ctl)) return false;
            }
        }
        // ---- merge, in place --------------------------------------------
        const unsigned long long dbits = a.delta_bits;
        const unsigned long long thr = s_pub.thr;
        const bool drop = thr > dbits;
        const uint32_t p_id = identity_part<W>(P);
        PushList push_to = pl;
        push_to.gn = &acc->cand_n;
        auto push = [&](bool hit, unsigned long long v, uint64_t idx) {
            push_cand(push_to, hit, v, idx);
        };
        InStats st{0u, 0u};
        uint32_t n_long = 0;
        // the third cursor array (two gates back) is the next scatter's
        for (uint32_t i = team.rank * kBlock + threadIdx.x; i < a.part_max; i += team.size * kBlock)
            arr.cnt(next3(next3(ci)))[(uint64_t)i * kPad] = 0u;
        InRows<W, kBlock> rows;
        auto stored = [&](uint32_t p) -> uint32_t {
            const uint32_t c = p < P ? __ldcg(arr.cnt(ci) + (uint64_t)p * kPad) : 0u;
            return c < R ? c : (uint32_t)R;
        };
        auto load = [&](uint32_t p, uint32_t n) {   // (a longer one is gathered later)
            if (n && n <= C)
                load_rows<W, kBlock, false>(rows, arr.home(hb) + (uint64_t)p * R,
                                            arr.coef(cx) + (uint64_t)p * R, n);
        };
        uint32_t np = stored(team.rank);
        for (uint32_t p = team.rank; p < P; p += team.size) {
            load(p, np);
            InPlace<W> io;
            io.first = (uint64_t)p * R;
            io.keys = arr.home(hb) + io.first;
            io.cin = arr.coef(cx) + io.first;
            io.cout = arr.coef(cx ^ 1) + io.first;
            io.n = np;
            io.room = (uint32_t)(R < 0xffffffffULL ? R : 0xffffffffULL);
            io.s_app = &s_app;
            io.s_rare = &s_rare;
            io.over = &s_over;
            const uint32_t pn = p + team.size;
            np = stored(pn);
            if (inplace_partition<W, kBlock, 12>(g, s_pub.T, s_pub.all_ties != 0, tk, s_pub.rnorm, thr,
                                             p == p_id, ctl, np_, &tag, io, st, s_pub.hi, &s_n, rows,
                                             push, [] {}))
                ++n_long;
            if (threadIdx.x == 0) {
                // (the others use these again only after the next pass's barrier)
                const uint64_t c = (uint64_t)io.n + s_app;
                arr.cnt(next3(ci))[(uint64_t)p * kPad] = (unsigned int)(c < R ? c : R);
                s_app = s_rare = 0u;
            }
            if (tag >= kHeadTagMax - 65536u) {   // tags start again
                inplace_init<W, kBlock, 12>();
                tag = 0;
                __syncthreads();
            }
        }
        // the CTA's counts and candidates
        auto flush = [&](Acc* to, const InStats& s) {
            const uint32_t hm = __reduce_max_sync(0xffffffffu, s.hi_max);
            const uint32_t kw = __reduce_add_sync(0xffffffffu, s.kept);
            if ((threadIdx.x & 31) == 0) {
                s_red[threadIdx.x >> 5] = hm;
                s_kept[threadIdx.x >> 5] = kw;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                uint32_t mx = 0, kept = 0;
                for (int w = 0; w < kBlock / 32; ++w) {
                    mx = max(mx, s_red[w]);
                    kept += s_kept[w];
                }
                if (mx) atomicMax(&to->out_max, ((unsigned long long)mx << 32) | 0xffffffffULL);
                if (kept) atomicAdd(&to->kept, (unsigned long long)kept);
                if (s_over) atomicExch(&to->over, 1u);
                if (n_long) atomicAdd(&to->n_long, n_long);
                s_n = s_cs ? atomicAdd(&to->cand_n, s_cs) : 0u;
            }
            __syncthreads();
            const uint32_t b = s_n, m = s_cs;
            for (uint32_t j = threadIdx.x; j < m; j += kBlock)
                if ((uint64_t)b + j < a.cand_cap) {
                    cand_v[b + j] = s_cv[j];
                    cand_i[b + j] = s_ci[j];
                }
        };
        // how this gate's and the next gate's thresholds moved in the last layer
        long long* drift_now = n_drift > 0 ? drift + (a.gate0 + k) % n_drift : nullptr;
        const long long* drift_next = n_drift > 0 ? drift + (a.gate0 + k + 1) % n_drift : nullptr;
        // the first CTA, once every CTA has arrived (s_acc read): statistics,
        // normaliser, bound, threshold; published for all
        auto lead_gate = [&](bool redone) {
            const unsigned long long kept = redone ? s_acc.alloc : s_acc.kept;
            const bool active = a.cap_policy == 1 && kept > a.cap_M;
            const unsigned long long lo = s_pub.lo, hi = s_pub.hi;
            const uint32_t cn = redone ? 0u : s_acc.cand_n;
            // kept children above the range: all that were not listed
            const unsigned long long above = kept - cn, omax = s_acc.out_max;
            // why not the listed candidates: 1 no range, 2 list too long,
            // 3 threshold above the range, 4 below it
            const int reason = hi == 0ULL ? 1 : redone ? 4 : cn > a.cand_cap ? 2
                               : above >= a.cap_M ? 3 : above + cn < a.cap_M ? 4 : 0;
            const int failed = s_status;
            SelOut so{0ULL, 1};
            PKey<W> key{};
            const bool listed = active && reason == 0 && !failed;
            // a long list is first cut down by the whole team
            const bool fast = listed && (cn <= kOneCta || cn > a.cand_cap / 4);
            if (fast)
                so = select_list<W>(g_stage + InPass<W>::kBytes, cand_v, cand_i, cn, a.cap_M - above, 0ULL, 0ULL,
                                    hi > lo ? 64 - __clzll((long long)(hi - lo)) : 0,
                                    arr.home(hb), ties, &key, ctl);
            if (threadIdx.x == 0) {
                constexpr unsigned long long kInfBits = 0x7ff0000000000000ULL;
                if (omax >= kInfBits) set_status(ctl, ST_STATE, 4);
                if (abs_pattern(s_norm) >= kInfBits) set_status(ctl, ST_STATE, 5);
                if (a.cap_policy == 0 && kept > a.cap_M) set_status(ctl, ST_CAPACITY, 1);
                Pub& p = s_next;
                p.rnorm = s_rnorm;
                p.n = active ? a.cap_M : kept;
                p.T = fast ? so.v + lo : 0ULL;
                p.all_ties = fast ? so.all_ties : 1;
#pragma unroll
                for (int w = 0; w < 4; ++w) p.tk[w] = 0;
                if (fast && !so.all_ties) {
#pragma unroll
                    for (int w = 0; w < W; ++w) { p.tk[w] = key.x[w]; p.tk[W + w] = key.z[w]; }
                }
                // 1: radix passes over the state, 2: over the candidates
                p.full = !active || fast || failed ? 0 : listed ? 2 : 1;
                p.base = listed ? lo : a.delta_bits;
                p.range = listed ? hi - lo : omax > a.delta_bits ? omax - a.delta_bits : 0ULL;
                p.rank = listed ? a.cap_M - above : a.cap_M;
                p.redo = 0;
                p.pad = 0;
                p.lo = lo;
                p.hi = hi;
                p.thr = s_pub.thr;
                if (redone && !active) {
                    // the state has fallen below its bound: with the old limit
                    // every gate from here on would be merged twice
                    p.lo = p.hi = 0ULL;
                    p.thr = a.delta_bits;
                    s_pred.tprev = 0ULL;
                }
                // a state that doubled since its scatter: more partitions, before
                // they outgrow the staging
                p.rescatter = !redone && p.n > 2ULL * n_scat && p.n > (C / 2) * (uint64_t)P;
                p.stop = failed || omax >= kInfBits || abs_pattern(s_norm) >= kInfBits ||
                         (a.cap_policy == 0 && kept > a.cap_M) ||
                         (fast && *(volatile int*)&ctl->status != 0);
                if (a.log) a.log[gi] = p.stop ? ~0ULL : p.n;
                s_stat[0] += 1;
                s_stat[1] += n_in;
                s_stat[2] += p.n;
                if (p.n > s_stat[3]) s_stat[3] = p.n;
                s_stat[5] += active ? 1 : 0;
                s_stat[6] += redone ? 1 : 0;
                s_stat[7] += s_long;
                if (active) {
                    s_pred.reason = reason;
                    s_pred.range = hi - lo;
                }
                if (fast)
                    next_range(&s_pred, a.cand_hi, drift_now, s_dn, p.T, p.rnorm, cn, a.delta_bits, &p);
                s_pred.full += p.full == 1 ? 1 : 0;
                if (p.full) rs->sel_n = 0u;
            }
            if (threadIdx.x < 32) publish(team, &s_next);
        };
        // the counters of a finished merge, one load per lane
        auto read_acc = [&](const Acc* from, Acc* to) {
            constexpr int N = sizeof(Acc) / 8;
            if (threadIdx.x < N)
                reinterpret_cast<unsigned long long*>(to)[threadIdx.x] =
                    __ldcg(reinterpret_cast<const unsigned long long*>(from) + threadIdx.x);
            else if (threadIdx.x == 32) {
                s_norm = *(volatile double*)&ctl->norm[np_];
                s_rnorm = __ddiv_rn(1.0, s_norm);
            } else if (threadIdx.x == 64)
                s_dn = drift_next ? *drift_next : 0LL;
            else if (threadIdx.x == 33)
                s_status = *(volatile int*)&ctl->status;
            else if (threadIdx.x == 34)
                s_long = *(volatile unsigned int*)&rs->acc[np_][0].n_long;
            else if (threadIdx.x >= 96 && threadIdx.x < 96 + 2 * N)
                // the next gate's counters (every CTA is done with them)
                reinterpret_cast<unsigned long long*>(&rs->acc[np_ ^ 1][0])[threadIdx.x - 96] = 0ULL;
            __syncthreads();
        };
        flush(acc, st);
        team_arrive(team);
        if (leader) {
            if (!team_wait(team, ctl)) return false;
            read_acc(acc, &s_acc);
            // children left out that the bound may need, or a stride that had
            // no room: the merge is done again
            if (s_acc.over != 0u || (drop && s_acc.kept < a.cap_M)) {
                if (threadIdx.x == 0) {
                    s_next = s_pub;
                    s_next.redo = 1;
                }
                if (threadIdx.x < 32) publish(team, &s_next);
            } else {
                lead_gate(false);
            }
        }
        if (!take_pub(team, ctl, &s_pub)) return false;
        const bool redo = s_pub.redo != 0;
        if (redo) {
            // again in full from the same input, into a contiguous run
            acc = &rs->acc[np_][1];
            for (uint32_t i = team.rank * kBlock + threadIdx.x; i < a.part_max;
                 i += team.size * kBlock)
                arr.cnt(next3(ci))[(uint64_t)i * kPad] = 0u;   // the first try's counts
            push_to.gn = &acc->cand_n;
            if (threadIdx.x == 0) {
                s_cn = s_cs = 0u;
                s_over = 0;
                g_cn = 0u;
                g_range[0] = s_pub.lo;
                g_range[1] = 0ULL;   // no candidates: the select passes over the state
            }
            pass_init<W, kBlock>();
            __syncthreads();
            PKey<W>* kout = arr.run_keys(arr.a);
            double* cout = arr.run_coef(arr.a);
            Pending<W> pd;
            pd.on = s_pub.T != 0ULL;
            pd.all_ties = s_pub.all_ties != 0;
            pd.T = s_pub.T;
            pd.tk = tk;
            auto room = [&](uint32_t n_out) -> unsigned long long {
                if (threadIdx.x == 0) {
                    unsigned long long at = n_out ? atomicAdd(&acc->alloc, (unsigned long long)n_out)
                                                  : 0ULL;
                    if (at + n_out > a.buf_cap) {
                        set_status(ctl, ST_CAPACITY, 62);
                        at = ~0ULL;
                    }
                    s_at = at;
                }
                __syncthreads();
                return s_at;
            };
            SelStats ss{0ULL};
            for (uint32_t p = team.rank; p < P; p += team.size) {
                uint64_t np = __ldcg(arr.cnt(ci) + (uint64_t)p * kPad);
                if (np > R) np = R;
                const PKey<W>* kp = arr.home(hb) + (uint64_t)p * R;
                const double* cp = arr.coef(cx) + (uint64_t)p * R;
                if (np <= (uint64_t)Stage<W>::C) {
                    ++pass;   // (merge_long numbers its own: consecutive passes alternate)
                    for (uint32_t i = threadIdx.x; i < np; i += kBlock) {
                        PassArgs<W>::keys()[i] = load_key_stream(kp + i);
                        PassArgs<W>::vals()[i] = __ldcs(cp + i);
                    }
                    __syncthreads();
                    stage_pass<W, kBlock, PassRoom::kExact>((uint32_t)np, g, pd, s_pub.rnorm,
                                                            dbits, p == p_id, ctl, np_, pass, kout,
                                                            cout, ss, room);
                } else {
                    merge_long<W, kBlock>(kp, cp, np, g, pd, s_pub.rnorm, dbits, p == p_id, ctl,
                                          np_, &pass, kout, cout, ss, room, &s_n);
                }
            }
            n_long = 0;
            const InStats s2{(uint32_t)(__reduce_max_sync(0xffffffffu, (uint32_t)(ss.out_max >> 32))), 0u};
            flush(acc, s2);
            inplace_init<W, kBlock, 12>();
            tag = 0;
            team_arrive(team);
            layout = 0;
            run_buf = arr.a;
            if (leader) {
                if (!team_wait(team, ctl)) return false;
                read_acc(acc, &s_acc);
                lead_gate(true);
            }
            if (!take_pub(team, ctl, &s_pub)) return false;
            run_n = __ldcg(&acc->alloc);
        } else {
            cx ^= 1;
            ci = next3(ci);
        }
        // ---- a threshold outside the listed range, or a long list: radix
        // passes by the whole team, every CTA picking the digit for itself ----
        if (s_pub.full && !s_pub.stop) {
            const bool of_list = s_pub.full == 2;
            const unsigned long long base = s_pub.base;
            const uint32_t cn = of_list ? __ldcg(&acc->cand_n) : 0u;
            // every value: f(in, pattern - base, place), whole warps
            auto each = [&](auto&& f) {
                const uint32_t lane = threadIdx.x & 31u;
                if (of_list || layout == 0) {
                    const double* c = arr.run_coef(run_buf);
                    const uint64_t n = of_list ? cn : run_n;
                    for (uint64_t i = (uint64_t)team.rank * kBlock + (threadIdx.x & ~31u); i < n;
                         i += (uint64_t)team.size * kBlock) {
                        const uint64_t j = i + lane;
                        if (of_list) {
                            f(j < n, j < n ? __ldcg(cand_v + j) : 0ULL,
                              j < n ? (uint64_t)__ldcg(cand_i + j) : 0ULL);
                        } else {
                            const unsigned long long b = j < n ? abs_pattern(__ldcs(c + j)) : 0ULL;
                            f(b > base, b - base, j);
                        }
                    }
                } else {
                    for (uint32_t p = team.rank; p < P; p += team.size) {
                        const uint32_t n = __ldcg(arr.cnt(ci) + (uint64_t)p * kPad);
                        const double* c = arr.coef(cx) + (uint64_t)p * R;
                        for (uint32_t i = threadIdx.x & ~31u; i < n; i += kBlock) {
                            const uint32_t j = i + lane;
                            const unsigned long long b = j < n ? abs_pattern(__ldcs(c + j)) : 0ULL;
                            f(b > base, b - base, (uint64_t)p * R + j);
                        }
                    }
                }
            };
            uint32_t* h = reinterpret_cast<uint32_t*>(g_stage + InPass<W>::kBytes);
            unsigned long long prefix = 0ULL, mask = 0ULL;
            uint32_t rank = (uint32_t)s_pub.rank, count = 0xffffffffu;
            int top = s_pub.range ? 64 - __clzll((long long)s_pub.range) : 0;
            for (int q = 0; top > 0 && count > kOneCta; ++q) {
                const int shift = top > kDigit ? top - kDigit : 0;
                const uint32_t dmask = (1u << (top - shift)) - 1u;
                uint32_t* hist = rs->hist[q % 3];
                uint32_t* spare = rs->hist[(q + 1) % 3];
                for (int b = threadIdx.x; b < kBins; b += kBlock) h[b] = 0u;
                for (uint32_t b = team.rank * kBlock + threadIdx.x; b < (uint32_t)kBins;
                     b += team.size * kBlock)
                    spare[b] = 0u;
                __syncthreads();
                each([&](bool in, unsigned long long v, uint64_t) {
                    if (in && (v & mask) == prefix)
                        atomicAdd(&h[(uint32_t)(v >> shift) & dmask], 1u);
                });
                __syncthreads();
                for (int b = threadIdx.x; b < kBins; b += kBlock)
                    if (h[b]) atomicAdd(hist + b, h[b]);
                if (!team_barrier(team, ctl)) return false;
                for (int b = threadIdx.x; b < kBins; b += kBlock) h[b] = __ldcg(hist + b);
                __syncthreads();
                pick_bin<true>(h, rank, s_w, &s_pick);
                prefix |= (unsigned long long)s_pick.digit << shift;
                mask |= (unsigned long long)dmask << shift;
                rank = s_pick.k_in;
                count = s_pick.count;
                top = shift;
                __syncthreads();
            }
            // the values left, for the first CTA (those of the list beside it)
            PushList gp = pl;
            unsigned long long* lv = of_list ? reinterpret_cast<unsigned long long*>(ties) : cand_v;
            uint32_t* li = of_list ? reinterpret_cast<uint32_t*>(lv + cn) : cand_i;
            gp.gv = lv;
            gp.gidx = li;
            gp.gn = &rs->sel_n;
            if (threadIdx.x == 0) s_cn = kPushBuf;   // straight to the global list
            __syncthreads();
            each([&](bool in, unsigned long long v, uint64_t idx) {
                push_cand(gp, in && (v & mask) == prefix, v, idx);
            });
            team_arrive(team);
            if (leader) {
                if (!team_wait(team, ctl)) return false;
                for (int b = threadIdx.x; b < 3 * kBins; b += kBlock) rs->hist[0][b] = 0u;
                PKey<W> key{};
                const uint32_t ln = __ldcg(&rs->sel_n);
                SelOut so{0ULL, 1};
                if (ln > a.cand_cap) {
                    if (threadIdx.x == 0) set_status(ctl, ST_CAPACITY, 63);
                } else {
                    PKey<W>* tl = of_list ? reinterpret_cast<PKey<W>*>(cand_v) : ties;
                    so = select_list<W>(g_stage + InPass<W>::kBytes, lv, li, ln, rank, prefix, mask, top,
                                        layout == 0 ? arr.run_keys(run_buf) : arr.home(hb), tl,
                                        &key, ctl);
                }
                if (threadIdx.x == 0) {
                    Pub& p = s_next;
                    p = s_pub;
                    p.T = so.v + base;
                    p.all_ties = so.all_ties;
                    if (!so.all_ties)
                        for (int w = 0; w < W; ++w) { p.tk[w] = key.x[w]; p.tk[W + w] = key.z[w]; }
                    p.full = 0;
                    p.stop = *(volatile int*)&ctl->status != 0;
                    next_range(&s_pred, a.cand_hi, drift_now, s_dn, p.T, p.rnorm, of_list ? cn : ln,
                               a.delta_bits, &p);
                }
                if (threadIdx.x < 32) publish(team, &s_next);
            }
            if (!take_pub(team, ctl, &s_pub)) return false;
        }
        any = true;
    }
    // ---- a contiguous run with the select applied -----------------------
    const bool ran = any;
    int out_buf = run_buf;
    bool copied = false;
    if (ran && !s_pub.stop && (layout == 1 || s_pub.T)) {
        copied = true;
        out_buf = layout == 1 ? arr.a : arr.a ^ 1;
        PKey<W> tk;
#pragma unroll
        for (int w = 0; w < W; ++w) { tk.x[w] = s_pub.tk[w]; tk.z[w] = s_pub.tk[W + w]; }
        PKey<W>* ko = arr.run_keys(out_buf);
        double* co = arr.run_coef(out_buf);
        unsigned long long* alloc = &rs->acc[total & 1][0].alloc;
        const uint32_t runs = layout == 1 ? P : 1u;
        for (uint32_t p = layout == 1 ? team.rank : 0u; p < runs; p += layout == 1 ? team.size : 1u) {
            const PKey<W>* ki = layout == 1 ? arr.home(hb) + (uint64_t)p * R : arr.run_keys(run_buf);
            const double* vi = layout == 1 ? arr.coef(cx) + (uint64_t)p * R : arr.run_coef(run_buf);
            const uint64_t n = layout == 1 ? __ldcg(arr.cnt(ci) + (uint64_t)p * kPad) : run_n;
            const uint64_t first = layout == 1 ? 0ULL : (uint64_t)team.rank * kBlock;
            const uint64_t step = layout == 1 ? (uint64_t)kBlock : (uint64_t)team.size * kBlock;
            for (uint64_t i0 = first; i0 < n; i0 += step) {
                const uint64_t i = i0 + threadIdx.x;
                PKey<W> K{};
                double c = 0.0;
                bool keep = false;
                if (i < n) {
                    K = load_key_stream(ki + i);
                    c = __ldcs(vi + i);
                    keep = abs_pattern(c) != 0ULL &&
                           cap_keep(K, c, s_pub.T, s_pub.all_ties != 0, tk);
                    if (!keep && key_is_zero(K)) set_status(ctl, ST_TRACE_ZERO, 3);
                }
                const uint32_t incl = block_scan_incl(keep ? 1u : 0u, s_w);
                if (threadIdx.x == kBlock - 1) s_at = incl ? atomicAdd(alloc, (unsigned long long)incl) : 0ULL;
                __syncthreads();
                if (keep) {
                    store_key_stream(ko + s_at + incl - 1u, K);
                    __stcs(co + s_at + incl - 1u, c);
                }
                __syncthreads();
            }
        }
    }
    if (!team_barrier(team, ctl)) return false;
    if (leader && threadIdx.x == 0 && ran) {
        const double norm = ctl->norm[(s_stat[0] & 1ULL) ? 0 : 1];
        ctl->cur = out_buf;
        ctl->count[out_buf] = copied ? rs->acc[total & 1][0].alloc : s_pub.n;
        ctl->count[out_buf ^ 1] = 0ULL;
        ctl->norm[out_buf] = norm;
        ctl->rnorm[out_buf] = s_pub.rnorm;
        ctl->pend = 0;
        ctl->home = 0;
        ctl->need_scatter = 0;
        ctl->part_over = 0;
        ctl->sel_active = 0;
        ctl->sp_lo = s_pub.lo;
        ctl->sp_hi = s_pub.hi;
        ctl->sp_thr = s_pub.thr;
        ctl->sp_tprev = s_pred.tprev;
        ctl->sp_shift = s_pred.shift;
        ctl->stat_cands += s_pred.cands;
        if (s_pred.range) ctl->stat_range = s_pred.range;
        ctl->stat_sel_full += s_pred.full;
        ctl->out_max = 0;
        const unsigned int gen = ctl->gen + (unsigned int)s_stat[0];
        if (gen < ctl->gen) set_status(ctl, ST_STATE, 1);   // generation counter wrapped
        ctl->gen = gen;
        ctl->stat_gates += s_stat[0];
        ctl->stat_in += s_stat[1];
        ctl->stat_out += s_stat[2];
        if (s_stat[3] > ctl->stat_peak) ctl->stat_peak = s_stat[3];
        ctl->stat_scatters += s_stat[4];
        ctl->stat_cap += s_stat[5];
        ctl->stat_retry += s_stat[6];
        ctl->stat_long += s_stat[7];
    }
    __syncthreads();
    return true;
}

template <int W, bool kWide>
__global__ void __launch_bounds__(kBlock, (W == 1 ? 3 : 2) + (kWide ? 1 : 0))
k_run(const RunArgs<W> a, const __grid_constant__ RunChunk<W> chunk) {
    Team team;
    uint32_t t = 0, teams = 1;
    if (a.team_of) {   // a batch: this CTA's team, its rank and the team's size
        const uint4 v = a.team_of[blockIdx.x];
        t = v.x;
        team.rank = v.y;
        team.size = v.z;
        teams = v.w;
    } else {
        team.rank = blockIdx.x;
        team.size = gridDim.x;
    }
    team.rs = reinterpret_cast<RunShared*>(static_cast<char*>(a.shared) + (uint64_t)t * a.shared_stride);
    team.target = 0;
    team.seq = 0;
    for (int inst = (int)t; inst < a.B; inst += (int)teams) {
        const RunGate<W>* gates = a.gates ? a.gates + (uint64_t)inst * a.max_gates : chunk.g;
        const int n = a.gates ? a.n_gates[inst] : a.one_gates;
        if (n > 0 && !run_instance<W>(a, gates, n, inst, team)) return;
    }
}

}  // namespace

template <int W>
static constexpr size_t run_smem() {
    return InPass<W>::kBytes + kScratch > Stage<W>::kBytes ? InPass<W>::kBytes + kScratch
                                                           : Stage<W>::kBytes;
}

template <int W, bool kWide>
int run_fit_as() {
    constexpr size_t smem = run_smem<W>();
    cudaFuncSetAttribute(k_run<W, kWide>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_run<W, kWide>, cudaFuncAttributePreferredSharedMemoryCarveout,
                         (int)cudaSharedmemCarveoutMaxShared);
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_run<W, kWide>, kBlock, smem);
    return n > 0 ? n : 1;
}

template <int W, bool kWide>
cudaError_t launch_run_as(const RunArgs<W>& a, const RunChunk<W>& chunk, int grid, cudaStream_t st) {
    void* args[2] = {const_cast<RunArgs<W>*>(&a), const_cast<RunChunk<W>*>(&chunk)};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_run<W, kWide>), dim3(grid),
                                       dim3(kBlock), args, run_smem<W>(), st);
}

}  // namespace itpp
