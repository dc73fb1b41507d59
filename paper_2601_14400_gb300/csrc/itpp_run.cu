// itpp_run.cu -- a run of gates in one launch.
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
//   select    the team's first CTA: statistics, the next normaliser, the
//             top-M threshold from the candidates the merge listed, published
//             for the next gate; the others clear cursors meanwhile
//
// that is two barriers per gate inside a window.  The rest is rare and decided
// on the device: a threshold outside the listed range takes radix passes over
// the state by the whole team; a merge that left children out which the bound
// then needed, or that ran out of a partition's stride, is done again from its
// unchanged input into a contiguous run.  Between launches the state is that
// contiguous run with the select applied, as every other entry point reads it.
//
// Every wait is bounded; a team that gives up stores the error and leaves.
#include <cstring>

#include "itpp_common.cuh"
#include "itpp_gate_body.cuh"
#include "itpp_launch.h"
#include "itpp_run.cuh"
#include "itpp_stage.cuh"
#include "itpp_inplace.cuh"

namespace itpp {

namespace {

constexpr int kBlock = 256;
constexpr int kDigit = 11, kBins = 1 << kDigit;   // radix digit of the select
constexpr uint32_t kFinal = 256;                  // strings ranked one per thread
constexpr uint32_t kPushBuf = 512;                // candidates a CTA lists in shared memory
constexpr int kRangeShift = 45;                   // first candidate range: T +- about 1/128 of T

// What the first CTA of a team publishes after a gate.
struct Pub {
    unsigned long long T;        // pending select: kept at or above this pattern (0: none)
    uint64_t tk[4];              // ... and at it up to this key
    unsigned long long lo, hi;   // candidate range of the next gate (hi == 0: none)
    unsigned long long n;        // logical terms
    double rnorm;
    int all_ties, stop, full, rescatter;
};

// Written by every CTA during a gate; one set per gate parity, one for the
// merge that is done again.
struct Acc {
    unsigned long long kept, above, out_max, alloc;
    unsigned int cand_n, over, n_long, scatter_over;
};

}  // namespace

struct RunShared {
    unsigned int bar;            // arrivals at the team's barrier so far
    unsigned int dead;           // a wait ran out
    Pub pub;
    Acc acc[2][2];
    unsigned int sel_n;          // full select: candidates gathered
    unsigned int pad;
    unsigned long long sel_prefix, sel_mask, sel_k, sel_count;
    unsigned int hist[kBins];
};

size_t run_shared_bytes() { return (sizeof(RunShared) + 255) / 256 * 256; }
size_t run_shared_head() { return offsetof(RunShared, pub); }

namespace {

// ---------------------------------------------------------------------------
// Team barrier
// ---------------------------------------------------------------------------
struct Team {
    RunShared* rs;
    uint32_t rank, size;
    uint32_t target;   // arrivals that complete the next barrier
};

// False: the wait ran out (about ten seconds) here or elsewhere in the team;
// the caller leaves the kernel.  Every thread calls it.
__device__ __forceinline__ bool team_barrier(Team& t, DevCtl* ctl) {
    __shared__ int s_ok;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        t.target += t.size;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(&t.rs->bar) : "memory");
        uint32_t it = 0;
        for (;;) {
            uint32_t v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&t.rs->bar) : "memory");
            if ((int32_t)(v - t.target) >= 0) break;
            if (++it > 64u) {
                __nanosleep(it > 4096u ? 1000u : 32u);
                if (it > 10000000u || *(volatile unsigned int*)&t.rs->dead) {
                    set_status(ctl, ST_TIMEOUT, 60);
                    *(volatile unsigned int*)&t.rs->dead = 1u;
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    const int ok = s_ok;
    __syncthreads();
    return ok != 0;
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
// Select among a list of n (v, idx): the k-th largest v (rank from 1), ties
// by ascending key.  One CTA; scratch in the staging memory.
// ---------------------------------------------------------------------------
struct SelOut {
    unsigned long long v;   // threshold value
    int all_ties;
};

__device__ __forceinline__ uint32_t block_scan_incl(uint32_t v, uint32_t* s_w) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    uint32_t before = 0;
    for (int w = 0; w < warp; ++w) before += s_w[w];
    __syncthreads();
    return before + x;
}

struct PickOut {
    uint32_t digit, k_in, count;
};

// The digit holding rank k (from 1) of a histogram of kBins counts, largest
// digit first (kDesc) or smallest first.  Every thread calls it.
template <bool kDesc>
__device__ __forceinline__ void pick_bin(const uint32_t* h, uint32_t k, uint32_t* s_w,
                                         PickOut* out) {
    constexpr int PER = kBins / kBlock;
    uint32_t c[PER], sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int b = (int)threadIdx.x * PER + j;
        c[j] = h[kDesc ? kBins - 1 - b : b];
        sum += c[j];
    }
    const uint32_t incl = block_scan_incl(sum, s_w);
    uint32_t run = incl - sum;
    if (run < k && k <= incl) {
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            if (run < k && k <= run + c[j]) {
                const int b = (int)threadIdx.x * PER + j;
                out->digit = (uint32_t)(kDesc ? kBins - 1 - b : b);
                out->k_in = k - run;
                out->count = c[j];
            }
            run += c[j];
        }
    }
    __syncthreads();
}

// Bits [off, off + kDigit) of a key, words in comparison order, off counted
// from the top of word 0; a digit may end early at a word's end (width out).
template <int W>
__device__ __forceinline__ uint32_t key_digit(const PKey<W>& k, int off, int* width) {
    const int w = off >> 6, in = off & 63;
    const int wd = 64 - in < kDigit ? 64 - in : kDigit;
    *width = wd;
    uint64_t word = 0;
#pragma unroll
    for (int j = 0; j < 2 * W; ++j) if (j == w) word = j < W ? k.x[j] : k.z[j - W];
    return (uint32_t)((word >> (64 - in - wd)) & ((1ULL << wd) - 1ULL));
}

// prefix, top: the bits of v from `top` up already agree with prefix.  Every
// thread calls it; *tk receives the largest kept key at the threshold.
// ties/tie_cap: global scratch for a long list of equal values.
template <int W>
__device__ SelOut select_list(const unsigned long long* gv, const uint32_t* gidx, uint64_t n,
                              uint64_t k, unsigned long long prefix, unsigned long long mask,
                              int top, const PKey<W>* keys, PKey<W>* ties, PKey<W>* tk,
                              DevCtl* ctl) {
    // scratch, behind one another in the staging memory
    uint32_t* h = reinterpret_cast<uint32_t*>(g_stage);                     // kBins
    unsigned long long* fv = reinterpret_cast<unsigned long long*>(h + kBins);
    PKey<W>* fk = reinterpret_cast<PKey<W>*>(fv + kFinal);
    __shared__ uint32_t s_w[kBlock / 32], s_n, s_gt, s_eq;
    __shared__ PickOut s_pick;
    __shared__ SelOut s_out;
    __shared__ uint64_t s_tk[4];
    const uint32_t lane = threadIdx.x & 31u;
    uint64_t cnt = n;          // entries that match the prefix
    uint32_t rank = (uint32_t)k;
    while (cnt > kFinal && top > 0) {
        const int shift = top > kDigit ? top - kDigit : 0;
        for (int b = threadIdx.x; b < kBins; b += kBlock) h[b] = 0u;
        __syncthreads();
        const uint32_t dmask = (1u << (top - shift)) - 1u;
        for (uint64_t j = threadIdx.x; j < n; j += kBlock) {
            const unsigned long long v = __ldcg(gv + j);
            if ((v & mask) == prefix) atomicAdd(&h[(uint32_t)(v >> shift) & dmask], 1u);
        }
        __syncthreads();
        pick_bin<true>(h, rank, s_w, &s_pick);
        prefix |= (unsigned long long)s_pick.digit << shift;
        mask |= (unsigned long long)dmask << shift;
        rank = s_pick.k_in;
        cnt = s_pick.count;
        top = shift;
        __syncthreads();
    }
    // a long list of exact ties: by key digits, from a list of their keys
    bool by_key = false;
    int off = 0;
    uint64_t kpre[2 * W];   // key bits fixed so far
#pragma unroll
    for (int w = 0; w < 2 * W; ++w) kpre[w] = 0;
    uint64_t n_tie = 0;
    if (cnt > kFinal) {
        if (rank == cnt) {   // every one of them is kept
            SelOut o;
            o.v = prefix;
            o.all_ties = 1;
            return o;
        }
        by_key = true;
        n_tie = cnt;
        if (threadIdx.x == 0) s_n = 0u;
        __syncthreads();
        for (uint64_t j0 = threadIdx.x & ~31u; j0 < n; j0 += kBlock) {
            const uint64_t j = j0 + lane;
            const bool hit = j < n && (__ldcg(gv + j) & mask) == prefix;
            const unsigned int m = __ballot_sync(0xffffffffu, hit);
            if (!m) continue;
            uint32_t q = 0;
            if (lane == 0) q = atomicAdd(&s_n, (uint32_t)__popc(m));
            q = __shfl_sync(0xffffffffu, q, 0) + __popc(m & ((1u << lane) - 1u));
            if (hit) ties[q] = load_key_stream(keys + __ldcg(gidx + j));
        }
        __syncthreads();
        auto matches = [&](const PKey<W>& key) {
            const int full = off >> 6, r = off & 63;
            bool ok = true;
#pragma unroll
            for (int w = 0; w < 2 * W; ++w) {
                const uint64_t word = w < W ? key.x[w] : key.z[w - W];
                if (w < full) ok = ok && word == kpre[w];
                else if (w == full && r) ok = ok && (word >> (64 - r)) == (kpre[w] >> (64 - r));
            }
            return ok;
        };
        while (cnt > kFinal && off < 128 * W) {
            for (int b = threadIdx.x; b < kBins; b += kBlock) h[b] = 0u;
            __syncthreads();
            int wd = kDigit;
            for (uint64_t j = threadIdx.x; j < n_tie; j += kBlock) {
                const PKey<W> key = load_key_stream(ties + j);
                const uint32_t d = key_digit(key, off, &wd);
                if (matches(key)) atomicAdd(&h[d], 1u);
            }
            {   // the digit's width, also for threads that saw no key
                const PKey<W> z{};
                key_digit(z, off, &wd);
            }
            __syncthreads();
            pick_bin<false>(h, rank, s_w, &s_pick);
            const int w = off >> 6, in = off & 63;
#pragma unroll
            for (int v = 0; v < 2 * W; ++v)
                if (v == w) kpre[v] |= (uint64_t)s_pick.digit << (64 - in - wd);
            rank = s_pick.k_in;
            cnt = s_pick.count;
            off += wd;
            __syncthreads();
        }
        // the strings that remain (distinct keys: at most kFinal)
        if (threadIdx.x == 0) s_n = 0u;
        __syncthreads();
        for (uint64_t j = threadIdx.x; j < n_tie; j += kBlock) {
            const PKey<W> key = load_key_stream(ties + j);
            if (matches(key)) {
                const uint32_t q = atomicAdd(&s_n, 1u);
                if (q < kFinal) {
                    fk[q] = key;
                    fv[q] = prefix;
                }
            }
        }
    } else {
        if (threadIdx.x == 0) s_n = 0u;
        __syncthreads();
        for (uint64_t j = threadIdx.x; j < n; j += kBlock) {
            const unsigned long long v = __ldcg(gv + j);
            if ((v & mask) == prefix) {
                const uint32_t q = atomicAdd(&s_n, 1u);
                if (q < kFinal) {
                    fv[q] = v;
                    fk[q] = load_key_stream(keys + __ldcg(gidx + j));
                }
            }
        }
    }
    if (threadIdx.x == 0) s_gt = s_eq = 0u;
    __syncthreads();
    const uint32_t m = s_n;
    if (m > kFinal || rank < 1u || rank > m) {   // uniform; the lists always agree with the counts
        if (threadIdx.x == 0) set_status(ctl, ST_STATE, 61);
        __syncthreads();
        SelOut o;
        o.v = prefix;
        o.all_ties = 1;
        return o;
    }
    // one string per thread: how many come before it
    bool mine = false;
    unsigned long long v = 0;
    if (threadIdx.x < m) {
        v = fv[threadIdx.x];
        const PKey<W> key = fk[threadIdx.x];
        uint32_t before = 0;
        for (uint32_t j = 0; j < m; ++j) {
            const unsigned long long u = fv[j];
            if (u > v) ++before;
            else if (u == v && key_less(fk[j], key)) ++before;
        }
        mine = before == rank - 1u;
        if (mine) {
            s_out.v = v;
            for (int w = 0; w < W; ++w) {
                s_tk[w] = key.x[w];
                s_tk[W + w] = key.z[w];
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < m) {
        if (v > s_out.v) atomicAdd(&s_gt, 1u);
        if (v == s_out.v) atomicAdd(&s_eq, 1u);
    }
    __syncthreads();
    SelOut o;
    o.v = s_out.v;
    // by_key: the strings outside the final set also tie, and some are dropped
    o.all_ties = !by_key && rank - s_gt == s_eq;
#pragma unroll
    for (int w = 0; w < W; ++w) { tk->x[w] = s_tk[w]; tk->z[w] = s_tk[W + w]; }
    __syncthreads();
    return o;
}

// ---------------------------------------------------------------------------
// The run
// ---------------------------------------------------------------------------
// The candidate range around the threshold predicted for the next gate: C +-
// 2^s in pattern units, narrower when the list ran long, wider when the
// threshold fell outside.  C is this threshold moved by what the next gate's
// moved in the last layer, or, without that, carried into the next gate's
// scale.
template <int W>
__device__ void next_range(const RunArgs<W>& a, DevCtl* ctl, long long* drift, int n_drift, int k,
                           unsigned long long T, double rnorm, int reason, uint32_t cn,
                           unsigned long long range, Pub* p) {
    const int gi = n_drift > 0 ? (a.gate0 + k) % n_drift : 0;
    const int gn = n_drift > 0 ? (a.gate0 + k + 1) % n_drift : 0;
    const unsigned long long Tp = ctl->sp_tprev;
    if (n_drift > 0) drift[gi] = Tp ? (long long)(T - Tp) : 0LL;
    ctl->sp_tprev = T;
    ctl->stat_cands += cn;
    ctl->stat_range = range;
    int sft = ctl->sp_shift ? ctl->sp_shift : kRangeShift;
    switch (reason) {
        case 0: if (cn > a.cand_hi) sft -= 1; break;
        case 1: sft = kRangeShift; break;
        case 2: sft -= 2; break;
        default: sft += 1; break;
    }
    sft = sft < 8 ? 8 : (sft > 60 ? 60 : sft);
    ctl->sp_shift = sft;
    const long long dn = n_drift > 0 ? drift[gn] : 0LL;
    unsigned long long C;
    if (dn != 0LL) {
        const long long c = (long long)T + dn;
        C = c > 0 ? (unsigned long long)c : 0ULL;
    } else {
        C = abs_pattern(__dmul_rn(__longlong_as_double((long long)T), rnorm));
    }
    const unsigned long long h = 1ULL << sft;
    p->lo = C > h ? C - h : 0ULL;
    p->hi = C + h;
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

template <int W>
__device__ __forceinline__ PartFn<W> part_fn_of(const RunGate<W>& r) {
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
    for (int w = 0; w < W; ++w) { f.kx[w] = ~r.win[w]; f.kz[w] = ~r.win[w]; }
    f.pair = r.pair;
    f.sites = r.sites;
    return f;
}

// The instance's arrays (by compare-select: a dynamic index into an array of
// pointers would put it in local memory).
template <int W>
struct Arrays {
    PKey<W>*k0, *k1, *kp;
    double *c0, *c1, *cp;
    unsigned int *n0, *n1;
    int a;   // the contiguous state's buffer at the start
    __device__ __forceinline__ PKey<W>* run_keys(int b) const { return b ? k1 : k0; }
    __device__ __forceinline__ double* run_coef(int b) const { return b ? c1 : c0; }
    __device__ __forceinline__ PKey<W>* home(int h) const { return h ? run_keys(a ^ 1) : kp; }
    __device__ __forceinline__ double* coef(int x) const { return x ? run_coef(a ^ 1) : cp; }
    __device__ __forceinline__ unsigned int* cnt(int p) const { return p ? n1 : n0; }
};

template <int W>
__device__ __forceinline__ void read_pub(const RunShared* rs, Pub* s_pub) {
    static_assert(sizeof(Pub) % 8 == 0, "words");
    constexpr int N = sizeof(Pub) / 8;
    if (threadIdx.x < N)
        reinterpret_cast<unsigned long long*>(s_pub)[threadIdx.x] =
            __ldcg(reinterpret_cast<const unsigned long long*>(&rs->pub) + threadIdx.x);
    __syncthreads();
}

// Run gates [0, n_gates) n_layers times on one instance.  Returns false when
// a wait ran out.
template <int W>
__device__ bool run_instance(const RunArgs<W>& a, const RunGate<W>* gates, int n_gates, int inst,
                             Team& team) {
    using A = InStage<W>;
    constexpr uint32_t C = A::C;
    __shared__ Pub s_pub;
    // raw storage: a shared variable gets no constructor, and GateArg has a
    // default member initialiser
    __shared__ __align__(16) unsigned char s_g_raw[sizeof(GateArg<W>)];
    GateArg<W>& s_g = *reinterpret_cast<GateArg<W>*>(s_g_raw);
    __shared__ PartFn<W> s_f;
    __shared__ unsigned long long s_cv[kPushBuf];
    __shared__ uint32_t s_ci[kPushBuf];
    __shared__ uint32_t s_cn, s_cs, s_app, s_n, s_base32;
    __shared__ int s_over;
    __shared__ unsigned long long s_red[kBlock / 32], s_at;
    __shared__ uint32_t s_kept[kBlock / 32], s_above[kBlock / 32], s_w[kBlock / 32];
    __shared__ unsigned long long s_stat[8];   // first CTA: statistics of the run

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
    arr.n0 = a.cnt + (uint64_t)inst * 2 * a.part_max;
    arr.n1 = arr.n0 + a.part_max;
    arr.a = ctl->cur;
    // candidates and ties share the merge table's memory
    char* scr = static_cast<char*>(a.scratch) + (uint64_t)inst * a.scratch_stride;
    unsigned long long* cand_v = reinterpret_cast<unsigned long long*>(scr);
    uint32_t* cand_i = reinterpret_cast<uint32_t*>(scr + a.cand_cap * 8);
    PKey<W>* ties = reinterpret_cast<PKey<W>*>(scr + a.tie_off);
    long long* drift = a.drift + (uint64_t)inst * (a.drift_stride);
    const int n_drift = a.drift_gates;
    const int sites = a.n ? a.n[inst] : a.one_n;

    const PushList pl{s_cv, s_ci, &s_cn, &s_cs, cand_v, cand_i, nullptr, a.cand_cap};

    // start: the published state from the control block, both cursor arrays
    // zero, no chain head of an earlier use
    if (threadIdx.x < 8) s_stat[threadIdx.x] = 0ULL;
    for (uint32_t i = threadIdx.x; i < (uint32_t)A::S; i += kBlock) A::heads()[i] = 0u;
    for (uint32_t i = team.rank * kBlock + threadIdx.x; i < a.part_max; i += team.size * kBlock) {
        arr.n0[i] = 0u;
        arr.n1[i] = 0u;
    }
    if (leader) {
        for (int b = threadIdx.x; b < kBins; b += kBlock) rs->hist[b] = 0u;
        if (threadIdx.x == 0) {
            Pub p;
            p.T = 0;
            p.all_ties = 1;
            for (int w = 0; w < 4; ++w) p.tk[w] = 0;
            p.lo = ctl->sp_lo;
            p.hi = ctl->sp_hi;
            p.n = live_count(ctl, arr.a);
            p.rnorm = ctl->rnorm[arr.a];
            p.stop = ctl->status != 0;
            p.full = 0;
            p.rescatter = 1;
            rs->pub = p;
            memset(rs->acc, 0, sizeof rs->acc);
        }
    }
    if (!team_barrier(team, ctl)) return false;
    read_pub<W>(rs, &s_pub);

    uint32_t tag = 0, pass = 0;
    int layout = 0, hb = 0, cx = 0, par = 0, run_buf = arr.a;
    bool any = false;                   // a gate ran
    uint64_t run_n = s_pub.n;           // terms stored there
    uint32_t P = 0;
    uint64_t R = 0;
    bool over_one = false;              // the partitions hold for one gate only
    const int total = n_gates * a.n_layers;
    for (int gi = 0; gi < total; ++gi) {
        const int k = gi % n_gates;
        const int np_ = gi & 1;         // parity of this gate's counters
        if (s_pub.stop) break;          // uniform over the team
        if (threadIdx.x == 0) {
            s_g = gate_arg_of<W>(gates[k], a.maxw);
            s_f = part_fn_of<W>(gates[k]);
            s_cn = s_cs = 0u;
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
        if (gi == 0 || layout == 0 || over_one || gates[k].start || s_pub.rescatter) {
            bool pair = s_f.pair || !window_fits(sites, s_f.sites, n_in);
            for (int tries = 0; tries < 2; ++tries) {
                // at least a partition for every CTA of the team, of no fewer
                // than kMinPart terms, so that a small state uses the chip
                uint64_t want = (n_in + a.target - 1) / a.target;
                const uint64_t most = (n_in + a.min_part - 1) / a.min_part;
                const uint64_t wide = most < team.size ? most : team.size;
                if (want < wide) want = wide;
                if (want < 1) want = 1;
                if (want > a.part_max) want = a.part_max;
                if (!pair) {   // a stride holds a whole group (up to 4^sites strings)
                    const uint64_t gmax = 1ULL << (2 * s_f.sites);
                    if (a.home_cap / want < gmax) want = a.home_cap / gmax > 0 ? a.home_cap / gmax : 1;
                }
                P = (uint32_t)want;
                R = a.home_cap / P;
                PartPlan plan;
                plan.P = P;
                plan.R = R;
                PartFn<W> f = s_f;
                f.pair = pair ? 1 : 0;
                Pending<W> pd;
                pd.on = s_pub.T != 0ULL;
                pd.all_ties = s_pub.all_ties != 0;
                pd.T = s_pub.T;
                pd.tk = tk;
                const int dh = layout == 0 ? 0 : hb ^ 1, dx = layout == 0 ? 0 : cx ^ 1;
                int* over = reinterpret_cast<int*>(&acc->scatter_over);
                if (layout == 0) {
                    scatter_run<W>(arr.run_keys(run_buf), arr.run_coef(run_buf), run_n,
                                   (uint64_t)team.rank * kBlock, (uint64_t)team.size * kBlock, pd,
                                   ctl, arr.home(dh), arr.coef(dx), arr.cnt(par ^ 1), plan, g, f,
                                   over);
                } else {
                    const uint32_t oldP = s_base32;
                    const uint64_t oldR = a.home_cap / oldP;
                    for (uint32_t p = team.rank; p < oldP; p += team.size) {
                        const uint64_t c = __ldcg(arr.cnt(par) + p);
                        scatter_run<W>(arr.home(hb) + p * oldR, arr.coef(cx) + p * oldR, c, 0,
                                       kBlock, pd, ctl, arr.home(dh), arr.coef(dx),
                                       arr.cnt(par ^ 1), plan, g, f, over);
                    }
                }
                if (!team_barrier(team, ctl)) return false;
                if (leader && threadIdx.x == 0) s_stat[4] += 1;
                if (pair || !__ldcg(&acc->scatter_over)) {
                    hb = dh;
                    cx = dx;
                    par ^= 1;
                    layout = 1;
                    break;
                }
                // a window group passed a stride: again, by the pair key
                for (uint32_t i = team.rank * kBlock + threadIdx.x; i < a.part_max;
                     i += team.size * kBlock)
                    arr.cnt(par ^ 1)[i] = 0u;
                pair = true;
                if (!team_barrier(team, ctl)) return false;
            }
            over_one = pair;
            if (threadIdx.x == 0) s_base32 = P;
            __syncthreads();
        }
        // ---- merge, in place --------------------------------------------
        const unsigned long long dbits = a.delta_bits;
        const bool drop = s_pub.hi != 0ULL && s_pub.lo > 0ULL && s_pub.lo - 1ULL > dbits;
        const unsigned long long thr = drop ? s_pub.lo - 1ULL : dbits;
        const uint32_t p_id = identity_part<W>(P);
        PushList push_to = pl;
        push_to.gn = &acc->cand_n;
        auto push = [&](bool hit, unsigned long long v, uint64_t idx) {
            push_cand(push_to, hit, v, idx);
        };
        InStats st{0ULL, 0u, 0u};
        uint32_t n_long = 0;
        for (uint32_t p = team.rank; p < P; p += team.size) {
            const uint32_t np = __ldcg(arr.cnt(par) + p);
            InPlace<W> io;
            io.first = (uint64_t)p * R;
            io.keys = arr.home(hb) + io.first;
            io.cout = arr.coef(cx ^ 1) + io.first;
            io.n = np < R ? np : (uint32_t)R;
            io.room = (uint32_t)(R < 0xffffffffULL ? R : 0xffffffffULL);
            io.s_app = &s_app;
            io.over = &s_over;
            const double* cin = arr.coef(cx) + io.first;
            if (threadIdx.x == 0) s_app = 0u;
            if (io.n <= C) {
                // stage: all loads of a thread before its stores
                constexpr int U = (int)(C / kBlock);
                PKey<W> kk[U];
                double cc[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t i = u * kBlock + threadIdx.x;
                    if (i < io.n) {
                        kk[u] = load_key_stream(io.keys + i);
                        cc[u] = __ldcs(cin + i);
                    }
                }
                if (threadIdx.x < C / 32) A::dup()[threadIdx.x] = 0u;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t i = u * kBlock + threadIdx.x;
                    if (i < io.n) {
                        A::keys()[i] = kk[u];
                        A::vals()[i] = cc[u];
                    }
                }
                __syncthreads();
                inplace_pass<W, kBlock, false>(io.n, 0u, g, s_pub.T, s_pub.all_ties != 0, tk,
                                               s_pub.rnorm, thr, p == p_id, ctl, np_, ++tag, io, st,
                                               s_pub.lo, s_pub.hi, push);
            } else if (io.n <= 0xffffu) {
                // a partition above the staging capacity: its hash classes one
                // after another, each gathered with the strings' indices
                const uint32_t kc = (2u * io.n + C - 1u) / C;
                ++n_long;
                for (uint32_t j = 0; j < kc; ++j) {
                    if (threadIdx.x == 0) s_n = 0u;
                    if (threadIdx.x < C / 32) A::dup()[threadIdx.x] = 0u;
                    __syncthreads();
                    for (uint32_t i = threadIdx.x; i < io.n; i += kBlock) {
                        const PKey<W> K = load_key_stream(io.keys + i);
                        if (sub_pass(K, g, kc) != j) continue;
                        const uint32_t q = atomicAdd(&s_n, 1u);
                        if (q < C) {
                            A::keys()[q] = K;
                            A::vals()[q] = __ldcs(cin + i);
                            A::src()[q] = (uint16_t)i;
                        } else {
                            s_over = 1;   // the merge is done again
                        }
                    }
                    __syncthreads();
                    const uint32_t m = s_n < C ? s_n : C;
                    inplace_pass<W, kBlock, true>(m, 0u, g, s_pub.T, s_pub.all_ties != 0, tk,
                                                  s_pub.rnorm, thr, p == p_id, ctl, np_, ++tag, io,
                                                  st, s_pub.lo, s_pub.hi, push);
                }
            } else {
                if (threadIdx.x == 0) s_over = 1;
                __syncthreads();
            }
            if (threadIdx.x == 0) {
                const uint64_t c = (uint64_t)io.n + s_app;
                arr.cnt(par ^ 1)[p] = (unsigned int)(c < R ? c : R);
            }
            if (tag >= kHeadTagMax - 65536u) {   // tags start again
                __syncthreads();
                for (uint32_t i = threadIdx.x; i < (uint32_t)A::S; i += kBlock) A::heads()[i] = 0u;
                tag = 0;
            }
            __syncthreads();
        }
        // the CTA's counts and candidates
        auto flush = [&](Acc* to, InStats& s) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                s.out_max = max(s.out_max, __shfl_xor_sync(0xffffffffu, s.out_max, o));
                s.above += __shfl_xor_sync(0xffffffffu, s.above, o);
                s.kept += __shfl_xor_sync(0xffffffffu, s.kept, o);
            }
            if ((threadIdx.x & 31) == 0) {
                s_red[threadIdx.x >> 5] = s.out_max;
                s_kept[threadIdx.x >> 5] = s.kept;
                s_above[threadIdx.x >> 5] = s.above;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                unsigned long long mx = 0, kept = 0, above = 0;
                for (int w = 0; w < kBlock / 32; ++w) {
                    mx = max(mx, s_red[w]);
                    kept += s_kept[w];
                    above += s_above[w];
                }
                if (mx) atomicMax(&to->out_max, mx);
                if (kept) atomicAdd(&to->kept, kept);
                if (above) atomicAdd(&to->above, above);
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
        flush(acc, st);
        if (!team_barrier(team, ctl)) return false;
        unsigned long long kept = __ldcg(&acc->kept);
        bool redo = __ldcg(&acc->over) != 0u || (drop && kept < a.cap_M);
        if (redo) {
            // again in full from the same input, into a contiguous run
            acc = &rs->acc[np_][1];
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
            SelStats ss{0ULL, 0u};
            const CandRegions none{};
            for (uint32_t p = team.rank; p < P; p += team.size) {
                uint64_t np = __ldcg(arr.cnt(par) + p);
                if (np > R) np = R;
                const PKey<W>* kp = arr.home(hb) + (uint64_t)p * R;
                const double* cp = arr.coef(cx) + (uint64_t)p * R;
                ++pass;
                if (np <= (uint64_t)Stage<W>::C) {
                    for (uint32_t i = threadIdx.x; i < np; i += kBlock) {
                        PassArgs<W>::keys()[i] = load_key_stream(kp + i);
                        PassArgs<W>::vals()[i] = __ldcs(cp + i);
                    }
                    __syncthreads();
                    stage_pass<W, kBlock, PassRoom::kExact>((uint32_t)np, 0u, g, pd, s_pub.rnorm,
                                                            dbits, p == p_id, ctl, np_, pass, kout,
                                                            cout, ss, none, room);
                } else {
                    merge_long<W, kBlock>(kp, cp, np, g, pd, s_pub.rnorm, dbits, p == p_id, ctl,
                                          np_, &pass, kout, cout, ss, none, ~0ULL, room, nullptr,
                                          &s_n);
                }
            }
            n_long = 0;
            InStats s2{ss.out_max, 0u, 0u};
            flush(acc, s2);
            for (uint32_t i = threadIdx.x; i < (uint32_t)A::S; i += kBlock) A::heads()[i] = 0u;
            tag = 0;
            if (!team_barrier(team, ctl)) return false;
            kept = __ldcg(&acc->alloc);
            layout = 0;
            run_buf = arr.a;
            run_n = kept;
        } else {
            cx ^= 1;
            par ^= 1;
        }
        // ---- post and select --------------------------------------------
        // the spare cursors: the next scatter's
        for (uint32_t i = team.rank * kBlock + threadIdx.x; i < a.part_max; i += team.size * kBlock)
            arr.cnt(par ^ 1)[i] = 0u;
        if (layout == 0)
            for (uint32_t i = team.rank * kBlock + threadIdx.x; i < a.part_max;
                 i += team.size * kBlock)
                arr.cnt(par)[i] = 0u;
        bool active = false;
        if (leader) {
            if (a.cap_policy == 1 && kept > a.cap_M) active = true;
            unsigned long long lo = s_pub.lo, hi = s_pub.hi;
            const uint32_t cn = redo ? 0u : __ldcg(&acc->cand_n);
            const unsigned long long above = redo ? 0ULL : __ldcg(&acc->above);
            const unsigned long long omax = __ldcg(&acc->out_max);
            const double norm = *(volatile double*)&ctl->norm[np_];
            // why not the listed candidates: 1 no range, 2 list too long,
            // 3 threshold above the range, 4 below it
            const int reason = (hi == 0ULL || redo) ? (redo && hi ? 4 : 1)
                               : cn > a.cand_cap ? 2 : above >= a.cap_M ? 3
                               : above + cn < a.cap_M ? 4 : 0;
            const int failed = *(volatile int*)&ctl->status;
            SelOut so{0ULL, 1};
            PKey<W> key{};
            const bool fast = active && reason == 0 && !failed;
            if (fast)
                so = select_list<W>(cand_v, cand_i, cn, a.cap_M - above, 0ULL, 0ULL,
                                    hi > lo ? 64 - __clzll((long long)(hi - lo)) : 0,
                                    arr.home(hb), ties, &key, ctl);
            if (threadIdx.x == 0) {
                constexpr unsigned long long kInfBits = 0x7ff0000000000000ULL;
                if (omax >= kInfBits) set_status(ctl, ST_STATE, 4);
                if (abs_pattern(norm) >= kInfBits) set_status(ctl, ST_STATE, 5);
                if (a.cap_policy == 0 && kept > a.cap_M) set_status(ctl, ST_CAPACITY, 1);
                Pub p;
                p.rnorm = __ddiv_rn(1.0, norm);
                p.n = active ? a.cap_M : kept;
                p.T = fast ? so.v + lo : 0ULL;
                p.all_ties = fast ? so.all_ties : 1;
                for (int w = 0; w < 4; ++w) p.tk[w] = 0;
                if (fast)
                    for (int w = 0; w < W; ++w) { p.tk[w] = key.x[w]; p.tk[W + w] = key.z[w]; }
                p.full = active && !fast && !failed;
                p.lo = lo;
                p.hi = hi;
                p.rescatter = 0;
                // a state that grew several times since its scatter
                if (layout == 1 && p.n > 2ULL * a.target * P) p.rescatter = 1;
                p.stop = *(volatile int*)&ctl->status != 0;
                if (a.log) a.log[gi] = p.stop ? ~0ULL : p.n;
                s_stat[0] += 1;
                s_stat[1] += n_in;
                s_stat[2] += p.n;
                if (p.n > s_stat[3]) s_stat[3] = p.n;
                s_stat[5] += active ? 1 : 0;
                s_stat[6] += redo ? 1 : 0;
                s_stat[7] += __ldcg(&rs->acc[np_][0].n_long);
                ctl->sp_reason = reason;
                if (fast) next_range(a, ctl, drift, n_drift, k, p.T, p.rnorm, reason, cn, hi - lo, &p);
                if (p.full) {   // the team takes radix passes over the state
                    ctl->stat_sel_full += 1;
                    const unsigned long long top = omax > dbits ? omax - dbits : 0ULL;
                    rs->sel_prefix = 0ULL;
                    rs->sel_mask = 0ULL;
                    rs->sel_k = a.cap_M;
                    rs->sel_count = kept;
                    rs->sel_n = 0u;
                    p.T = top;   // the passes' value range (T itself comes after them)
                }
                memset(&rs->acc[np_ ^ 1][0], 0, sizeof rs->acc[0]);
                rs->pub = p;
            }
        }
        if (!team_barrier(team, ctl)) return false;
        read_pub<W>(rs, &s_pub);
        {
            if (s_pub.full && !s_pub.stop) {
                int top = s_pub.T ? 64 - __clzll((long long)s_pub.T) : 0;
                // every stored value: v = pattern - delta's
                auto each = [&](auto&& f) {
                    if (layout == 0) {
                        const double* c = arr.run_coef(run_buf);
                        for (uint64_t i = (uint64_t)team.rank * kBlock + (threadIdx.x & ~31u);
                             i < run_n; i += (uint64_t)team.size * kBlock) {
                            const uint64_t j = i + (threadIdx.x & 31u);
                            const unsigned long long b = j < run_n ? abs_pattern(__ldcs(c + j)) : 0ULL;
                            f(b > dbits, b - dbits, j);
                        }
                    } else {
                        for (uint32_t p = team.rank; p < P; p += team.size) {
                            const uint32_t n = __ldcg(arr.cnt(par) + p);
                            const double* c = arr.coef(cx) + (uint64_t)p * R;
                            for (uint32_t i = threadIdx.x & ~31u; i < n; i += kBlock) {
                                const uint32_t j = i + (threadIdx.x & 31u);
                                const unsigned long long b = j < n ? abs_pattern(__ldcs(c + j)) : 0ULL;
                                f(b > dbits, b - dbits, (uint64_t)p * R + j);
                            }
                        }
                    }
                };
                uint32_t* h = reinterpret_cast<uint32_t*>(g_stage);
                for (;;) {
                    const unsigned long long prefix = __ldcg(&rs->sel_prefix),
                                             mask = __ldcg(&rs->sel_mask),
                                             count = __ldcg(&rs->sel_count);
                    if (top <= 0 || (mask && count <= 4096ULL)) break;
                    const int shift = top > kDigit ? top - kDigit : 0;
                    const uint32_t dmask = (1u << (top - shift)) - 1u;
                    for (int b = threadIdx.x; b < kBins; b += kBlock) h[b] = 0u;
                    __syncthreads();
                    each([&](bool in, unsigned long long v, uint64_t) {
                        if (in && (v & mask) == prefix)
                            atomicAdd(&h[(uint32_t)(v >> shift) & dmask], 1u);
                    });
                    __syncthreads();
                    for (int b = threadIdx.x; b < kBins; b += kBlock)
                        if (h[b]) atomicAdd(&rs->hist[b], h[b]);
                    if (!team_barrier(team, ctl)) return false;
                    if (leader) {
                        __shared__ PickOut s_p;
                        for (int b = threadIdx.x; b < kBins; b += kBlock) {
                            h[b] = __ldcg(&rs->hist[b]);
                            rs->hist[b] = 0u;
                        }
                        __syncthreads();
                        pick_bin<true>(h, (uint32_t)__ldcg(&rs->sel_k), s_w, &s_p);
                        if (threadIdx.x == 0) {
                            rs->sel_prefix = prefix | ((unsigned long long)s_p.digit << shift);
                            rs->sel_mask = mask | ((unsigned long long)dmask << shift);
                            rs->sel_k = s_p.k_in;
                            rs->sel_count = s_p.count;
                        }
                    }
                    top = shift;
                    if (!team_barrier(team, ctl)) return false;
                }
                const unsigned long long prefix = __ldcg(&rs->sel_prefix),
                                         mask = __ldcg(&rs->sel_mask);
                PushList gp = pl;
                gp.gn = &rs->sel_n;
                if (threadIdx.x == 0) s_cn = kPushBuf;   // straight to the global list
                __syncthreads();
                each([&](bool in, unsigned long long v, uint64_t idx) {
                    push_cand(gp, in && (v & mask) == prefix, v, idx);
                });
                if (!team_barrier(team, ctl)) return false;
                if (leader) {
                    PKey<W> key{};
                    const uint32_t cn = __ldcg(&rs->sel_n);
                    SelOut so{0ULL, 1};
                    if (cn > a.cand_cap) {
                        if (threadIdx.x == 0) set_status(ctl, ST_CAPACITY, 63);
                    } else {
                        so = select_list<W>(cand_v, cand_i, cn, __ldcg(&rs->sel_k), prefix, mask,
                                            top, layout == 0 ? arr.run_keys(run_buf) : arr.home(hb),
                                            ties, &key, ctl);
                    }
                    if (threadIdx.x == 0) {
                        Pub p = s_pub;
                        p.T = so.v + dbits;
                        p.all_ties = so.all_ties;
                        for (int w = 0; w < W; ++w) { p.tk[w] = key.x[w]; p.tk[W + w] = key.z[w]; }
                        p.full = 0;
                        p.stop = *(volatile int*)&ctl->status != 0;
                        next_range(a, ctl, drift, n_drift, k, p.T, p.rnorm, ctl->sp_reason, cn,
                                   s_pub.T, &p);
                        rs->pub = p;
                    }
                }
                if (!team_barrier(team, ctl)) return false;
                read_pub<W>(rs, &s_pub);
            }
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
            const double* ci = layout == 1 ? arr.coef(cx) + (uint64_t)p * R : arr.run_coef(run_buf);
            const uint64_t n = layout == 1 ? __ldcg(arr.cnt(par) + p) : run_n;
            const uint64_t first = layout == 1 ? 0ULL : (uint64_t)team.rank * kBlock;
            const uint64_t step = layout == 1 ? (uint64_t)kBlock : (uint64_t)team.size * kBlock;
            for (uint64_t i0 = first; i0 < n; i0 += step) {
                const uint64_t i = i0 + threadIdx.x;
                PKey<W> K{};
                double c = 0.0;
                bool keep = false;
                if (i < n) {
                    K = load_key_stream(ki + i);
                    c = __ldcs(ci + i);
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
        ctl->seg = 0;
        ctl->need_scatter = 0;
        ctl->part_over = 0;
        ctl->sel_active = 0;
        ctl->sp_lo = s_pub.lo;
        ctl->sp_hi = s_pub.hi;
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

template <int W>
__global__ void __launch_bounds__(kBlock, W == 1 ? 4 : 3)
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
    for (int inst = (int)t; inst < a.B; inst += (int)teams) {
        const RunGate<W>* gates = a.gates ? a.gates + (uint64_t)inst * a.max_gates : chunk.g;
        const int n = a.gates ? a.n_gates[inst] : a.one_gates;
        if (n > 0 && !run_instance<W>(a, gates, n, inst, team)) return;
    }
}

}  // namespace

template <int W>
static int run_fit_w() {
    constexpr size_t smem = InStage<W>::kBytes;
    cudaFuncSetAttribute(k_run<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_run<W>, cudaFuncAttributePreferredSharedMemoryCarveout,
                         (int)cudaSharedmemCarveoutMaxShared);
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_run<W>, kBlock, smem);
    return n > 0 ? n : 1;
}

int run_fit(int W) { return W == 1 ? run_fit_w<1>() : run_fit_w<2>(); }

template <int W>
cudaError_t launch_run(const RunArgs<W>& a, const RunChunk<W>& chunk, int grid, cudaStream_t st) {
    void* args[2] = {const_cast<RunArgs<W>*>(&a), const_cast<RunChunk<W>*>(&chunk)};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_run<W>), dim3(grid),
                                       dim3(kBlock), args, InStage<W>::kBytes, st);
}

template cudaError_t launch_run<1>(const RunArgs<1>&, const RunChunk<1>&, int, cudaStream_t);
template cudaError_t launch_run<2>(const RunArgs<2>&, const RunChunk<2>&, int, cudaStream_t);

}  // namespace itpp
