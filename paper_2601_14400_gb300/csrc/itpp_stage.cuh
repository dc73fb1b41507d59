// itpp_stage.cuh -- building blocks of the partitioned merge, shared by the
// separate kernels (itpp_part.cu) and the run kernel (itpp_run_impl.cuh): the
// partition function and plan, the scatter, and the merge in full of a
// partition staged in shared memory (pair table, merged children, threshold,
// write into a contiguous run), which is what a gate falls back to when the
// in-place merge (itpp_inplace.cuh) left out children that the bound then
// needed, or ran out of a partition's stride.
#pragma once

#include "itpp_common.cuh"
#include "itpp_gate_body.cuh"
#include "itpp_launch.h"

namespace itpp {

namespace {


// Partition geometry per word count: the mean partition size the scatter
// aims for, and the largest window (sites; a group holds at most 4^sites
// terms).  A pass has fixed costs and a partition beyond its capacity goes in
// sub-passes.  Merge per gate of the 64-site chain at 2^23 terms: 144, 136, 128
// and 144 us for targets of 500, 600, 700 and 850; of the 11 x 11 lattice at
// 2^22: 98, 94, 99 and 120 us for 300, 350, 400 and 440.  Windows of 6 or 7 sites
// instead of 5: a layer of 230 and 235 ms instead of 234 at 2^26.
template <int W> struct PartGeom;
template <> struct PartGeom<1> {
    static constexpr int kTarget = 700, kWinSites = 5;
};
template <> struct PartGeom<2> {
    static constexpr int kTarget = 350, kWinSites = 4;
};

struct PartPlan {
    uint32_t P;     // partitions
    uint64_t R;     // stride (capacity) of one partition in the scatter buffer
};

__device__ __forceinline__ PartPlan part_plan(uint64_t n, uint64_t pbuf_cap, uint32_t p_max,
                                              int target) {
    uint64_t P = (n + target - 1) / target;
    if (P < 1) P = 1;
    if (P > p_max) P = p_max;
    PartPlan pl;
    pl.P = (uint32_t)P;
    pl.R = pbuf_cap / P;
    return pl;
}

// The partition function of a window: the hash of the key with the
// window's sites cleared, or (pair mode) of the gate's pair key.
template <int W>
struct PartFn {
    uint64_t kx[W], kz[W];   // bits kept by the mask
    int pair;                // 1: pair-key mode
    int sites;               // sites of the window (mask mode)
    uint64_t px[W], pz[W];   // the pivot: the gate's lowest bit (all zero for Q = I)
};

// Mask mode needs many more possible groups than terms: a group (the terms
// with one pattern outside the window) holds up to 4^sites of them, and a
// partition that collects several large groups could outgrow its stride or
// the shared table.  So the window's mask is used only while
// 4^(n - sites) >= 64 N; a denser state (a small or saturated chain) falls
// back to the pair key of the window's first gate, valid for that gate only.
__device__ __forceinline__ bool window_fits(int n_sites, int w_sites, uint64_t n_terms) {
    const int free_bits = 2 * (n_sites - w_sites);
    const int need_bits = 6 + (n_terms > 1 ? 64 - __clzll((long long)(n_terms - 1)) : 0);
    return free_bits >= need_bits;
}

template <int W>
__device__ __forceinline__ uint32_t part_of(const PKey<W>& K, const GateArg<W>& g,
                                            const PartFn<W>& f, uint32_t P) {
    // masks and element-wise selects only: a conditional copy of the key,
    // or a selection of one of its words by index, puts the caller's key
    // arrays in local memory
    uint64_t piv = 0;
#pragma unroll
    for (int v = 0; v < W; ++v) piv |= (K.x[v] & f.px[v]) | (K.z[v] & f.pz[v]);
    const uint64_t flip = piv ? ~0ULL : 0ULL;   // pivot set: the pair key is K.Q
    PKey<W> k;
    if (f.pair) {   // the pair key K.Q when the pivot is set
#pragma unroll
        for (int v = 0; v < W; ++v) { k.x[v] = K.x[v] ^ (g.qx[v] & flip); k.z[v] = K.z[v] ^ (g.qz[v] & flip); }
    } else {        // the key with the window's sites cleared
#pragma unroll
        for (int v = 0; v < W; ++v) { k.x[v] = K.x[v] & f.kx[v]; k.z[v] = K.z[v] & f.kz[v]; }
    }
    const uint64_t h = key_hash(k);   // 32 significant bits
    return (uint32_t)((h * (uint64_t)P) >> 32);
}

// The kept set of a deferred top-M select, applied where terms are read.
template <int W>
struct Pending {
    bool on, all_ties;
    unsigned long long T;
    PKey<W> tk;
};

template <int W>
__device__ __forceinline__ Pending<W> pending_of(const DevCtl* ctl) {
    Pending<W> q;
    q.on = ctl->pend != 0;
    // without a pending select every pattern passes: none lies below zero
    q.all_ties = !q.on || ctl->pend_all_ties != 0;
    q.T = q.on ? ctl->pend_T : 0ULL;
#pragma unroll
    for (int w = 0; w < W; ++w) { q.tk.x[w] = ctl->pend_tie_key[w]; q.tk.z[w] = ctl->pend_tie_key[W + w]; }
    return q;
}

// Scatter terms [0, n) of a run (this CTA's part of it: from `first` on, every
// `stride`) into the partitions of a plan: the kept set of a pending select,
// one cursor claim per distinct partition of a warp.  over() is called where a
// stride has run out.
template <int W, class Over>
__device__ __forceinline__ void scatter_run(const PKey<W>* __restrict__ kin,
                                            const double* __restrict__ cin, uint64_t n,
                                            uint64_t first, uint64_t stride, const Pending<W>& pd,
                                            DevCtl* ctl, PKey<W>* pk, double* pc,
                                            unsigned int* cursor, const PartPlan& pl,
                                            const GateArg<W>& g, const PartFn<W>& f,
                                            Over&& over, uint32_t pad = 1u) {
    // whole warps iterate together (the cursor claim below is warp-wide);
    // U items per thread per round, their loads issued before any claim
    constexpr int U = 4;
    const unsigned int lt = (1u << (threadIdx.x & 31)) - 1u;
    for (uint64_t i0 = first; i0 < n; i0 += U * stride) {
        PKey<W> K[U];
        double c[U];
        bool live[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t i = i0 + (uint64_t)u * stride + threadIdx.x;
            live[u] = i < n;
            c[u] = 0.0;
#pragma unroll
            for (int w = 0; w < W; ++w) { K[u].x[w] = 0; K[u].z[w] = 0; }
            if (live[u]) {
                K[u] = load_key_stream(kin + i);
                c[u] = __ldcs(cin + i);
                live[u] = abs_pattern(c[u]) != 0ULL;   // a zero is no term
            }
        }
        // partitions and claims of all items before the first position is used:
        // their atomics are in flight together
        uint32_t part[U], peers[U], base[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (live[u] && pd.on && !cap_keep(K[u], c[u], pd.T, pd.all_ties, pd.tk)) {
                if (key_is_zero(K[u])) set_status(ctl, ST_TRACE_ZERO, 42);
                live[u] = false;
            }
            // one cursor claim per distinct partition in the warp: terms of
            // one group arrive together and would otherwise serialise on it
            part[u] = live[u] ? part_of(K[u], g, f, pl.P) : 0xffffffffu;
            peers[u] = __match_any_sync(0xffffffffu, part[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            base[u] = 0;
            if (live[u] && !(peers[u] & lt))
                base[u] = atomicAdd(cursor + (uint64_t)part[u] * pad, __popc(peers[u]));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t b = __shfl_sync(0xffffffffu, base[u], __ffs(peers[u]) - 1);
            if (!live[u]) continue;
            const unsigned int pos = b + __popc(peers[u] & lt);
            if (pos < pl.R) {
                const uint64_t d = (uint64_t)part[u] * pl.R + pos;
                store_key(pk + d, K[u]);
                pc[d] = c[u];
            } else {
                over();
            }
        }
    }
}

// Prefetch [p, p + bytes) into L2 with one bulk (TMA) request; the range is
// widened to 16-byte boundaries, which every buffer it is used on allows
// (its byte size is a multiple of 16).
__device__ __forceinline__ void l2_prefetch_bulk(const void* p, uint64_t bytes) {
    const uint64_t a = reinterpret_cast<uint64_t>(p);
    const uint64_t lo = a & ~15ULL;
    uint64_t sz = ((a + bytes + 15ULL) & ~15ULL) - lo;
    if (sz > (1ULL << 20)) sz = 1ULL << 20;
    if (sz) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(lo), "r"((uint32_t)sz)
                         : "memory");
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Sub-pass of a long partition's commuting string: a hash of its pair key (the
// member of {K, Q.K} without the gate's lowest bit), so a string and its partner
// always fall into the same one.  (With the gate's sites cleared instead, a gate
// on every site of a small system leaves a few keys for all strings, and one
// sub-pass gets more than it holds.)  The hash is seeded apart from the
// partition hash, which would put all strings of a partition in one class.
template <int W>
__device__ __forceinline__ uint32_t sub_pass(const PKey<W>& K, const GateArg<W>& g, uint32_t k) {
    uint64_t bit = 0, seen = 0;   // the lowest bit in K; bits of the gate so far
#pragma unroll
    for (int w = 0; w < 2 * W; ++w) {
        const uint64_t q = w < W ? g.qx[w] : g.qz[w - W];
        const uint64_t v = w < W ? K.x[w] : K.z[w - W];
        if (!seen) bit = v & q & (~q + 1ULL);
        seen |= q;
    }
    const uint64_t flip = bit ? ~0ULL : 0ULL;
    uint32_t h = 0x3c6ef372u;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const uint64_t mx = K.x[w] ^ (g.qx[w] & flip), mz = K.z[w] ^ (g.qz[w] & flip);
        h = murmur_mix(h, (uint32_t)mx);
        h = murmur_mix(h, (uint32_t)(mx >> 32));
        h = murmur_mix(h, (uint32_t)mz);
        h = murmur_mix(h, (uint32_t)(mz >> 32));
    }
    h ^= h >> 16;
    h *= 0x7feb352du;
    h ^= h >> 15;
    h *= 0x846ca68bu;
    h ^= h >> 16;
    return (uint32_t)(((uint64_t)h * k) >> 32);
}

// Append one value per lane that has one (every lane of the warp calls it)
// to this CTA's region of the candidate list: one shared-memory atomic per
// warp; entries past the region's end are dropped and counted, and the
// select then falls back to its full passes.
__device__ __forceinline__ void cand_push(bool hit, unsigned long long v, uint64_t pos,
                                          const CandRegions& cd, uint32_t* s_cn) {
    const unsigned int m = __ballot_sync(0xffffffffu, hit);
    if (!m) return;
    const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
    uint32_t q = 0;
    if (lane == leader) q = atomicAdd(s_cn, (uint32_t)__popc(m));
    q = __shfl_sync(0xffffffffu, q, leader);
    if (hit) {
        const uint64_t r = (uint64_t)q + __popc(m & ((1u << lane) - 1u));
        if (r < cd.region) {
            const uint64_t e = (uint64_t)blockIdx.x * cd.region + r;
            cd.v[e] = v;
            cd.idx[e] = (uint32_t)pos;
        }
    }
}

// Items a CTA stages in shared memory for one pass, and the slots of its
// pair table (at most half full).
template <int W> struct StageGeom;
template <> struct StageGeom<1> { static constexpr int kItems = 1024, kSlots = 2048; };
template <> struct StageGeom<2> { static constexpr int kItems = 512, kSlots = 1024; };

// Dynamic shared memory of the merge: the staged keys, their values (raw
// coefficient in, normalised coefficient after the join), the pair table and
// the pass's work list.
template <int W>
struct Stage {
    static constexpr int C = StageGeom<W>::kItems, S = StageGeom<W>::kSlots;
    static constexpr size_t kKeys = 0;
    static constexpr size_t kVals = kKeys + sizeof(PKey<W>) * C;
    static constexpr size_t kTab = kVals + sizeof(double) * C;
    static constexpr size_t kList = kTab + sizeof(uint32_t) * S;
    static constexpr size_t kBytes = (kList + sizeof(uint16_t) * C + 15) / 16 * 16;
    static_assert(kVals % 16 == 0 && kTab % 16 == 0, "alignment");
    static_assert(C <= 1024 && S <= 65536, "slot and index fields");
};

// The merge's dynamic shared memory (Stage<W> layout) and its small shared
// counters, at file scope so that every access is a constant offset from the
// CTA's shared window rather than a pointer held in registers.
extern __shared__ __align__(16) unsigned char g_stage[];
__shared__ uint32_t g_cn;        // this CTA's candidates
__shared__ unsigned long long g_range[2];   // candidate range [lo, hi] (hi == 0: none)
__shared__ unsigned long long g_delta;      // the threshold's own pattern
// per pass (indexed by its parity): the work list's lengths (pairs in the low
// half, pass-through strings in the high half) and the children kept so far
__shared__ uint32_t g_lists[2], g_kept[2];

// Commutation and the sign of Q P = s R in one pass over the masks.  Site by
// site Q and P anticommute where bit (x qz ^ z qx) is set, and there their
// product is +i or -i times a letter: minus for (Q, P) = (X, Z), (Z, Y),
// (Y, X), that is where (x qx) ^ (z qz ~qx) ^ (qx ~qz) is set.  With a
// anticommuting sites, m of them minus, the phase is i^(a - 2m): P and Q
// commute when a is even, and then s = -1 when a/2 - m is odd.  Only a
// modulo 4 and the parity of m are needed, so the second count is one popc of
// the xor of the halves (popc runs at a quarter of the integer rate).
template <int W>
__device__ __forceinline__ bool commute_sign(const PKey<W>& k, const GateArg<W>& g, bool* neg) {
    int a = 0;
    uint32_t mw = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const uint64_t an = (k.x[w] & g.qz[w]) ^ (k.z[w] & g.qx[w]);
        const uint64_t mi = an & ((k.x[w] & g.qx[w]) ^ (k.z[w] & (g.qz[w] & ~g.qx[w])) ^
                                  (g.qx[w] & ~g.qz[w]));
        a += __popcll(an);
        mw ^= (uint32_t)mi ^ (uint32_t)(mi >> 32);
    }
    *neg = (((a >> 1) ^ __popc(mw)) & 1) != 0;
    return (a & 1) == 0;
}

// Multilinear hash of the key with the gate's bits cleared, on which K and Q.K
// agree; its high bits are a slot (32-bit multiplies: the 64-bit ones cost four
// times as many issue slots).
template <int W>
__device__ __forceinline__ uint32_t pair_hash(const PKey<W>& K, const GateArg<W>& g) {
    uint32_t h = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const uint64_t mx = K.x[w] & ~g.qx[w], mz = K.z[w] & ~g.qz[w];
        h = h * 0x2c1b3c6du + (uint32_t)mx * 0x9e3779b1u + (uint32_t)(mx >> 32) * 0x85ebca77u +
            (uint32_t)mz * 0xc2b2ae3du + (uint32_t)(mz >> 32) * 0x27d4eb2fu;
    }
    return h;
}

template <int W>
__device__ __forceinline__ uint32_t pair_slot(const PKey<W>& K, const GateArg<W>& g) {
    constexpr uint32_t S = StageGeom<W>::kSlots;
    constexpr int kBits = S == 2048 ? 11 : 10;
    static_assert(S == (1u << kBits), "slots");
    return pair_hash(K, g) >> (32 - kBits);
}

// Pair table of one pass.  A commuting string K and its partner Q.K agree
// outside the gate's bits, so both hash to the same slot and walk the same
// probe sequence.  An occupied slot holds the index of the first string of a
// pair to arrive and the sign, and, once its partner has come by, the
// partner's index; 0 is a free slot.  The first free slot of the sequence is
// claimed by exactly one of the two (compare-and-swap), and the other finds
// the claim on its way; only it changes a claimed slot, with a plain store.
// The phase that consumes the table leaves every slot free again.
constexpr uint32_t kSlotUsed = 0x80000000u, kSlotNeg = 0x00200000u, kSlotPair = 0x00100000u;

// Enter string i into its pair; true when it claimed the pair's slot (*slot).
template <int W>
__device__ __forceinline__ bool pair_enter(const PKey<W>& K, const GateArg<W>& g, uint32_t i,
                                           bool neg, const PKey<W>* keys_s, uint32_t* tab,
                                           DevCtl* ctl, uint32_t* slot) {
    constexpr uint32_t S = StageGeom<W>::kSlots;
    const uint32_t claim = kSlotUsed | (neg ? kSlotNeg : 0u) | i;
    uint32_t h = pair_slot(K, g);
    for (uint32_t q = 0; q < S; ++q) {
        const uint32_t v = atomicCAS(tab + h, 0u, claim);
        if (v == 0u) {
            *slot = h;
            return true;
        }
        if (!(v & kSlotPair) && key_is_partner(keys_s[v & 0x3ffu], K, g)) {
            tab[h] = v | kSlotPair | (i << 10);
            return false;
        }
        h = (h + 1) & (S - 1);
    }
    set_status(ctl, ST_CAPACITY, 41);   // not reached: the table is at most half full
    return false;
}

// The identity as the gate: every string is its own partner.
template <int W>
__device__ __forceinline__ bool gate_is_identity(const GateArg<W>& g) {
    uint64_t q = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) q |= g.qx[w] | g.qz[w];
    return q == 0;
}

// Of the kept children: the largest pattern.
struct SelStats {
    unsigned long long out_max;
};

template <int W>
struct PassArgs {
    __device__ __forceinline__ static PKey<W>* keys() {
        return reinterpret_cast<PKey<W>*>(g_stage + Stage<W>::kKeys);
    }
    __device__ __forceinline__ static double* vals() {
        return reinterpret_cast<double*>(g_stage + Stage<W>::kVals);
    }
    __device__ __forceinline__ static uint32_t* tab() {
        return reinterpret_cast<uint32_t*>(g_stage + Stage<W>::kTab);
    }
    __device__ __forceinline__ static uint16_t* list() {
        return reinterpret_cast<uint16_t*>(g_stage + Stage<W>::kList);
    }
};

// The shared state of the passes before a CTA's first one (a barrier must
// follow): every slot free, both parities' counters zero.
template <int W, int BLOCK>
__device__ __forceinline__ void pass_init() {
    uint32_t* tab = PassArgs<W>::tab();
    for (uint32_t k = threadIdx.x; k < (uint32_t)StageGeom<W>::kSlots; k += BLOCK) tab[k] = 0u;
    if (threadIdx.x < 2) {
        g_lists[threadIdx.x] = 0u;
        g_kept[threadIdx.x] = 0u;
    }
}

// Count (and with kWrite store) a warp's kept children: K with va, and KQ with
// vb.  One shared atomic per warp gives the run; the order inside a
// run is immaterial.  Every lane of the warp calls it.
template <int W, bool kWrite>
__device__ __forceinline__ void emit_children(bool ka, bool kb, const PKey<W>& K,
                                              const GateArg<W>& g, double va, double vb,
                                              PKey<W>* kout, double* cout, uint64_t base,
                                              uint32_t* kept, SelStats& st) {
    const unsigned int ba = __ballot_sync(0xffffffffu, ka), bb = __ballot_sync(0xffffffffu, kb);
    const uint32_t na = __popc(ba), tot = na + __popc(bb);
    if (!tot) return;
    const int lane = threadIdx.x & 31;
    uint32_t q = 0;
    if (lane == 0) q = atomicAdd(kept, tot);
    if (!kWrite) return;
    q = __shfl_sync(0xffffffffu, q, 0);
    const unsigned int lt = (1u << lane) - 1u;
    const uint64_t pa = base + q + __popc(ba & lt), pb = base + q + na + __popc(bb & lt);
    unsigned long long a = 0, b = 0;
    if (ka) {
        store_key_stream(kout + pa, K);
        __stcs(cout + pa, va);
        a = abs_pattern(va);
    }
    if (kb) {
        store_key_stream(kout + pb, key_xor(K, g));
        __stcs(cout + pb, vb);
        b = abs_pattern(vb);
    }
    st.out_max = max(st.out_max, max(a, b));
}

// Phase B of a pass: the work list, pairs first (whole warps), then the
// strings that pass through.  kWrite: store the kept children from `base` on;
// kClear: leave the pair table free for the next pass.
template <int W, int BLOCK, bool kWrite, bool kClear>
__device__ __forceinline__ void pass_children(uint32_t n_pair, uint32_t n_through,
                                              const GateArg<W>& g, unsigned long long dbits,
                                              bool has_id, DevCtl* ctl, int nxt, PKey<W>* kout,
                                              double* cout, uint64_t base, uint32_t* kept,
                                              SelStats& st) {
    using A = PassArgs<W>;
    const double* vals = A::vals();
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t pair_end = (n_pair + 31u) & ~31u;
    for (uint32_t j0 = threadIdx.x & ~31u; j0 < pair_end + n_through; j0 += BLOCK) {
        PKey<W> K;
#pragma unroll
        for (int w = 0; w < W; ++w) { K.x[w] = 0; K.z[w] = 0; }
        double va = 0.0, vb = 0.0;
        bool ka = false, kb = false;
        if (j0 < pair_end) {   // warp-uniform
            const uint32_t j = j0 + lane;
            if (j < n_pair) {
                const uint32_t slot = A::list()[j];
                const uint32_t v = A::tab()[slot];
                if (kClear) A::tab()[slot] = 0u;
                const uint32_t e = v & 0x3ffu;
                K = A::keys()[e];
                const double c = vals[e];
                // a lone string's absent partner contributes a zero addend,
                // which changes no nonzero sum
                const double cq = (v & kSlotPair) ? vals[(v >> 10) & 0x3ffu] : 0.0;
                const double m = __longlong_as_double(
                    __double_as_longlong(g.msh) ^
                    ((v & kSlotNeg) ? (long long)0x8000000000000000ULL : 0LL));
                va = __dadd_rn(__dmul_rn(c, g.ch), __dmul_rn(cq, m));
                vb = __dadd_rn(__dmul_rn(cq, g.ch), __dmul_rn(c, m));
                ka = above(va, dbits) && light(K, g.maxw);
                kb = above(vb, dbits) && light(key_xor(K, g), g.maxw);
                if (has_id) {
                    if (key_is_zero(K)) {
                        if (kWrite) ctl->norm[nxt] = va;
                        if (!ka) set_status(ctl, ST_TRACE_ZERO, 1);
                        ka = true;
                    }
                    if (key_is_zero_xor(K, g)) {
                        if (kWrite) ctl->norm[nxt] = vb;
                        if (!kb) set_status(ctl, ST_TRACE_ZERO, 1);
                        kb = true;
                    }
                }
            }
        } else {
            const uint32_t j = j0 - pair_end + lane;
            if (j < n_through) {   // {P,Q} = 0: unchanged (or Q = I)
                const uint32_t i = A::list()[Stage<W>::C - 1 - j];
                K = A::keys()[i];
                va = vals[i];
                if (gate_is_identity(g)) va = __dadd_rn(__dmul_rn(va, g.ch), __dmul_rn(va, g.msh));
                ka = above(va, dbits) && light(K, g.maxw);
                if (has_id && key_is_zero(K)) {
                    if (kWrite) ctl->norm[nxt] = va;
                    if (!ka) set_status(ctl, ST_TRACE_ZERO, 1);
                    ka = true;
                }
            }
        }
        emit_children<W, kWrite>(ka, kb, K, g, va, vb, kout, cout, base, kept, st);
    }
}

// How a pass learns where its children go.  kExact: the children are counted
// first and room(kept) gives a run with no holes.  kCount: they are counted
// only.  kAt: the caller holds room for all of them at room().
enum class PassRoom { kAt, kExact, kCount };

// One pass of the gate over n staged strings.
//
// Join: the deferred select's kept set, commutation and sign, the normalised
// coefficient c; each commuting string enters its pair in the table, the
// claimers go on the work list and so do the strings that pass through.
// Children: one thread per pair (not per string) computes both merged
// children,
//   K:   c_K cosh(theta) + c_QK (-sinh(theta)) s,
//   QK:  c_QK cosh(theta) + c_K (-sinh(theta)) s
// (the sign s of Q.K = s QK is also that of Q.QK = s K, Sec. II.B), tests them
// and stores the kept ones.
//
// What bounds it: instruction issue, and the double-precision pipe (about two
// lanes per clock and SM on GB300, a whole warp's slot for every instruction
// however few lanes take part): hence the work list.
// Two barriers (and any the room call takes); returns the kept children
// (the same on every thread).  `pass` numbers the CTA's passes: counters
// alternate by its parity.
template <int W, int BLOCK, PassRoom kRoom, class Room>
__device__ __forceinline__ uint32_t stage_pass(uint32_t n, const GateArg<W>& g,
                                               const Pending<W>& pd, double rnorm,
                                               unsigned long long dbits, bool has_id, DevCtl* ctl,
                                               int nxt, uint32_t pass, PKey<W>* kout, double* cout,
                                               SelStats& st, Room&& room) {
    using A = PassArgs<W>;
    double* vals = A::vals();
    const uint32_t lane = threadIdx.x & 31u, par = pass & 1u;
    const unsigned int lt = (1u << lane) - 1u;
    for (uint32_t i0 = threadIdx.x & ~31u; i0 < n; i0 += BLOCK) {   // whole warps
        const uint32_t i = i0 + lane;
        uint32_t slot = 0;
        bool owner = false, through = false;
        if (i < n) {
            const PKey<W> K = A::keys()[i];
            const double raw = vals[i];
            const unsigned long long b = abs_pattern(raw);
            // pd.T == 0 with every tie kept: no select pending; a zero is no term
            bool live = b >= pd.T && b != 0ULL;
            if (b == pd.T && !pd.all_ties) live = live && !key_less(pd.tk, K);
            double c = __dmul_rn(raw, rnorm);
            if (has_id && key_is_zero(K)) {
                c = 1.0;   // the identity's normalised value is exactly 1
                if (!live) set_status(ctl, ST_TRACE_ZERO, 43);
            }
            vals[i] = c;
            bool neg;
            const bool comm = commute_sign(K, g, &neg) && !gate_is_identity(g);
            through = live && !comm;
            if (live && comm) owner = pair_enter(K, g, i, neg, A::keys(), A::tab(), ctl, &slot);
        }
        __syncwarp();
        const unsigned int bo = __ballot_sync(0xffffffffu, owner);
        const unsigned int bt = __ballot_sync(0xffffffffu, through);
        uint32_t q = 0;
        if (lane == 0) q = atomicAdd(&g_lists[par], (uint32_t)__popc(bo) | (__popc(bt) << 16));
        q = __shfl_sync(0xffffffffu, q, 0);
        if (owner) A::list()[(q & 0xffffu) + __popc(bo & lt)] = (uint16_t)slot;
        if (through) A::list()[Stage<W>::C - 1 - ((q >> 16) + __popc(bt & lt))] = (uint16_t)i;
    }
    __syncthreads();                                                  // (1) pairs and list built
    const uint32_t lists = g_lists[par];
    const uint32_t n_pair = lists & 0xffffu, n_through = lists >> 16;
    // the other parity's counters: last read before barrier (1), next used
    // after barrier (2)
    if (threadIdx.x == 0) {
        g_lists[par ^ 1u] = 0u;
        g_kept[par ^ 1u] = 0u;
    }
    uint32_t* kept = &g_kept[par];
    if (kRoom == PassRoom::kAt) {
        const unsigned long long base = room(n_through + 2u * n_pair);
        if (base != ~0ULL)
            pass_children<W, BLOCK, true, true>(n_pair, n_through, g, dbits, has_id, ctl,
                                                nxt, kout, cout, base, kept, st);
        __syncthreads();                                              // (2) staging free
        return *kept;
    }
    if (kRoom == PassRoom::kCount) {
        pass_children<W, BLOCK, false, true>(n_pair, n_through, g, dbits, has_id, ctl, nxt,
                                             kout, cout, 0ULL, kept, st);
        __syncthreads();
        return *kept;
    }
    pass_children<W, BLOCK, false, false>(n_pair, n_through, g, dbits, has_id, ctl, nxt,
                                          kout, cout, 0ULL, kept, st);
    __syncthreads();
    const uint32_t tot = *kept;
    const unsigned long long base = room(tot);
    __syncthreads();   // every thread has read the count: it restarts as the write position
    if (threadIdx.x == 0) *kept = 0u;
    __syncthreads();
    if (base != ~0ULL)
        pass_children<W, BLOCK, true, true>(n_pair, n_through, g, dbits, has_id, ctl, nxt,
                                            kout, cout, base, kept, st);
    else   // no room: the caller goes on with other instances, the table free
        pass_children<W, BLOCK, false, true>(n_pair, n_through, g, dbits, has_id, ctl, nxt,
                                             kout, cout, 0ULL, kept, st);
    __syncthreads();
    return tot;
}

// A partition above the staging capacity, in k sub-passes over the hash
// classes of the pair key (about C/2 strings each,
// gathered into the staging arrays).  A first round of the sub-passes only
// counts their children, room(total) gives a run's position (~0: none, nothing
// is written) and a second round writes them.  Every thread calls it.
template <int W, int BLOCK, class Room>
__device__ __forceinline__ void merge_long(const PKey<W>* kp, const double* cp, uint64_t np,
                                            const GateArg<W>& g, const Pending<W>& pd,
                                            double rnorm, unsigned long long dbits, bool has_id,
                                            DevCtl* ctl, int nxt, uint32_t* pass,
                                            PKey<W>* kout, double* cout, SelStats& st,
                                            Room&& room, uint32_t* s_n) {
    using A = PassArgs<W>;
    constexpr uint32_t C = Stage<W>::C;
    const uint32_t k = (uint32_t)((2 * np + C - 1) / C);
    uint32_t total = 0;
    for (int write = 0; write < 2; ++write) {
        unsigned long long base = 0ULL;
        if (write) {
            base = room(total);
            if (base == ~0ULL) break;
        }
        uint32_t done = 0;
        for (uint32_t j = 0; j < k; ++j) {
            if (threadIdx.x == 0) *s_n = 0u;
            __syncthreads();
            for (uint64_t i = threadIdx.x; i < np; i += BLOCK) {
                const PKey<W> K = load_key_stream(kp + i);
                const double raw = __ldcs(cp + i);
                const bool live = abs_pattern(raw) != 0ULL &&
                                  cap_keep(K, raw, pd.T, pd.all_ties, pd.tk);
                if (!live) {
                    if (key_is_zero(K)) set_status(ctl, ST_TRACE_ZERO, 43);
                    continue;
                }
                const uint32_t cls = commutes(K, g) ? sub_pass(K, g, k) : (uint32_t)(i % k);
                if (cls != j) continue;
                const uint32_t q = atomicAdd(s_n, 1u);
                if (q < C) {
                    A::keys()[q] = K;
                    A::vals()[q] = raw;
                } else {
                    set_status(ctl, ST_CAPACITY, 44);
                }
            }
            __syncthreads();
            const uint32_t n = *s_n < C ? *s_n : C;
            *pass += 1u;
            if (write) {
                const unsigned long long at = base + done;
                done += stage_pass<W, BLOCK, PassRoom::kAt>(
                    n, g, pd, rnorm, dbits, has_id, ctl, nxt, *pass, kout, cout, st,
                    [at](uint32_t) { return at; });
            } else {
                done += stage_pass<W, BLOCK, PassRoom::kCount>(
                    n, g, pd, rnorm, dbits, has_id, ctl, nxt, *pass, kout, cout, st,
                    [](uint32_t) { return 0ULL; });
            }
        }
        total = done;
    }
}

// The partition that holds the identity (the all-zero key, in every mode of
// the partition function): only there the identity and the child that falls
// on it need looking for.
template <int W>
__device__ __forceinline__ uint32_t identity_part(uint32_t P) {
    PKey<W> k;
#pragma unroll
    for (int w = 0; w < W; ++w) { k.x[w] = 0; k.z[w] = 0; }
    return (uint32_t)((key_hash(k) * (uint64_t)P) >> 32);
}

template <int W, int BLOCK>
struct PartOcc {
    // CTAs per SM that the launch bound of the merge in full asks for
    static constexpr int kMin = BLOCK <= 256 ? (W == 1 ? 6 : 5) : 2;
};

}  // namespace

}  // namespace itpp
