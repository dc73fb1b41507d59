// itpp_inplace.cuh -- one gate over one staged partition, in place.
//
// A gate leaves almost every string where it is.  On the states of the
// measured chains and lattices 92 to 98 % of the strings commute with a gate,
// but only 1 to 8 % of them have their partner Q.K present, and the child
// sinh(theta) c of a lone string mostly lies below the threshold: a gate
// scales coefficients, and adds and drops a few strings.  So inside a window
// the partitions stay where the scatter put them: the keys are not written
// again, every coefficient goes to the same index of a second coefficient
// array (a dropped one as zero, which no reader takes for a term), and the
// few new strings are appended behind the partition.  That is 32 bytes per
// term and gate instead of 48, with no compaction, no output claims and no
// segment lists; the next window's scatter leaves the zeros behind.
//
// What bounds the pass is instruction issue and the double-precision pipe (two
// lanes per clock and SM; a warp holds it for every instruction however few
// lanes take part).  Hence: one multiplication for the normalisation and one
// for cosh over whole warps, and everything rare (a partner, a child that may
// pass the threshold) is put on a list per warp and done densely at its end.
// Whether a child can pass is decided before it is computed, on the exponent
// fields.  Two barriers per partition.
#pragma once

#include "itpp_common.cuh"
#include "itpp_stage.cuh"

namespace itpp {

namespace {

// Shared memory of one pass: staged keys and values, the heads of the chains
// of strings that share a pair slot, the chain links with two state bits, the
// original index of a gathered string (sub-passes), the warps' lists of rare
// strings and a bit per string that shares its slot with another.
template <int W>
struct InStage {
    static constexpr int C = StageGeom<W>::kItems, S = StageGeom<W>::kSlots;
    static constexpr size_t kKeys = 0;
    static constexpr size_t kVals = kKeys + sizeof(PKey<W>) * C;
    static constexpr size_t kHeads = kVals + sizeof(double) * (C + 2);
    static constexpr size_t kNext = kHeads + sizeof(uint32_t) * S;
    static constexpr size_t kSrc = kNext + sizeof(uint16_t) * C;
    static constexpr size_t kRare = kSrc + sizeof(uint16_t) * C;
    static constexpr size_t kDup = kRare + sizeof(uint16_t) * C;
    static constexpr size_t kBytes = (kDup + sizeof(uint32_t) * (C / 32) + 15) / 16 * 16;
    static_assert(kVals % 16 == 0 && kHeads % 16 == 0 && kNext % 16 == 0, "alignment");
    __device__ __forceinline__ static PKey<W>* keys() { return reinterpret_cast<PKey<W>*>(g_stage + kKeys); }
    __device__ __forceinline__ static double* vals() { return reinterpret_cast<double*>(g_stage + kVals); }
    __device__ __forceinline__ static uint32_t* heads() { return reinterpret_cast<uint32_t*>(g_stage + kHeads); }
    __device__ __forceinline__ static uint16_t* next() { return reinterpret_cast<uint16_t*>(g_stage + kNext); }
    __device__ __forceinline__ static uint16_t* src() { return reinterpret_cast<uint16_t*>(g_stage + kSrc); }
    __device__ __forceinline__ static uint16_t* rare() { return reinterpret_cast<uint16_t*>(g_stage + kRare); }
    __device__ __forceinline__ static uint32_t* dup() { return reinterpret_cast<uint32_t*>(g_stage + kDup); }
};

// A chain head holds (tag << 11) | (index + 1): heads of earlier passes carry
// another tag and read as empty, so nothing is cleared between passes.
constexpr uint32_t kHeadTagMax = (1u << 21) - 1u;
constexpr uint32_t kInLive = 0x8000u, kInComm = 0x4000u, kInPrev = 0x7ffu;

// Where a pass puts things and what it counts.  Every pointer is the
// partition's own: index 0 is its first string.
template <int W>
struct InPlace {
    PKey<W>* keys;        // the home (new strings are appended)
    double* cout;         // the other coefficient array, same indices
    uint64_t first;       // index of the partition's first string in the home
    uint32_t n;           // strings stored before the gate
    uint32_t room;        // the partition's stride
    uint32_t* s_app;      // strings appended so far (shared)
    int* over;            // set when the stride has no room for one
};

// What a thread counts over its partitions.
struct InStats {
    unsigned long long out_max;
    uint32_t kept, above;
};

// Whether |c m| can exceed the threshold, from the high words of the patterns
// (hm: m's with the exponent bias taken off, ht: the threshold's).  A pattern
// is the logarithm up to (1+a)(1+b) against 1+a+b, at most 0.1716 of an
// octave, and the low words and the rounding add at most 3 units: 0x2c140.
// The bound needs a normal threshold; below that everything may pass.
__device__ __forceinline__ bool child_may_pass(double c, int hm, int ht) {
    const int hc = (int)(__double2hiint(c) & 0x7fffffff);
    return hc + hm + 0x2c140 >= ht || ht < 0x00100000;
}

// One pass over n staged strings (keys(), vals() + shift; dup() cleared; a
// barrier since).  kGathered: string i is the partition's src()[i].
// sel_lo / sel_w: the candidate range of the select, width 0 when there is
// none; push(hit, pattern - lo, index) takes the candidates (warp-wide).
// Two barriers; the staging arrays are free again when it returns.
template <int W, int BLOCK, bool kGathered, class Push>
__device__ __forceinline__ void inplace_pass(uint32_t n, uint32_t shift, const GateArg<W>& g,
                                             unsigned long long pd_T, bool pd_ties,
                                             const PKey<W>& pd_key, double rnorm,
                                             unsigned long long thr, bool has_id, DevCtl* ctl,
                                             int nxt, uint32_t tag, const InPlace<W>& io,
                                             InStats& st, unsigned long long sel_lo,
                                             unsigned long long sel_hi, Push&& push) {
    using A = InStage<W>;
    double* vals = A::vals() + shift;
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned int lt = (1u << lane) - 1u;
    // A: live strings, normalised values, the chains of shared pair slots
    for (uint32_t i0 = threadIdx.x & ~31u; i0 < n; i0 += BLOCK) {
        const uint32_t i = i0 + lane;
        uint32_t f = 0, prev = 0;
        if (i < n) {
            const PKey<W> K = A::keys()[i];
            const double raw = vals[i];
            const unsigned long long b = abs_pattern(raw);
            bool live = b >= pd_T && b != 0ULL;   // pd_T == 0: no select pending
            if (b == pd_T && !pd_ties) live = live && !key_less(pd_key, K);
            double c = __dmul_rn(raw, rnorm);
            if (has_id && key_is_zero(K)) {
                c = 1.0;   // the identity's normalised value is exactly 1
                if (!live) set_status(ctl, ST_TRACE_ZERO, 43);
            }
            vals[i] = live ? c : 0.0;
            if (live) {
                f = kInLive;
                if (commutes(K, g)) {
                    const uint32_t o = atomicExch(A::heads() + pair_slot(K, g),
                                                  (tag << 11) | (i + 1u));
                    prev = (o >> 11) == tag ? (o & kInPrev) : 0u;
                    f |= kInComm | prev;
                    if (prev) atomicOr(A::dup() + ((prev - 1u) >> 5), 1u << ((prev - 1u) & 31u));
                }
            }
            A::next()[i] = (uint16_t)f;
        }
        const unsigned int m = __ballot_sync(0xffffffffu, prev != 0u);
        if (m && lane == 0) atomicOr(A::dup() + (i0 >> 5), m);
    }
    __syncthreads();                                                  // (1) chains built
    // B: every string that is alone in its slot (its partner is absent)
    const int hm = (int)(__double2hiint(g.msh) & 0x7fffffff) - 0x3ff00000;
    const int ht = (int)(thr >> 32);
    const bool weigh = g.maxw < 64 * W;
    // the identity as the gate: every string is its own partner
    uint64_t qbits = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) qbits |= g.qx[w] | g.qz[w];
    const bool self = qbits == 0;
    uint16_t* rare = A::rare() + (threadIdx.x >> 5) * (A::C / (BLOCK / 32));
    uint32_t n_rare = 0;
    for (uint32_t i0 = threadIdx.x & ~31u; i0 < n; i0 += BLOCK) {
        const uint32_t i = i0 + lane;
        const bool in = i < n;
        const uint32_t f = in ? A::next()[i] : 0u;
        const double c = in ? vals[i] : 0.0;
        const bool comm = (f & kInComm) != 0;
        const bool dup = comm && (self || ((A::dup()[i0 >> 5] >> lane) & 1u));
        double va = c;
        if (comm) va = __dmul_rn(c, g.ch);
        const unsigned int rb =
            __ballot_sync(0xffffffffu, dup || (comm && child_may_pass(c, hm, ht)));
        if ((rb >> lane) & 1u) rare[n_rare + __popc(rb & lt)] = (uint16_t)i;
        n_rare += __popc(rb);
        unsigned long long a = abs_pattern(va);
        bool keep = (f & kInLive) && !dup && a > thr;
        const uint32_t at = kGathered && in ? A::src()[i] : i;
        if (weigh && keep) keep = light(A::keys()[i], g.maxw);
        if (has_id && (f & kInLive) && !dup && key_is_zero(A::keys()[i])) {
            ctl->norm[nxt] = va;
            if (!keep) set_status(ctl, ST_TRACE_ZERO, 1);
            keep = true;
        }
        if (in && !dup) __stcs(io.cout + at, keep ? va : 0.0);
        if (!keep) a = 0ULL;
        st.out_max = max(st.out_max, a);
        st.kept += keep ? 1u : 0u;
        if (sel_hi) {   // uniform
            st.above += a > sel_hi ? 1u : 0u;
            push(keep && a - sel_lo <= sel_hi - sel_lo, a - sel_lo, io.first + at);
        }
    }
    __syncwarp();
    // C: this warp's rare strings, densely
    for (uint32_t r0 = 0; r0 < n_rare; r0 += 32u) {
        const bool in = r0 + lane < n_rare;
        const uint32_t i = in ? rare[r0 + lane] : 0u;
        PKey<W> K;
#pragma unroll
        for (int w = 0; w < W; ++w) { K.x[w] = 0; K.z[w] = 0; }
        double va = 0.0, vb = 0.0;
        bool ka = false, kb = false, dup = false;
        uint32_t at = i;
        if (in) {
            K = A::keys()[i];
            const double c = vals[i];
            if (kGathered) at = A::src()[i];
            dup = self || ((A::dup()[i >> 5] >> (i & 31u)) & 1u);
            bool neg, found = false;
            commute_sign(K, g, &neg);
            const double m = __longlong_as_double(
                __double_as_longlong(g.msh) ^ (neg ? (long long)0x8000000000000000ULL : 0LL));
            double cq = 0.0;
            if (dup) {
                // the chain of this slot; every string of it commutes
                uint32_t e = A::heads()[pair_slot(K, g)] & kInPrev;
                while (e) {
                    // (a string is its own partner only for Q = I)
                    if (key_is_partner(A::keys()[e - 1u], K, g)) {
                        found = true;
                        cq = vals[e - 1u];
                        break;
                    }
                    e = A::next()[e - 1u] & kInPrev;
                }
                va = __dmul_rn(c, g.ch);
                if (found) va = __dadd_rn(va, __dmul_rn(cq, m));
                ka = above(va, thr) && (!weigh || light(K, g.maxw));
                if (has_id && key_is_zero(K)) {
                    ctl->norm[nxt] = va;
                    if (!ka) set_status(ctl, ST_TRACE_ZERO, 1);
                    ka = true;
                }
                __stcs(io.cout + at, ka ? va : 0.0);
            }
            if (!found) {   // the child of a lone string
                vb = __dmul_rn(c, m);
                kb = above(vb, thr) && (!weigh || light(key_xor(K, g), g.maxw));
            }
        }
        const unsigned int bb = __ballot_sync(0xffffffffu, kb);
        uint32_t pos = 0;
        if (bb) {
            uint32_t q = 0;
            if (lane == 0) q = atomicAdd(io.s_app, (uint32_t)__popc(bb));
            pos = io.n + __shfl_sync(0xffffffffu, q, 0) + __popc(bb & lt);
            if (kb) {
                if (pos < io.room) {
                    store_key(io.keys + pos, key_xor(K, g));
                    __stcs(io.cout + pos, vb);
                } else {
                    *io.over = 1;
                    kb = false;
                }
            }
        }
        const unsigned long long a = ka ? abs_pattern(va) : 0ULL, b = kb ? abs_pattern(vb) : 0ULL;
        st.out_max = max(st.out_max, max(a, b));
        st.kept += (ka ? 1u : 0u) + (kb ? 1u : 0u);
        if (sel_hi) {
            st.above += (a > sel_hi ? 1u : 0u) + (b > sel_hi ? 1u : 0u);
            push(ka && a - sel_lo <= sel_hi - sel_lo, a - sel_lo, io.first + at);
            push(kb && b - sel_lo <= sel_hi - sel_lo, b - sel_lo, io.first + pos);
        }
    }
    __syncthreads();                                                  // (2) staging free
}

}  // namespace

}  // namespace itpp
