// itpp_inplace.cuh -- one gate over one partition, in place.
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
// What bounds the pass is instruction issue (56 % of the slots at 2^23 terms of
// the 64-site chain) and the double-precision pipe (44 %: two lanes per clock
// and SM; a warp holds it for every instruction however few lanes take part),
// and the latency of a partition's few dependent steps.  Hence: one
// multiplication for the normalisation and one for cosh over whole warps, and
// everything rare (a partner, a child that may pass the threshold) is put on a
// list and done densely afterwards.  Whether a child can pass is decided before
// it is computed, on the exponent fields.  A gate at 2^26 terms takes 1.03 ms
// this way (3.1 TB/s of the 48 bytes a term that a gate reads and writes at
// least without it); staging, pairing and writing all children took 1.81 ms.
//
// Two sets of shared arrays, so that a partition's last barrier can go, made it
// slower (1.35 ms): the second set's addresses spill.
#pragma once

#include "itpp_common.cuh"
#include "itpp_stage.cuh"

namespace itpp {

namespace {

// Slots of the separate kernel's passes, where shared memory has room for them:
// a string that shares its slot with another that is not its partner is looked
// at twice (700 strings in 4,096 slots: 15 %, in 8,192: 8 %).  Merge per gate of
// the 64-site chain at 2^26 terms 1074 us with 4,096, 1024 with 8,192.
constexpr int kLargeBits = 13;

// Geometry and shared memory of one pass: up to kItems strings, each read from
// global memory into registers (nothing is staged: the rare ones are read
// again, from L1 or L2), the heads of the chains of strings that share a slot,
// the chain links, the index of a gathered string (sub-passes) and the list of
// rare strings.
template <int W, int BITS = 12>
struct InPass {
    static constexpr int C = StageGeom<W>::kItems, kSlotBits = BITS, S = 1 << BITS;
    static constexpr size_t kHeads = 0;
    static constexpr size_t kNext = kHeads + sizeof(uint32_t) * S;
    static constexpr size_t kSrc = kNext + sizeof(uint16_t) * C;
    static constexpr size_t kRare = kSrc + sizeof(uint16_t) * C;
    static constexpr size_t kBytes = (kRare + sizeof(uint16_t) * C + 15) / 16 * 16;
    __device__ __forceinline__ static uint32_t* heads() { return reinterpret_cast<uint32_t*>(g_stage + kHeads); }
    __device__ __forceinline__ static uint16_t* next() { return reinterpret_cast<uint16_t*>(g_stage + kNext); }
    __device__ __forceinline__ static uint16_t* src() { return reinterpret_cast<uint16_t*>(g_stage + kSrc); }
    __device__ __forceinline__ static uint16_t* rare() { return reinterpret_cast<uint16_t*>(g_stage + kRare); }
    __device__ __forceinline__ static uint32_t slot(const PKey<W>& K, const GateArg<W>& g) {
        return pair_hash(K, g) >> (32 - kSlotBits);
    }
};

// A chain head holds (tag << 11) | (index + 1): heads of earlier passes carry
// another tag and read as empty, so nothing is cleared between passes.
constexpr uint32_t kHeadTagMax = (1u << 21) - 1u;
constexpr uint32_t kInPrev = 0x7ffu;

// Where a pass puts things and what it counts.  Every pointer is the
// partition's own: index 0 is its first string.
template <int W>
struct InPlace {
    PKey<W>* keys;        // the home (new strings are appended)
    const double* cin;    // its coefficients
    double* cout;         // the other coefficient array, same indices
    uint64_t first;       // index of the partition's first string in the home
    uint32_t n;           // strings stored before the gate
    uint32_t room;        // the partition's stride
    uint32_t* s_app;      // strings appended so far (shared, zero at first)
    uint32_t* s_rare;     // rare strings listed so far (shared, zero at first)
    int* over;            // set when the stride has no room for one
};

// What a thread counts over its partitions: the high word of the largest
// pattern, the kept strings.
struct InStats {
    uint32_t hi_max, kept;
};

// Whether a lone string's child can pass the threshold is decided on the high
// words of the patterns of |c|, |m| and the threshold.  A pattern is the
// logarithm up to (1+a)(1+b) against 1+a+b, at most 0.1716 of an octave, and the
// low words and the rounding add at most 3 units: 0x2c140.  The bound needs a
// normal threshold; below that everything may pass.

// Predicated shared-memory steps of the main rows, without the branches that a
// conditional atomic otherwise costs every row.
__device__ __forceinline__ uint32_t exch_if(bool on, uint32_t* p, uint32_t v) {
    uint32_t o;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\tmov.u32 %0, 0;\n\t"
                 "@p atom.shared.exch.b32 %0, [%1], %2;\n\t}"
                 : "=r"(o) : "r"(smem_addr(p)), "r"(v), "r"((uint32_t)on) : "memory");
    return o;
}

__device__ __forceinline__ void list_if(bool on, uint32_t* count, uint16_t* list, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .u32 q;\n\t.reg .u16 h;\n\t"
                 "setp.ne.u32 p, %3, 0;\n\tmov.u32 q, 0;\n\tcvt.u16.u32 h, %2;\n\t"
                 "@p atom.shared.add.u32 q, [%0], 1;\n\tshl.b32 q, q, 1;\n\t"
                 "add.u32 q, q, %1;\n\t@p st.shared.u16 [q], h;\n\t}"
                 :: "r"(smem_addr(count)), "r"(smem_addr(list)), "r"(v), "r"((uint32_t)on)
                 : "memory");
}

// The identity's merged child, of pattern a.  At or below the threshold the
// trace is lost; at or below the limit predicted for the select only the
// prediction is wrong (the thresholds of a state's first gates move by octaves),
// and the gate is merged again in full.
__device__ __forceinline__ void identity_kept(bool keep, unsigned long long a, DevCtl* ctl, int* over) {
    if (keep) return;
    if (a <= g_delta) set_status(ctl, ST_TRACE_ZERO, 1);
    else *over = 1;
}

// A thread's strings of a pass (row r: string r * BLOCK + thread), zero past the
// end.
template <int W, int BLOCK>
struct InRows {
    static constexpr int N = InPass<W>::C / BLOCK;
    PKey<W> K[N];
    double c[N];
};

template <int W, int BLOCK, bool kGathered>
__device__ __forceinline__ void load_rows(InRows<W, BLOCK>& rows, const PKey<W>* keys,
                                          const double* cin, uint32_t n,
                                          const uint16_t* src = nullptr) {
    const PKey<W>* kp = keys + threadIdx.x;
    const double* cp = cin + threadIdx.x;
#pragma unroll
    for (int r = 0; r < InRows<W, BLOCK>::N; ++r) {
#pragma unroll
        for (int w = 0; w < W; ++w) { rows.K[r].x[w] = 0; rows.K[r].z[w] = 0; }
        rows.c[r] = 0.0;
        if (threadIdx.x + r * BLOCK < n) {
            if (kGathered) {
                const uint32_t at = src[threadIdx.x + r * BLOCK];
                rows.K[r] = load_key_ca(keys + at);
                rows.c[r] = cin[at];
            } else {
                rows.K[r] = load_key_ca(kp + r * BLOCK);
                rows.c[r] = cp[r * BLOCK];
            }
        }
    }
}

// One pass over n >= 1 strings: string i is the partition's i-th, or (kGathered)
// its src()[i]-th; rows holds them.  *s_app and *s_rare are zero (seen by every
// thread after the first barrier here).  thr: kept is what lies above it;
// near_hi: kept strings up to this pattern are candidates of the select (0:
// none), push(hit, pattern - thr - 1, index) takes them (warp-wide).  kPlain:
// neither the identity's partition nor a weight cutoff nor Q = I.  then() is
// called when the rows are done with and before the rare strings are: the
// caller loads its next ones there, so that their latency is not waited for.
// Three barriers; the shared arrays are free again when it returns.
template <int W, int BLOCK, int BITS, bool kGathered, bool kPlain, class Push, class Then>
__device__ __forceinline__ void inplace_pass(uint32_t n, const GateArg<W>& g,
                                             unsigned long long pd_T, bool pd_ties,
                                             const PKey<W>& pd_key, double rnorm,
                                             unsigned long long thr, bool has_id, DevCtl* ctl,
                                             int nxt, uint32_t tag, const InPlace<W>& io,
                                             InStats& st, unsigned long long near_hi,
                                             InRows<W, BLOCK>& rows, Push&& push, Then&& then) {
    using A = InPass<W, BITS>;
    constexpr int ROWS = InRows<W, BLOCK>::N;
    PKey<W>(&K)[ROWS] = rows.K;
    double(&c)[ROWS] = rows.c;
    // per row: slot | commutes | not the first to arrive in its chain | live,
    // and (special) the identity or past the weight cutoff; two rows a word
    // where they fit
    constexpr uint32_t kComm = 1u << BITS, kPrev = 2u << BITS, kLive = 4u << BITS, kSpecial = 8u << BITS;
    constexpr int PER = BITS <= 12 ? 2 : 1;
    const uint32_t lane = threadIdx.x & 31u, w0 = threadIdx.x & ~31u;
    const unsigned int lt = (1u << lane) - 1u;
    const bool weigh = !kPlain && g.maxw < 64 * W;
    const uint32_t me0 = (tag << 11) + threadIdx.x + 1u;   // + r * BLOCK: this thread's string of row r
    const unsigned long long floor_T = pd_T ? pd_T - 1ULL : 0ULL;   // live: above it (a zero is no term)
    // the identity as the gate: every string is its own partner
    uint64_t qbits = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) qbits |= g.qx[w] | g.qz[w];
    const bool self = !kPlain && qbits == 0;
    // A: live strings, normalised values, the chains of shared slots
    uint32_t flags[(ROWS + PER - 1) / PER];
#pragma unroll
    for (int r = 0; r < (ROWS + PER - 1) / PER; ++r) flags[r] = 0u;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        if (r * BLOCK + w0 >= n) break;   // whole warps
        const unsigned long long b = abs_pattern(c[r]);   // 0 past the end
        bool live = b > floor_T;
        if (!pd_ties) live = live && (b != pd_T || !key_less(pd_key, K[r]));
        c[r] = __dmul_rn(c[r], rnorm);
        uint32_t f = 0;
        if (!kPlain) {
            if (has_id && threadIdx.x + r * BLOCK < n && key_is_zero(K[r])) {
                c[r] = 1.0;   // the identity's normalised value is exactly 1
                f = kSpecial;
                if (!live) set_status(ctl, ST_TRACE_ZERO, 43);
            }
            if (weigh && !light(K[r], g.maxw)) f = kSpecial;
        }
        const bool comm = live && commutes(K[r], g);
        const uint32_t slot = A::slot(K[r], g);
        const uint32_t d = exch_if(comm, A::heads() + slot, me0 + r * BLOCK) ^ (tag << 11);
        const uint32_t prev = d <= kInPrev ? d : 0u;
        if (comm) A::next()[threadIdx.x + r * BLOCK] = (uint16_t)prev;
        f |= comm ? slot | kComm : 0u;
        f |= prev ? kPrev : 0u;
        f |= live ? kLive : 0u;
        flags[r / PER] |= f << (16 * (r % PER));
    }
    __syncthreads();                                                  // (1) chains built
    // B: every string that is alone in its slot (its partner is absent).
    // child_may_pass as one sum: the high words of |c| and |m| against the
    // threshold's
    const int ht = (int)(thr >> 32);
    // (a sum at or above zero whatever |c| is: cut off, so that |c| of 2 and
    // more does not carry it past the largest int)
    const int hm = ht < 0x00100000 ? 0
                                   : min(0, (int)(__double2hiint(g.msh) & 0x7fffffff) - 0x3ff00000 +
                                                0x2c140 - ht);
    double* op = io.cout + threadIdx.x;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        if (r * BLOCK + w0 >= n) break;   // whole warps
        const uint32_t f = flags[r / PER] >> (16 * (r % PER));
        const bool comm = (f & kComm) != 0;
        const uint32_t me = me0 + r * BLOCK;
        uint32_t head = me;
        if (comm) head = A::heads()[f & (uint32_t)(A::S - 1)];
        bool dup = ((f & kPrev) | (head ^ me)) != 0u;
        if (!kPlain) dup = dup || (self && comm);
        const bool may = comm && (int)(__double2hiint(c[r]) & 0x7fffffff) + hm >= 0;
        list_if(dup || may, io.s_rare, A::rare(), (threadIdx.x + r * BLOCK) | (dup ? 0x8000u : 0u));
        double va = c[r];
        if (comm) va = __dmul_rn(va, g.ch);
        const unsigned long long a = abs_pattern(va);
        bool keep = (f & kLive) && !dup && a > thr;
        const bool in = threadIdx.x + r * BLOCK < n;
        uint32_t at = threadIdx.x + r * BLOCK;
        if (kGathered) at = A::src()[in ? at : 0u];
        if (!kPlain && (f & kSpecial) && (f & kLive) && !dup) {
            if (has_id && key_is_zero(load_key_ca(io.keys + at))) {
                ctl->norm[nxt] = va;
                identity_kept(keep, a, ctl, io.over);
                keep = true;
            } else {
                keep = false;
            }
        }
        if (in && !dup) __stcs(kGathered ? io.cout + at : op + r * BLOCK, keep ? va : 0.0);
        st.hi_max = max(st.hi_max, keep ? (uint32_t)(a >> 32) : 0u);
        st.kept += keep ? 1u : 0u;
        if (near_hi) {   // uniform
            const bool hit = keep && a <= near_hi;
            if (__any_sync(0xffffffffu, hit)) push(hit, a - thr - 1ULL, io.first + at);
        }
    }
    then();
    __syncthreads();                                                  // (2) the list is complete
    // C: the rare strings, densely (read again)
    const uint32_t n_rare = *io.s_rare;
    for (uint32_t r0 = w0; r0 < n_rare; r0 += BLOCK) {
        const bool in = r0 + lane < n_rare;
        const uint32_t e0 = in ? A::rare()[r0 + lane] : 0u;
        const uint32_t i = e0 & 0x7fffu;
        const bool dup = (e0 & 0x8000u) != 0;
        const uint32_t at = kGathered && in ? A::src()[i] : i;
        PKey<W> X;
#pragma unroll
        for (int w = 0; w < W; ++w) { X.x[w] = 0; X.z[w] = 0; }
        double va = 0.0, vb = 0.0;
        bool ka = false, kb = false;
        if (in) {
            X = load_key_ca(io.keys + at);
            const bool id = has_id && key_is_zero(X);
            const double cx = id ? 1.0 : __dmul_rn(io.cin[at], rnorm);
            bool neg, found = false;
            commute_sign(X, g, &neg);
            const double m = __longlong_as_double(
                __double_as_longlong(g.msh) ^ (neg ? (long long)0x8000000000000000ULL : 0LL));
            if (dup) {
                // the chain of this slot; every string of it is live and
                // commutes (a string is its own partner only for Q = I)
                uint32_t e = A::heads()[A::slot(X, g)] & kInPrev;
                double cq = 0.0;
                for (uint32_t q = 0; e && q < n; ++q) {
                    const uint32_t ea = kGathered ? A::src()[e - 1u] : e - 1u;
                    const PKey<W> Y = load_key_ca(io.keys + ea);
                    if (key_is_partner(Y, X, g)) {
                        found = true;
                        cq = has_id && key_is_zero(Y) ? 1.0 : __dmul_rn(io.cin[ea], rnorm);
                        break;
                    }
                    e = A::next()[e - 1u];
                }
                va = __dmul_rn(cx, g.ch);
                if (found) va = __dadd_rn(va, __dmul_rn(cq, m));
                ka = above(va, thr) && (!weigh || light(X, g.maxw));
                if (id) {
                    ctl->norm[nxt] = va;
                    identity_kept(ka, abs_pattern(va), ctl, io.over);
                    ka = true;
                }
                __stcs(io.cout + at, ka ? va : 0.0);
            }
            if (!found) {   // the child of a lone string
                vb = __dmul_rn(cx, m);
                kb = above(vb, thr) && (!weigh || light(key_xor(X, g), g.maxw));
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
                    store_key(io.keys + pos, key_xor(X, g));
                    __stcs(io.cout + pos, vb);
                } else {
                    *io.over = 1;
                    kb = false;
                }
            }
        }
        const unsigned long long a = ka ? abs_pattern(va) : 0ULL, b = kb ? abs_pattern(vb) : 0ULL;
        st.hi_max = max(st.hi_max, max((uint32_t)(a >> 32), (uint32_t)(b >> 32)));
        st.kept += (ka ? 1u : 0u) + (kb ? 1u : 0u);
        if (near_hi) {
            push(ka && a <= near_hi, a - thr - 1ULL, io.first + at);
            push(kb && b <= near_hi, b - thr - 1ULL, io.first + pos);
        }
    }
    __syncthreads();                                                  // (3) shared arrays free
}

// A partition of any size up to 65,535 strings: one pass, or its hash classes
// one after another, each a list of indices (strings and partners agree on
// the class).  Every thread calls it, with the partition in rows when one pass
// holds it; *s_app and *s_rare are zero.  Returns whether it took sub-passes.
template <int W, int BLOCK, int BITS, class Push, class Then>
__device__ __forceinline__ bool inplace_partition(const GateArg<W>& g, unsigned long long pd_T,
                                                  bool pd_ties, const PKey<W>& pd_key,
                                                  double rnorm, unsigned long long thr,
                                                  bool has_id, DevCtl* ctl, int nxt, uint32_t* tag,
                                                  const InPlace<W>& io, InStats& st,
                                                  unsigned long long near_hi, uint32_t* s_n,
                                                  InRows<W, BLOCK>& rows, Push&& push,
                                                  Then&& then) {
    using A = InPass<W, BITS>;
    constexpr uint32_t C = A::C;
    if (io.n == 0u) {
        then();
        return false;
    }
    uint64_t qbits = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) qbits |= g.qx[w] | g.qz[w];
    const bool plain = !has_id && g.maxw >= 64 * W && qbits != 0;
    if (io.n <= C) {
        if (plain)
            inplace_pass<W, BLOCK, BITS, false, true>(io.n, g, pd_T, pd_ties, pd_key, rnorm, thr, false,
                                                ctl, nxt, ++*tag, io, st, near_hi, rows, push, then);
        else
            inplace_pass<W, BLOCK, BITS, false, false>(io.n, g, pd_T, pd_ties, pd_key, rnorm, thr, has_id,
                                                 ctl, nxt, ++*tag, io, st, near_hi, rows, push,
                                                 then);
        return false;
    }
    if (io.n > 0xffffu) {
        if (threadIdx.x == 0) *io.over = 1;   // the gate is merged again
        then();
        return true;
    }
    const uint32_t kc = (2u * io.n + C - 1u) / C;
    for (uint32_t j = 0; j < kc; ++j) {
        if (threadIdx.x == 0) *s_n = *io.s_rare = 0u;
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < io.n; i += BLOCK) {
            if (sub_pass(load_key_ca(io.keys + i), g, kc) != j) continue;
            const uint32_t q = atomicAdd(s_n, 1u);
            if (q < C) A::src()[q] = (uint16_t)i;
            else *io.over = 1;
        }
        __syncthreads();
        const uint32_t m = *s_n < C ? *s_n : C;
        if (m == 0u) continue;   // uniform
        load_rows<W, BLOCK, true>(rows, io.keys, io.cin, m, A::src());
        inplace_pass<W, BLOCK, BITS, true, false>(m, g, pd_T, pd_ties, pd_key, rnorm, thr, has_id, ctl, nxt,
                                            ++*tag, io, st, near_hi, rows, push, [] {});
    }
    then();
    return true;
}

// CTAs per SM that the in-place merge's launch bound asks for.
template <int W, int BLOCK>
struct InOcc {
    static constexpr int kMin = BLOCK <= 128 ? 6 : BLOCK == 256 ? 4 : 2;
};

// Heads clear of an earlier use of the shared memory, or of a tag that comes
// round again (a barrier must follow).
template <int W, int BLOCK, int BITS>
__device__ __forceinline__ void inplace_init() {
    for (uint32_t i = threadIdx.x; i < (uint32_t)InPass<W, BITS>::S; i += BLOCK)
        InPass<W, BITS>::heads()[i] = 0u;
}

}  // namespace

}  // namespace itpp
