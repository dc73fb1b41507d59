// itpp_select.cu -- the top-M select of the partitioned merge (term bound,
// cap_policy 1; Sec. II.C "Practical considerations": keep the cap_M largest
// |c|, ties broken by ascending key).
//
// The values selected on are the 63-bit magnitude patterns b of the raw
// coefficients (monotone in |c|), offset by sel_lo: v = b - sel_lo.  Two ways
// to the threshold, which k_part_post chooses between:
//   fast   the merge compared every kept child with a range [lo, hi] around
//          the predicted threshold, counted the children above hi and listed
//          those inside, per CTA; the cap_M-th largest lies inside
//          (above < cap_M <= above + listed; sel_lo = lo);
//   full   otherwise (no range yet, the threshold moved outside it, a list
//          overflowed): k_sel_hist takes the first 13-bit digit over every
//          stored coefficient, with sel_lo = delta's pattern and the digit
//          scaled to the largest pattern the merge wrote (bits [sh, sh+13)
//          of v, sh = max(0, bitlen(hi - lo) - 13)), so the values spread over
//          thousands of bins; k_sel_gather lists the terms of the picked digit.
// k_sel_resolve then finishes on the list, one cooperative launch: digits of v
// and then of the keys of exact ties by all CTAs, with a barrier after each,
// until few enough values are left for the first CTA, which records the kept
// set as the predicate (threshold, tie key) that the next gate's reads apply,
// and the next gate's range.  In its place were 5 launches for the digits of
// v, 8 or 16 for those of a key and 3 more, a few microseconds each whether
// they had work or not: 117 us a gate at 2^23 terms (W = 1), 154 us at 2^22
// (W = 2).
#include <cstring>

#include "itpp_common.cuh"
#include "itpp_gate_body.cuh"
#include "itpp_launch.h"
#include "itpp_team.cuh"

namespace itpp {

namespace {

__device__ __forceinline__ int bit_length(unsigned long long v) {
    return v ? 64 - __clzll((long long)v) : 0;
}

// Shift of the full path's first digit: its top digit of v = b - lo, with
// the largest pattern the merge wrote as the top of the range.
__device__ __forceinline__ void sel_geometry(const DevCtl* ctl, unsigned long long lo,
                                             int* sh) {
    const unsigned long long hi = ctl->sel_hi;
    const int bits = bit_length(hi > lo ? hi - lo : 0ULL);
    *sh = bits > kSelBits ? bits - kSelBits : 0;
}

__device__ __forceinline__ unsigned long long sel_value(double c, unsigned long long lo) {
    const unsigned long long b = abs_bits(c);
    return b > lo ? b - lo : 0ULL;
}

// Inclusive scan of one value per thread over NT threads (s: NT slots).
template <int NT>
__device__ __forceinline__ unsigned long long scan_nt(unsigned long long v, unsigned long long* s) {
    const int t = threadIdx.x;
    s[t] = v;
    __syncthreads();
    for (int o = 1; o < NT; o <<= 1) {
        const unsigned long long a = t >= o ? s[t - o] : 0ULL;
        __syncthreads();
        s[t] += a;
        __syncthreads();
    }
    const unsigned long long r = s[t];
    __syncthreads();
    return r;
}

struct Pick {
    int digit;
    unsigned long long k_in;    // rank of the target inside the digit
    unsigned long long count;   // values in the digit
};

// The digit (in descending order) holding the k-th largest value, from a
// histogram of kSelBins counts; NT threads, result in *out (shared).
template <int NT>
__device__ __forceinline__ void pick_digit(const unsigned long long* hist, unsigned long long k,
                                           unsigned long long* s_part, Pick* out) {
    constexpr int PER = kSelBins / NT;
    const int t = threadIdx.x;
    if (t == 0) *out = Pick{0, 0, 0};
    // two passes over this thread's bins (sum, then find) instead of
    // holding PER counts in registers
    unsigned long long sum = 0;
    for (int j = 0; j < PER; ++j) sum += __ldcg(hist + kSelBins - 1 - PER * t - j);
    const unsigned long long incl = scan_nt<NT>(sum, s_part);
    unsigned long long run = incl - sum;
    if (run < k && k <= incl) {
        for (int j = 0; j < PER; ++j) {
            const unsigned long long hv = __ldcg(hist + kSelBins - 1 - PER * t - j);
            if (run < k && k <= run + hv) {
                out->digit = kSelBins - 1 - PER * t - j;
                out->k_in = k - run;
                out->count = hv;
            }
            run += hv;
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// 1. First digit (full path)
// ---------------------------------------------------------------------------
template <int W>
__global__ void __launch_bounds__(256, 4)
k_sel_hist(Bufs<W> B, Homes<W> H, DevCtl* ctl) {
    __shared__ unsigned int h[kSelBins];
    __shared__ unsigned long long s_part[256];
    __shared__ int s_last;
    __shared__ Pick s_pick;
    if (!ctl->sel_active || ctl->status || ctl->sel_fast) return;
    const unsigned long long lo = ctl->sel_lo;
    int sh;
    sel_geometry(ctl, lo, &sh);
    for (int b = threadIdx.x; b < kSelBins; b += blockDim.x) h[b] = 0u;
    __syncthreads();
    const StateRuns<W> rs = state_runs(ctl, B, H);
    // the coefficients' bit patterns, read as integers (no floating point)
    const unsigned long long* __restrict__ c =
        reinterpret_cast<const unsigned long long*>(rs.coef);
    auto count = [&](unsigned long long raw) {
        const unsigned long long b = raw & 0x7fffffffffffffffULL;   // |c| pattern
        if (!b) return;   // a zero is no term
        unsigned long long d = (b > lo ? b - lo : 0ULL) >> sh;
        if (d > (unsigned long long)(kSelBins - 1)) d = kSelBins - 1;   // not reached: hi is the max
        atomicAdd(&h[d], 1u);
    };
    if (rs.cnt) {
        for (uint32_t s = blockIdx.x; s < rs.P; s += gridDim.x) {
            const uint64_t off = (uint64_t)s * rs.R;
            const uint32_t cnt = rs.cnt[s] < rs.R ? rs.cnt[s] : (uint32_t)rs.R;
            for (uint32_t j = threadIdx.x; j < cnt; j += blockDim.x) count(__ldcs(c + off + j));
        }
    } else {
        // eight independent loads in flight per thread, then their counts
        const uint64_t n = rs.n;
        constexpr int U = 8;
        const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
        for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += U * stride) {
            unsigned long long v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t i = i0 + (uint64_t)u * stride;
                v[u] = i < n ? __ldcs(c + i) : 0ULL;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (i0 + (uint64_t)u * stride >= n) break;
                count(v[u]);
            }
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kSelBins; b += blockDim.x)
        if (h[b]) atomicAdd(&ctl->sel_hist[b], (unsigned long long)h[b]);
    // the last CTA to finish picks the digit (no CTA waits for another)
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&ctl->sel_done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    pick_digit<256>(ctl->sel_hist, ctl->sel_k, s_part, &s_pick);
    if (threadIdx.x == 0) {
        const Pick pk = s_pick;
        ctl->sel_prefix = (unsigned long long)pk.digit << sh;
        ctl->sel_mask = (unsigned long long)(kSelBins - 1) << sh;
        ctl->sel_k = pk.k_in;
        ctl->sel_top = sh;
        ctl->sel_done = 0u;
    }
    for (int b = threadIdx.x; b < kSelBins; b += blockDim.x) ctl->sel_hist[b] = 0ULL;
}

// ---------------------------------------------------------------------------
// 2. Candidates (full path): the terms of the threshold's first digit.  A
// warp claims room for its hits in the CTA's shared stage (one shared atomic
// per warp and load round that has hits, no block barrier in the loop); once
// the stage is full, later hits go straight to the global list.  The
// successful claims form a prefix of the stage (after the first claim that
// does not fit, every later one starts past the end), which the CTA copies
// out at the end with one global claim.  The order of the candidates is
// immaterial: every later pass histograms them and the ties are sorted by key.
// ---------------------------------------------------------------------------
constexpr int kStage = 3072;      // staged candidates per CTA (36 KB)
constexpr int kRangeShift0 = 45;  // the first candidate range: T +- about 1/128 of T

struct GatherStage {
    unsigned long long* st_v;
    uint32_t* st_i;
    unsigned int* s_claimed;
    unsigned int* s_staged;
};

// One round of up to 32 values per warp (every lane calls it).
__device__ __forceinline__ void gather_one(bool hit, unsigned long long x, uint64_t i,
                                           const GatherStage& gs, DevCtl* ctl,
                                           unsigned long long* cand_v, uint32_t* cand_idx,
                                           uint64_t cand_cap) {
    const unsigned int lane = threadIdx.x & 31u, lt = (1u << lane) - 1u;
    const unsigned int b = __ballot_sync(0xffffffffu, hit);
    if (!b) return;                                      // warp-uniform
    const int leader = __ffs(b) - 1;
    const unsigned int nb = __popc(b), r = __popc(b & lt);
    unsigned int q = 0u;
    if ((int)lane == leader) q = atomicAdd(gs.s_claimed, nb);
    q = __shfl_sync(0xffffffffu, q, leader);
    if (q + nb <= (unsigned int)kStage) {               // warp-uniform
        if (hit) {
            gs.st_v[q + r] = x;
            gs.st_i[q + r] = (uint32_t)i;
        }
        if ((int)lane == leader) atomicAdd(gs.s_staged, nb);
    } else {
        unsigned long long g = 0ULL;
        if ((int)lane == leader) g = atomicAdd(&ctl->sel_cand_n, (unsigned long long)nb);
        g = __shfl_sync(0xffffffffu, g, leader);
        if (hit) {
            if (g + r < cand_cap) {
                cand_v[g + r] = x;
                cand_idx[g + r] = (uint32_t)i;
            } else {
                set_status(ctl, ST_CAPACITY, 30);
            }
        }
    }
}

template <int W>
__global__ void __launch_bounds__(256)
k_sel_gather(Bufs<W> B, Homes<W> H, DevCtl* ctl, unsigned long long* cand_v,
             uint32_t* cand_idx, uint64_t cand_cap) {
    __shared__ unsigned long long st_v[kStage];
    __shared__ uint32_t st_i[kStage];
    __shared__ unsigned int s_claimed, s_staged;
    __shared__ unsigned long long s_base;
    if (!ctl->sel_active || ctl->status || ctl->sel_fast) return;
    const StateRuns<W> rs = state_runs(ctl, B, H);
    const unsigned long long lo = ctl->sel_lo;
    const unsigned long long prefix = ctl->sel_prefix, mask = ctl->sel_mask;
    const double* __restrict__ c = rs.coef;
    const GatherStage gs{st_v, st_i, &s_claimed, &s_staged};
    if (threadIdx.x == 0) {
        s_claimed = 0u;
        s_staged = 0u;
    }
    __syncthreads();
    // whole warps iterate together (the claims are warp-wide)
    if (rs.cnt) {
        for (uint32_t s = blockIdx.x; s < rs.P; s += gridDim.x) {
            const uint64_t off = (uint64_t)s * rs.R;
            const uint32_t cnt = rs.cnt[s] < rs.R ? rs.cnt[s] : (uint32_t)rs.R;
            for (uint32_t j0 = 0; j0 < cnt; j0 += blockDim.x) {
                const uint32_t j = j0 + threadIdx.x;
                const double v = j < cnt ? __ldcs(c + off + j) : 0.0;
                const unsigned long long x = sel_value(v, lo);
                gather_one(j < cnt && v != 0.0 && (x & mask) == prefix, x, off + j, gs, ctl, cand_v, cand_idx,
                           cand_cap);
            }
        }
    } else {
        const uint64_t n = rs.n;
        constexpr int U = 8;
        const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
        for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
             i0 - threadIdx.x < n; i0 += U * stride) {
            double v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t i = i0 + (uint64_t)u * stride;
                v[u] = i < n ? __ldcs(c + i) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t i = i0 + (uint64_t)u * stride;
                const unsigned long long x = sel_value(v[u], lo);
                gather_one(i < n && (x & mask) == prefix, x, i, gs, ctl, cand_v, cand_idx,
                           cand_cap);
            }
        }
    }
    __syncthreads();
    const unsigned int m = s_staged;
    if (threadIdx.x == 0) s_base = m ? atomicAdd(&ctl->sel_cand_n, (unsigned long long)m) : 0ULL;
    __syncthreads();
    const unsigned long long base = s_base;
    for (unsigned int j = threadIdx.x; j < m; j += blockDim.x) {
        if (base + j < cand_cap) {
            cand_v[base + j] = st_v[j];
            cand_idx[base + j] = st_i[j];
        } else {
            set_status(ctl, ST_CAPACITY, 30);
        }
    }
}

// ---------------------------------------------------------------------------
// 3. The rest of the select on the list: every CTA's candidates of the merge
// where they are (fast), or the gathered list (full).
// ---------------------------------------------------------------------------
struct SelPredict {   // the next gate's range
    uint64_t cap_M, cand_hi;
    long long* drift;
    int n_drift, gate;
    unsigned long long delta_bits;
};

// One thread: the kept set as the next gate's predicate, and its range.
template <int W>
__device__ __forceinline__ void sel_finish(DevCtl* ctl, unsigned long long T, bool all_ties,
                                           const PKey<W>& tk, const SelPredict& q) {
    const int cur = ctl->cur;
    ctl->pend = 1;
    ctl->pend_n = ctl->count[cur];
    ctl->pend_T = T;
    ctl->pend_all_ties = all_ties;
    for (int w = 0; w < 4; ++w) ctl->pend_tie_key[w] = 0ULL;
    if (!all_ties)
        for (int w = 0; w < W; ++w) {
            ctl->pend_tie_key[w] = tk.x[w];
            ctl->pend_tie_key[W + w] = tk.z[w];
        }
    ctl->count[cur] = q.cap_M;   // the logical term count
    ctl->stat_cands += ctl->sel_cand_n;
    const unsigned long long lo = ctl->sel_lo;
    ctl->stat_range = ctl->sel_fast ? ctl->sp_hi - ctl->sp_lo
                                    : (ctl->sel_hi > lo ? ctl->sel_hi - lo : 0ULL);
    // the next gate's candidate range: C +- 2^s in pattern units (a
    // relative width of about 2^(s-52)), narrower when the list ran long
    // or overflowed, wider when the threshold fell outside.  Its centre C:
    // this threshold moved by what the next gate's threshold moved in the
    // last layer (the schedule repeats every layer), or, without that,
    // carried into the next gate's scale (the next gate reads the state
    // rescaled by 1/c_I, rnorm of the buffer this gate wrote).
    const unsigned long long Tp = ctl->sp_tprev;
    const int gi = q.n_drift > 0 ? q.gate % q.n_drift : 0;
    const int gn = q.n_drift > 0 ? (q.gate + 1) % q.n_drift : 0;
    if (q.n_drift > 0) q.drift[gi] = Tp ? (long long)(T - Tp) : 0LL;
    ctl->sp_tprev = T;
    int sft = ctl->sp_shift ? ctl->sp_shift : kRangeShift0;
    switch (ctl->sel_fast ? 0 : ctl->sp_reason) {
        case 0: if (ctl->sel_cand_n > q.cand_hi) sft -= 1; break;
        case 1: sft = kRangeShift0; break;
        case 2: sft -= 2; break;
        default: sft += 1; break;
    }
    sft = sft < 8 ? 8 : (sft > kRangeShiftMax ? kRangeShiftMax : sft);
    ctl->sp_shift = sft;
    const long long dn = q.n_drift > 0 ? q.drift[gn] : 0LL;
    unsigned long long C;
    if (dn != 0LL) {
        const long long c = (long long)T + dn;
        C = c > 0 ? (unsigned long long)c : 0ULL;
    } else {
        C = abs_pattern(__dmul_rn(__longlong_as_double((long long)T), ctl->rnorm[cur]));
    }
    const SelRange r = sel_range(C, sft, q.delta_bits);
    ctl->sp_thr = r.thr;
    ctl->sp_lo = r.thr + 1ULL;
    ctl->sp_hi = r.hi;
    ctl->sel_active = 0;
}

// CTAs of the launch per SM: two read a list of a few hundred thousand values
// in a few rounds; a barrier grows with every CTA.
constexpr int kResolvePerSm = 2;

template <int W>
__global__ void __launch_bounds__(kBlock, kResolvePerSm)
k_sel_resolve(Bufs<W> B, Homes<W> H, DevCtl* ctl, CandRegions cr, unsigned long long* cand_v,
              uint32_t* cand_idx, PKey<W>* ties, SelPredict q) {
    __shared__ __align__(16) unsigned char s_scratch[kScratch];
    __shared__ uint32_t s_off[1024];
    __shared__ uint32_t s_scan[kBlock / 32];
    __shared__ PickOut s_pick;
    uint32_t* s_hist = reinterpret_cast<uint32_t*>(s_scratch);
    if (!ctl->sel_active) return;
    const bool first = blockIdx.x == 0;
    if (ctl->status) {
        if (first && threadIdx.x == 0) ctl->sel_active = 0;
        return;
    }
    const uint64_t n = ctl->sel_cand_n;
    // few values: the first CTA alone, among them all
    if (!first && n <= kOneCta) return;
    const bool fast = ctl->sel_fast != 0;
    const unsigned long long lo = ctl->sel_lo;
    unsigned long long prefix = ctl->sel_prefix, mask = ctl->sel_mask, rank = ctl->sel_k;
    int top = ctl->sel_top;
    TeamOf<SelTeam> team{&ctl->sel, blockIdx.x, gridDim.x, 0u, 0u};
    const PKey<W>* keys = state_runs(ctl, B, H).keys;
    const unsigned long long* sv = fast ? cr.v : cand_v;
    const uint32_t* si = fast ? cr.idx : cand_idx;
    uint32_t nreg = 0;
    if (fast) {   // where each CTA's candidates start
        nreg = ctl->cand_regions < 1024u ? ctl->cand_regions : 1024u;
        uint32_t c[4], sum = 0, tot;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t r = threadIdx.x * 4u + u;
            c[u] = r < nreg ? cr.cnt[r] : 0u;
            sum += c[u];
        }
        uint32_t at = block_exclusive_scan<kBlock>(sum, &tot, s_scan);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            s_off[threadIdx.x * 4u + u] = at;
            at += c[u];
        }
        __syncthreads();
    }
    // place of the j-th value (j < n)
    auto place = [&](uint64_t j) -> uint64_t {
        if (!fast) return j;
        uint32_t r = 0;   // the last region that starts at or before j
#pragma unroll
        for (uint32_t b = 512u; b > 0u; b >>= 1)
            if (s_off[r + b] <= (uint32_t)j) r += b;
        if (r >= nreg) r = nreg - 1u;   // (empty ones at the end start at n)
        return (uint64_t)r * cr.region + (j - s_off[r]);
    };
    const uint64_t tid = (uint64_t)blockIdx.x * kBlock + threadIdx.x;
    const uint64_t all = (uint64_t)(n <= kOneCta ? 1u : gridDim.x) * kBlock;
    // f(value, place) for every value that matches, its loads four at a time
    auto each = [&](auto&& f) {
        constexpr int U = 4;
        for (uint64_t j0 = tid; j0 < n; j0 += U * all) {
            uint64_t at[U];
            unsigned long long v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t j = j0 + u * all;
                at[u] = j < n ? place(j) : 0ULL;
                v[u] = j < n ? __ldcg(sv + at[u]) : ~prefix;
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j0 + u * all < n && (v[u] & mask) == prefix) f(v[u], at[u]);
        }
    };
    uint64_t cnt = n;
    int koff = 0;          // key bits fixed
    uint64_t kpre[2 * W];
#pragma unroll
    for (int w = 0; w < 2 * W; ++w) kpre[w] = 0;
    auto key_matches = [&](const PKey<W>& key) {
        const int full = koff >> 6, r = koff & 63;
        bool ok = true;
#pragma unroll
        for (int w = 0; w < 2 * W; ++w) {
            const uint64_t word = w < W ? key.x[w] : key.z[w - W];
            if (w < full) ok = ok && word == kpre[w];
            else if (w == full && r) ok = ok && (word >> (64 - r)) == (kpre[w] >> (64 - r));
        }
        return ok;
    };
    if (n > kOneCta) {
        for (int hb = 0; cnt > kOneCta; hb = (hb + 1) % 3) {
            const bool by_key = top == 0;
            if (by_key && (rank == cnt && koff == 0)) break;   // every tie is kept
            if (koff >= 128 * W) break;                        // (keys are distinct)
            for (int b = threadIdx.x; b < kBins; b += kBlock) s_hist[b] = 0u;
            __syncthreads();
            const int wd = by_key ? (64 - (koff & 63) < kDigit ? 64 - (koff & 63) : kDigit)
                                  : (top > kDigit ? kDigit : top);
            if (!by_key) {
                const int shift = top - wd;
                each([&](unsigned long long v, uint64_t) {
                    atomicAdd(&s_hist[(uint32_t)(v >> shift) & ((1u << wd) - 1u)], 1u);
                });
            } else {
                each([&](unsigned long long, uint64_t at) {
                    const PKey<W> key = load_key_stream(keys + __ldcg(si + at));
                    if (key_matches(key)) atomicAdd(&s_hist[key_digit(key, koff, wd)], 1u);
                });
            }
            __syncthreads();
            for (int b = threadIdx.x; b < kBins; b += kBlock)
                if (s_hist[b]) atomicAdd(&ctl->sel.hist[hb][b], s_hist[b]);
            if (!team_barrier(team, ctl)) return;
            for (int b = threadIdx.x; b < kBins; b += kBlock) {
                s_hist[b] = __ldcg(&ctl->sel.hist[hb][b]);
                if (first) ctl->sel.hist[(hb + 2) % 3][b] = 0u;   // read before this barrier
            }
            if (threadIdx.x == 0) s_pick = PickOut{0u, 1u, 0u};
            __syncthreads();
            if (by_key) pick_bin<false>(s_hist, (uint32_t)rank, s_scan, &s_pick);
            else pick_bin<true>(s_hist, (uint32_t)rank, s_scan, &s_pick);
            const PickOut o = s_pick;
            __syncthreads();
            rank = o.k_in;
            cnt = o.count;
            if (by_key) {
                const int w = koff >> 6, in = koff & 63;
#pragma unroll
                for (int u = 0; u < 2 * W; ++u)
                    if (u == w) kpre[u] |= (uint64_t)o.digit << (64 - in - wd);
                koff += wd;
            } else {
                top -= wd;
                prefix |= (unsigned long long)o.digit << top;
                mask |= (unsigned long long)((1u << wd) - 1u) << top;
            }
        }
    }
    if (cnt > kOneCta) {   // a long class of ties, all kept
        if (first && threadIdx.x == 0) {
            const PKey<W> none{};
            sel_finish(ctl, prefix + lo, true, none, q);
        }
        return;
    }
    // the values left, for the first CTA
    unsigned long long* lv = cand_v;
    uint32_t* li = cand_idx;
    if (!fast && n > kOneCta) {   // the merge's lists are free
        lv = cr.v;
        li = cr.idx;
    }
    if (fast || n > kOneCta) {
        each([&](unsigned long long v, uint64_t at) {
            const uint32_t idx = __ldcg(si + at);
            if (koff && !key_matches(load_key_stream(keys + idx))) return;
            const uint32_t p = atomicAdd(&ctl->sel.list_n, 1u);
            if (p < kOneCta) {
                lv[p] = v;
                li[p] = idx;
            }
        });
        if (n > kOneCta) {
            team_arrive(team);
            if (!first) return;
            if (!team_wait(team, ctl)) return;
        } else {
            __syncthreads();
        }
        cnt = __ldcg(&ctl->sel.list_n);
        if (cnt > kOneCta) cnt = kOneCta;
    }
    PKey<W> tk{};
    const SelOut so = select_list<W>(s_scratch, lv, li, cnt, rank, prefix, mask, top, keys, ties,
                                     &tk, ctl, koff > 0);
    if (threadIdx.x == 0) {
        if (ctl->status) ctl->sel_active = 0;
        else sel_finish(ctl, so.v + lo, so.all_ties != 0, tk, q);
    }
}

template <int W>
static Bufs<W> sel_bufs(const DeviceState& s) {
    Bufs<W> b;
    for (int i = 0; i < 2; ++i) {
        b.k[i] = reinterpret_cast<PKey<W>*>(s.keys[i]);
        b.c[i] = s.coef[i];
    }
    return b;
}

// The candidate list and the tie list in the merge table's memory (free on
// this path): v and idx of up to cand_cap candidates, then the tie keys.
template <int W>
struct SelScratch {
    unsigned long long* cand_v;
    uint32_t* cand_idx;
    uint64_t cand_cap;
    PKey<W>* ties;
    uint64_t tie_cap;
};

template <int W>
static SelScratch<W> sel_scratch(const DeviceState& s) {
    SelScratch<W> r;
    const uint64_t bytes = s.table_slots * sizeof(Slot<W>);
    char* base = static_cast<char*>(s.table);
    uint64_t cc = bytes / (12 + sizeof(PKey<W>));
    if (cc > s.buf_cap) cc = s.buf_cap;
    r.cand_cap = cc;
    r.cand_v = reinterpret_cast<unsigned long long*>(base);
    r.cand_idx = reinterpret_cast<uint32_t*>(base + cc * 8);
    const uint64_t toff = (cc * 12 + 255) / 256 * 256;
    r.ties = reinterpret_cast<PKey<W>*>(base + toff);
    r.tie_cap = (bytes - toff) / sizeof(PKey<W>);
    return r;
}

template <int W>
static cudaError_t select_w(const DeviceState& s, cudaStream_t st, int gate) {
    unsigned long long lo;
    std::memcpy(&lo, &s.delta, sizeof lo);   // delta >= +0: its pattern bounds every kept |c|
    const SelScratch<W> sc = sel_scratch<W>(s);
    const Bufs<W> B = sel_bufs<W>(s);
    Homes<W> H;
    H.kp = reinterpret_cast<PKey<W>*>(s.part_keys);
    H.cp = s.part_coef;
    H.cnt = s.part_cursor;
    H.part_max = s.part_max;
    H.cap = 0;
    k_sel_hist<W><<<s.num_sms * 4, 256, 0, st>>>(B, H, s.ctl);
    k_sel_gather<W><<<s.num_sms * 4, 256, 0, st>>>(B, H, s.ctl, sc.cand_v, sc.cand_idx,
                                                   sc.cand_cap);
    SelPredict q{s.cap_M, s.cand_hi, s.sp_drift, s.sp_drift ? s.layer_gates : 0, gate, lo};
    CandRegions cr = s.cand;
    DevCtl* ctl = s.ctl;
    void* args[8] = {const_cast<Bufs<W>*>(&B), &H, &ctl, &cr, const_cast<unsigned long long**>(&sc.cand_v),
                     const_cast<uint32_t**>(&sc.cand_idx), const_cast<PKey<W>**>(&sc.ties), &q};
    cudaError_t e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_sel_resolve<W>),
                                                dim3(s.num_sms * kResolvePerSm), dim3(kBlock),
                                                args, 0, st);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_select_deferred(const DeviceState& s, cudaStream_t st, int gate) {
    return s.W == 1 ? select_w<1>(s, st, gate) : select_w<2>(s, st, gate);
}

uint64_t select_list_cap(const DeviceState& s) {
    return s.W == 1 ? sel_scratch<1>(s).cand_cap : sel_scratch<2>(s).cand_cap;
}

}  // namespace itpp
