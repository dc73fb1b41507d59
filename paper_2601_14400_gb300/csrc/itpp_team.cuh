// itpp_team.cuh -- what a persistent kernel over many gates is made of: a team
// of CTAs that are all resident, its barrier in global memory, and the select
// by one CTA among a list of candidates.
//
// Every wait is bounded; a team that gives up stores the error and leaves.
#pragma once

#include "itpp_common.cuh"
#include "itpp_gate_body.cuh"

namespace itpp {

constexpr int kBlock = 256;
constexpr uint32_t kFinal = 128;                  // values ranked one per thread
constexpr size_t kScratch = 16384;                // shared scratch of a select
constexpr uint32_t kOneCta = 4096;                // candidates one CTA selects among

// ---------------------------------------------------------------------------
// Arrivals
// ---------------------------------------------------------------------------
template <class S>
struct TeamOf {
    S* rs;
    uint32_t rank, size;
    uint32_t target;   // arrivals that complete the current phase
    uint32_t seq;      // publications so far
};

// One thread waits for *p to reach v (in wrapping order); false after about
// ten seconds here, or when another wait of the team ran out.
__device__ __forceinline__ bool wait_for(const unsigned int* p, uint32_t v, TeamHead* head,
                                         DevCtl* ctl) {
    for (uint32_t it = 0;; ++it) {
        uint32_t x;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(p) : "memory");
        if ((int32_t)(x - v) >= 0) return true;
        if (it > 2048u) {
            __nanosleep(it > 16384u ? 1000u : 64u);
            if (it > 10000000u || *(volatile unsigned int*)&head->dead) {
                set_status(ctl, ST_TIMEOUT, 60);
                *(volatile unsigned int*)&head->dead = 1u;
                return false;
            }
        }
    }
}

// This CTA's writes so far are done; every thread calls it.
template <class S>
__device__ __forceinline__ void team_arrive(TeamOf<S>& t) {
    t.target += t.size;
    __syncthreads();   // the release below covers every thread's writes before it
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(&t.rs->head.bar) : "memory");
    }
}

// Wait until every CTA of the team has arrived; every thread calls it.  False:
// the wait ran out and the caller leaves the kernel.
template <class S>
__device__ __forceinline__ bool team_wait(const TeamOf<S>& t, DevCtl* ctl) {
    __shared__ int s_ok;
    if (threadIdx.x == 0) {
        s_ok = wait_for(&t.rs->head.bar, t.target, &t.rs->head, ctl);
    }
    __syncthreads();
    const int ok = s_ok;
    __syncthreads();
    return ok != 0;
}

template <class S>
__device__ __forceinline__ bool team_barrier(TeamOf<S>& t, DevCtl* ctl) {
    team_arrive(t);
    return team_wait(t, ctl);
}

// ---------------------------------------------------------------------------
// Select among a list of n (v, idx): the k-th largest v (rank from 1), ties
// by ascending key.  One CTA; kScratch bytes of shared scratch.
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

// Bits [off, off + wd) of a key, counted from the top of word 0 in comparison
// order, within one word.
template <int W>
__device__ __forceinline__ uint32_t key_digit(const PKey<W>& k, int off, int wd) {
    const int w = off >> 6, in = off & 63;
    uint64_t word = 0;
#pragma unroll
    for (int j = 0; j < 2 * W; ++j) if (j == w) word = j < W ? k.x[j] : k.z[j - W];
    return (uint32_t)((word >> (64 - in - wd)) & ((1ULL << wd) - 1ULL));
}

// prefix, top: the bits of v from `top` up already agree with prefix.  more:
// there are further ties beyond the list, all dropped.  Every
// thread calls it; *tk receives the largest kept key at the threshold when
// some of its ties are dropped.  ties: global scratch for a long list of equal
// values.  What bounds it is latency, a pass over a few thousand candidates
// being about a microsecond: so the values are read once (up to 4,096 stay in
// registers), a digit usually leaves few enough to rank by counting, and keys
// are read for ties alone.
template <int W>
__device__ SelOut select_list(unsigned char* scratch, const unsigned long long* gv, const uint32_t* gidx, uint64_t n,
                              uint64_t k, unsigned long long prefix, unsigned long long mask,
                              int top, const PKey<W>* keys, PKey<W>* ties, PKey<W>* tk,
                              DevCtl* ctl, bool more = false) {
    constexpr int kReg = (int)kOneCta / kBlock;
    constexpr uint32_t kTieMax = 512 / W;   // keys held in shared memory
    uint32_t* h = reinterpret_cast<uint32_t*>(scratch);                    // kBins
    PKey<W>* sk = reinterpret_cast<PKey<W>*>(h + kBins);                    // kTieMax
    unsigned long long* fv = reinterpret_cast<unsigned long long*>(sk);     // kFinal
    uint32_t* fi = reinterpret_cast<uint32_t*>(fv + kFinal);
    PKey<W>* fk = reinterpret_cast<PKey<W>*>(fi + kFinal);
    static_assert(kBins * 4 + kTieMax * sizeof(PKey<W>) <= kScratch, "scratch");
    static_assert(kFinal * (12 + sizeof(PKey<W>)) <= kTieMax * sizeof(PKey<W>), "scratch");
    __shared__ uint32_t s_w[kBlock / 32], s_n, s_gt, s_eq;
    __shared__ PickOut s_pick;
    __shared__ unsigned long long s_T;
    __shared__ uint64_t s_tk[4];
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned int lt = (1u << lane) - 1u;
    const bool held = n <= (uint64_t)(kReg * kBlock);
    unsigned long long rv[kReg];
#pragma unroll
    for (int u = 0; u < kReg; ++u) {
        const uint32_t j = u * kBlock + threadIdx.x;
        rv[u] = held && j < n ? __ldcg(gv + j) : ~prefix;
    }
    uint64_t cnt = n;          // entries that match the prefix
    uint32_t rank = (uint32_t)k;
    while (cnt > kFinal && top > 0) {
        const int shift = top > kDigit ? top - kDigit : 0;
        const uint32_t dmask = (1u << (top - shift)) - 1u;
        for (int b = threadIdx.x; b < kBins; b += kBlock) h[b] = 0u;
        __syncthreads();
        if (held) {
#pragma unroll
            for (int u = 0; u < kReg; ++u)
                if (u * kBlock + threadIdx.x < n && (rv[u] & mask) == prefix)
                    atomicAdd(&h[(uint32_t)(rv[u] >> shift) & dmask], 1u);
        } else {
            for (uint64_t j = threadIdx.x; j < n; j += kBlock) {
                const unsigned long long v = __ldcg(gv + j);
                if ((v & mask) == prefix) atomicAdd(&h[(uint32_t)(v >> shift) & dmask], 1u);
            }
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
    SelOut o;
    o.v = prefix;
    o.all_ties = 1;
    if (threadIdx.x == 0) s_n = s_gt = s_eq = 0u;
    __syncthreads();
    if (cnt > kFinal && rank == cnt && !more) return o;   // a class of equal values, all kept
    if (cnt <= kFinal) {
        // the entries left: value and place
        auto take = [&](uint64_t j, unsigned long long v) {
            if ((v & mask) == prefix) {
                const uint32_t q = atomicAdd(&s_n, 1u);
                if (q < kFinal) {
                    fv[q] = v;
                    fi[q] = (uint32_t)j;
                }
            }
        };
        if (held) {
#pragma unroll
            for (int u = 0; u < kReg; ++u)
                if (u * kBlock + threadIdx.x < n) take(u * kBlock + threadIdx.x, rv[u]);
        } else {
            for (uint64_t j = threadIdx.x; j < n; j += kBlock) take(j, __ldcg(gv + j));
        }
        __syncthreads();
        const uint32_t m = s_n;
        if (m > kFinal || rank < 1u || rank > m) {   // uniform; the list agrees with the counts
            if (threadIdx.x == 0) set_status(ctl, ST_STATE, 61);
            __syncthreads();
            return o;
        }
        uint32_t gt = 0, eq = 0;
        unsigned long long v = 0;
        if (threadIdx.x < m) {
            v = fv[threadIdx.x];
#pragma unroll 4
            for (uint32_t j = 0; j < m; ++j) {
                const unsigned long long u = fv[j];
                gt += u > v ? 1u : 0u;
                eq += u == v ? 1u : 0u;
            }
            if (gt < rank && rank <= gt + eq) {   // the same values from every tie
                s_T = v;
                s_gt = gt;
                s_eq = eq;
            }
        }
        __syncthreads();
        const uint32_t need = rank - s_gt, ne = s_eq;
        o.v = s_T;
        o.all_ties = need == ne && !more;
        if (o.all_ties) {
            __syncthreads();
            return o;
        }
        // some ties are dropped: the need-th smallest key among them
        if (threadIdx.x == 0) s_n = 0u;
        __syncthreads();
        if (threadIdx.x < m && v == o.v) {
            const PKey<W> key = load_key_stream(keys + __ldcg(gidx + fi[threadIdx.x]));
            fk[atomicAdd(&s_n, 1u)] = key;
        }
        __syncthreads();
        if (threadIdx.x < ne) {
            const PKey<W> key = fk[threadIdx.x];
            uint32_t before = 0;
            for (uint32_t j = 0; j < ne; ++j) before += key_less(fk[j], key) ? 1u : 0u;
            if (before == need - 1u) {
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    s_tk[w] = key.x[w];
                    s_tk[W + w] = key.z[w];
                }
            }
        }
    } else {
        // a long class of equal values of which some are dropped: the rank-th
        // smallest key, by key digits over a list of the keys (in shared
        // memory when it fits)
        o.all_ties = 0;
        const uint32_t nt = (uint32_t)cnt;
        const bool local = nt <= kTieMax;
        auto put = [&](uint64_t j, bool hit) {   // whole warps
            const unsigned int m = __ballot_sync(0xffffffffu, hit);
            if (!m) return;
            uint32_t q = 0;
            if (lane == 0) q = atomicAdd(&s_n, (uint32_t)__popc(m));
            q = __shfl_sync(0xffffffffu, q, 0) + __popc(m & lt);
            if (hit && q < nt) {
                const PKey<W> key = load_key_stream(keys + __ldcg(gidx + j));
                if (local) sk[q] = key;
                else ties[q] = key;
            }
        };
        if (held) {
#pragma unroll
            for (int u = 0; u < kReg; ++u) {
                const uint32_t j = u * kBlock + threadIdx.x;
                put(j, j < n && (rv[u] & mask) == prefix);
            }
        } else {
            for (uint64_t j0 = threadIdx.x & ~31u; j0 < n; j0 += kBlock)
                put(j0 + lane, j0 + lane < n && (__ldcg(gv + j0 + lane) & mask) == prefix);
        }
        __syncthreads();
        const PKey<W>* list = local ? sk : ties;
        uint64_t kpre[2 * W];   // key bits fixed so far
#pragma unroll
        for (int w = 0; w < 2 * W; ++w) kpre[w] = 0;
        int off = 0;
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
        uint32_t left = nt;
        while (left > 1u && off < 128 * W) {
            for (int b = threadIdx.x; b < kBins; b += kBlock) h[b] = 0u;
            __syncthreads();
            int wd = 64 - (off & 63) < kDigit ? 64 - (off & 63) : kDigit;
            for (uint32_t j = threadIdx.x; j < nt; j += kBlock) {
                const PKey<W> key = list[j];
                if (matches(key)) atomicAdd(&h[key_digit(key, off, wd)], 1u);
            }
            __syncthreads();
            pick_bin<false>(h, rank, s_w, &s_pick);
            const int w = off >> 6, in = off & 63;
#pragma unroll
            for (int v = 0; v < 2 * W; ++v)
                if (v == w) kpre[v] |= (uint64_t)s_pick.digit << (64 - in - wd);
            rank = s_pick.k_in;
            left = s_pick.count;
            off += wd;
            __syncthreads();
        }
        // the one key that matches (keys are distinct)
        for (uint32_t j = threadIdx.x; j < nt; j += kBlock) {
            const PKey<W> key = list[j];
            if (matches(key)) {
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    s_tk[w] = key.x[w];
                    s_tk[W + w] = key.z[w];
                }
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < W; ++w) { tk->x[w] = s_tk[w]; tk->z[w] = s_tk[W + w]; }
    __syncthreads();
    return o;
}

}  // namespace itpp
