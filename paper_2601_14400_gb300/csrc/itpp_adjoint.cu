// itpp_adjoint.cu -- gradients of a propagated expectation value with respect
// to every gate coefficient alpha_k, by a reverse sweep over the steps with
// the kept support of every step frozen (the paper has no such step; this is
// the linear algebra of Eq. (ITPP_PropRules) and the per-step normalisation).
//
// With u_s the normalised state after step s (support S_s), D_s its identity
// coefficient before normalisation and f = sum_j w_j u_L[P_j]:
//   nu_s[K] = mu_s[K] / D_s (K != I),  nu_s[I] = -sum_{K != I} mu_s[K] u_s[K] / D_s
//   mu_{s-1}[P] = nu_s[P]                                ({P,Q} = 0)
//               = cosh nu_s[P] + s (-sinh) nu_s[Q P]    ([P,Q] = 0)
//   df/dtheta_s = sum_{[P,Q]=0} u_{s-1}[P] (sinh nu_s[P] - s cosh nu_s[Q P])
// where mu_s = df/du_s, nu_s = 0 outside S_s and theta_s = alpha_k dtau.
// S_s is the kept set of step s: after the threshold and, with the top-M
// bound, after the select.
//
// Memory: the forward saves a snapshot every ckpt_every layers; each segment
// is recomputed from its snapshot into an arena that keeps every step's state
// and, per input term, the output positions of its children (itself, a new
// partner string, or the partner that was present).  The reverse sweep then
// gathers through those positions -- no atomics, fixed-order reductions.
// Output order inside a recomputed segment need not match the first forward,
// so the adjoint vector is carried across a segment boundary by key (a
// table lookup into the snapshot's keys).
#include <cmath>
#include <cstring>
#include <vector>

#include "itpp.h"
#include "itpp_common.cuh"
#include "itpp_ctx.h"
#include "itpp_gate_body.cuh"
#include "itpp_launch.h"
#include "itpp_team.cuh"

using namespace itpp;

namespace {

constexpr int kRB = 256;      // reduction block
constexpr int kAdjLoad = 25;  // table load: most probes end at the first slot
constexpr int kRGrid = 512;   // fixed reduction grid: deterministic partial order

template <int W>
GateArg<W> gate_arg_of(const HostGate& h) {
    GateArg<W> g;
    for (int w = 0; w < W; ++w) { g.qx[w] = h.qx[w]; g.qz[w] = h.qz[w]; }
    g.ch = h.ch;
    g.msh = h.msh;
    g.qyy = h.qyy;
    g.maxw = h.maxw;
    return g;
}

__device__ __forceinline__ double block_sum(double v, double* s) {
    s[threadIdx.x] = v;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) s[threadIdx.x] = __dadd_rn(s[threadIdx.x], s[threadIdx.x + o]);
        __syncthreads();
    }
    const double r = s[0];
    __syncthreads();
    return r;
}

__global__ void k_adj_log(const DevCtl* ctl, unsigned long long* log, int s) {
    if (threadIdx.x == 0) log[s] = ctl->status ? ~0ULL : ctl->count[ctl->cur];
}

// Snapshot of the current state: AoS keys and normalised coefficients.
template <int W>
__global__ void __launch_bounds__(256)
k_adj_snapshot(const PKey<W>* k0, const double* c0, const PKey<W>* k1, const double* c1,
               const DevCtl* ctl, PKey<W>* keys, double* coef) {
    const int cur = ctl->cur;
    const uint64_t n = live_count(ctl, cur);
    const double rn = ctl->rnorm[cur];
    const PKey<W>* ks = cur ? k1 : k0;
    const double* cs = cur ? c1 : c0;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const PKey<W> K = ks[i];
        keys[i] = K;
        coef[i] = normalised(cs[i], rn, key_is_zero(K));
    }
}

// One recomputed step: where its input, its kept output and its maps lie.
template <int W>
struct AdjStep {
    const PKey<W>* kin;
    const double* cin;
    PKey<W>* kout;
    double* cout;
    int *self_out, *emit_out, *part_src;   // [ci]
    int* cmap;                             // [2 ci]
    uint64_t ci, co;                       // terms in and kept
    GateArg<W> g;
    double sh, chd;
};

// Shared by the CTAs of a sweep; zero before its launch.
struct AdjShared {
    TeamHead head;
    unsigned int hist[3][kBins];
    unsigned int list_n[2];
    unsigned long long kept[2];
    int stop[2];
    unsigned long long T;
    uint64_t tk[4];
    int all_ties, pad;
};

template <int W>
struct AdjSweep {
    const AdjStep<W>* steps;
    int n_steps;
    PKey<W>* kpre;              // a step's output before the term bound
    double* cpre;
    DevCtl* ctl;
    Slot<W>* table;
    uint64_t slots;
    int probe_limit, cap_policy;
    double delta;
    unsigned long long cap_M;
    const unsigned long long* cnt0;   // terms of the first input
    double* rn;                       // [n_steps + 1]
    unsigned long long *id, *id_pre;  // [n_steps + 1] the identity's position
    AdjShared* sh;
    unsigned long long* cand_v;       // [2 terms] select: candidates
    uint32_t* cand_i;
    PKey<W>* ties;
};

// Recompute a segment's steps, recording the output positions, by one
// persistent launch.  A step is a few tens of microseconds of work at most;
// it was made of 35 launches (reset, table, merge, five radix passes over |c|
// and eight over the ties of two launches each, compaction), with four more in
// the reverse sweep: 273 us a step of both at 2^18 terms, nearly all of it
// between launches.  Persistent, they take 64 and 22 us.  Here a step is
//
//   merge      every input's children against the table, with a histogram of
//              |c| around the last threshold (512 bins an octave)
//   list       the values of the bin that holds the bound (more histograms
//              first where it is a long one)
//   select     the first CTA, among the list
//   compact    the kept terms, which enter the next step's table at once
//
// with a barrier after each.  What bounds it is latency, one tile a CTA: the
// merge 30 us (two lookups one after the other, histogram), compaction 22, the
// list and the select 11.
template <int W>
__global__ void __launch_bounds__(kBlock, 4) k_adj_recompute(const AdjSweep<W> a) {
    __shared__ __align__(16) unsigned char s_scratch[kScratch];
    __shared__ uint32_t s_scan[kBlock / 32];
    __shared__ unsigned long long s_base;
    __shared__ PickOut s_pick;
    uint32_t* s_hist = reinterpret_cast<uint32_t*>(s_scratch);
    DevCtl* ctl = a.ctl;
    AdjShared* sh = a.sh;
    TeamOf<AdjShared> team{sh, blockIdx.x, gridDim.x, 0u, 0u};
    const bool first = blockIdx.x == 0;
    const uint64_t tid = (uint64_t)blockIdx.x * kBlock + threadIdx.x;
    const uint64_t all = (uint64_t)gridDim.x * kBlock;
    const unsigned long long dbits = (unsigned long long)__double_as_longlong(a.delta);
    if (ctl->status) return;   // from an earlier segment: the same for all
    unsigned gen = ctl->gen;
    uint64_t n = *a.cnt0;
    double rnorm = a.rn[0];
    int probes = 0;
    if (n > a.steps[0].ci) n = a.steps[0].ci;
    {
        const AdjStep<W>& S = a.steps[0];
        const uint64_t mask = table_mask(n, a.slots, kAdjLoad);
        for (uint64_t i = tid; i < n; i += all)
            insert_one(S.kin, S.cin, i, ctl, a.table, mask, gen, S.g, a.probe_limit, &probes);
    }
    if (!team_barrier(team, ctl)) return;
    int hb = 0;                       // this pass's histogram
    unsigned long long tprev = 0ULL;  // the last threshold
    auto clear_hist = [&] {
        for (int b = threadIdx.x; b < kBins; b += kBlock) s_hist[b] = 0u;
        __syncthreads();
    };
    auto flush_hist = [&] {
        __syncthreads();
        for (int b = threadIdx.x; b < kBins; b += kBlock)
            if (s_hist[b]) atomicAdd(&sh->hist[hb][b], s_hist[b]);
    };
    for (int r = 1; r <= a.n_steps; ++r) {
        const AdjStep<W>& S = a.steps[r - 1];
        const int x = r & 1;   // this step's counters
        // bins of the first histogram: four octaves around the last threshold,
        // or 32 from the drop threshold up; what lies outside falls into the
        // first and the last
        unsigned long long base = tprev > (2ULL << 52) ? tprev - (2ULL << 52) : 0ULL;
        int shift = 43;
        if (!tprev) {
            base = dbits;
            shift = 46;
        }
        const bool may = a.cap_policy == 1 && 2 * n > a.cap_M;   // uniform
        auto bin_of = [&](unsigned long long p) {
            const unsigned long long d = p > base ? (p - base) >> shift : 0ULL;
            return d < (unsigned long long)kBins ? (uint32_t)d : (uint32_t)kBins - 1u;
        };
        if (may) clear_hist();
        {
            const uint64_t mask = table_mask(n, a.slots, kAdjLoad);
            const GlobalLookup<W, true> lk{a.table, mask, gen, a.probe_limit, ctl, &probes};
            const StepMaps maps{S.self_out, S.emit_out, S.part_src, a.id_pre + r};
            auto sink = [&](double c) {
                if (may) atomicAdd(&s_hist[bin_of(abs_pattern(c))], 1u);
            };
            const uint64_t tiles = (n + 2 * kBlock - 1) / (2 * kBlock);
            for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x)
                gate_tile<W, kBlock, 2, true>(t, n, S.kin, S.cin, a.kpre, a.cpre, ctl, x ^ 1, lk,
                                              S.g, rnorm, dbits, 2 * S.ci, s_scan, &s_base, maps,
                                              sink);
        }
        if (may) flush_hist();
        if (!team_barrier(team, ctl)) return;
        unsigned long long np = __ldcg(&ctl->count[x]);
        if (np > 2 * S.ci) np = 2 * S.ci;
        const double norm = __ldcg(&ctl->norm[x]);
        const double rnew = __ddiv_rn(1.0, norm);
        const bool active = may && np > a.cap_M;
        const unsigned gnext = gen + 1u;
        if (first && threadIdx.x == 0) {
            if (abs_pattern(norm) >= 0x7ff0000000000000ULL) set_status(ctl, ST_STATE, 5);
            if (gnext == 0u) set_status(ctl, ST_STATE, 1);   // generation counter wrapped
            if (a.cap_policy == 0 && a.cap_M && np > a.cap_M) set_status(ctl, ST_CAPACITY, 1);
            ctl->count[x ^ 1] = 0ULL;   // the next step's; read last in the step before
            sh->kept[x ^ 1] = 0ULL;
            sh->list_n[x ^ 1] = 0u;
            a.rn[r] = rnew;
        }
        unsigned long long T = 0ULL;
        bool all_ties = true;
        PKey<W> tk{};
        if (active) {
            // the bin that holds the cap_M-th largest value, narrowed until
            // one CTA can select in it
            unsigned long long lo = 0ULL, hi = 1ULL << 63, rank = a.cap_M;
            for (int pass = 0; pass < 8; ++pass) {
                __syncthreads();
                for (int b = threadIdx.x; b < kBins; b += kBlock) {
                    s_hist[b] = __ldcg(&sh->hist[hb][b]);
                    if (first) sh->hist[(hb + 2) % 3][b] = 0u;   // read last before this barrier
                }
                if (threadIdx.x == 0) s_pick = PickOut{0u, 1u, 0u};
                __syncthreads();
                pick_bin<true>(s_hist, (uint32_t)rank, s_scan, &s_pick);
                const PickOut o = s_pick;
                const unsigned long long b0 = base + ((unsigned long long)o.digit << shift);
                if (o.digit + 1u < (uint32_t)kBins) hi = b0 + (1ULL << shift);
                if (o.digit > 0u) lo = b0;
                rank = o.k_in;
                if (o.count <= kOneCta || hi - lo <= 1ULL) break;   // uniform
                hb = (hb + 1) % 3;
                base = lo;
                const int bits = 64 - __clzll((long long)(hi - lo - 1ULL));
                shift = bits > kDigit ? bits - kDigit : 0;
                __syncthreads();
                clear_hist();
                for (uint64_t i = tid; i < np; i += all) {
                    const unsigned long long p = abs_pattern(__ldcg(a.cpre + i));
                    if (p >= lo && p < hi) atomicAdd(&s_hist[bin_of(p)], 1u);
                }
                flush_hist();
                if (!team_barrier(team, ctl)) return;
            }
            for (uint64_t t = blockIdx.x; t * kBlock < np; t += gridDim.x) {
                const uint64_t i = t * kBlock + threadIdx.x;
                const unsigned long long p = i < np ? abs_pattern(__ldcg(a.cpre + i)) : 0ULL;
                const bool in = i < np && p >= lo && p < hi;
                uint32_t tot;
                const uint32_t off = block_exclusive_scan<kBlock>(in ? 1u : 0u, &tot, s_scan);
                if (threadIdx.x == 0) s_base = tot ? atomicAdd(&sh->list_n[x], tot) : 0u;
                __syncthreads();
                if (in) {
                    a.cand_v[s_base + off] = p - lo;
                    a.cand_i[s_base + off] = (uint32_t)i;
                }
                __syncthreads();
            }
            if (!team_barrier(team, ctl)) return;
            if (first) {
                const unsigned long long span = hi - lo - 1ULL;
                const SelOut so = select_list<W>(
                    s_scratch, a.cand_v, a.cand_i, __ldcg(&sh->list_n[x]), rank, 0ULL, 0ULL,
                    span ? 64 - __clzll((long long)span) : 0, a.kpre, a.ties, &tk, ctl);
                if (threadIdx.x == 0) {
                    sh->T = lo + so.v;
                    sh->all_ties = so.all_ties;
                    for (int w = 0; w < W; ++w) { sh->tk[w] = tk.x[w]; sh->tk[W + w] = tk.z[w]; }
                }
            }
            if (!team_barrier(team, ctl)) return;
            T = __ldcg(&sh->T);
            all_ties = __ldcg(&sh->all_ties) != 0;
#pragma unroll
            for (int w = 0; w < W; ++w) { tk.x[w] = __ldcg(sh->tk + w); tk.z[w] = __ldcg(sh->tk + W + w); }
            tprev = T;
        } else if (first) {
            for (int b = threadIdx.x; b < kBins; b += kBlock) sh->hist[(hb + 2) % 3][b] = 0u;
        }
        hb = (hb + 1) % 3;
        // compaction; what commutes with the next gate enters its table
        uint64_t nn = active ? a.cap_M : np;
        if (nn > S.co) nn = S.co;
        const bool more = r < a.n_steps;
        const GateArg<W> gn = a.steps[more ? r : r - 1].g;
        const uint64_t mask = table_mask(nn, a.slots, kAdjLoad);
        PKey<W>* kout = S.kout;
        double* cout = S.cout;
        int* cmap = S.cmap;
        const uint64_t co = S.co;
        constexpr int U = 2;   // terms per thread, their table probes in flight together
        for (uint64_t t = blockIdx.x; t * (U * kBlock) < np; t += gridDim.x) {
            PKey<W> K[U];
            double c[U];
            uint32_t keep = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t i = (t * U + u) * kBlock + threadIdx.x;
                K[u] = PKey<W>{};
                c[u] = 0;
                if (i < np) {
                    K[u] = load_key_stream(a.kpre + i);
                    c[u] = __ldcg(a.cpre + i);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t i = (t * U + u) * kBlock + threadIdx.x;
                if (i < np) {
                    const bool k = !active || cap_keep(K[u], c[u], T, all_ties, tk);
                    if (key_is_zero(K[u]) && !k) set_status(ctl, ST_TRACE_ZERO, 32);
                    keep |= k ? 1u << u : 0u;
                }
            }
            uint32_t tot;
            uint32_t off = block_exclusive_scan<kBlock>(__popc(keep), &tot, s_scan);
            if (threadIdx.x == 0)
                s_base = tot ? atomicAdd(&sh->kept[x], (unsigned long long)tot) : 0ULL;
            __syncthreads();
            uint64_t pos[U], h[U];
            unsigned old[U];
            bool in[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t i = (t * U + u) * kBlock + threadIdx.x;
                bool k = (keep >> u) & 1u;
                pos[u] = s_base + off;
                off += k ? 1u : 0u;
                if (k && pos[u] >= co) {   // the first forward's support is another
                    set_status(ctl, ST_STATE, 33);
                    k = false;
                }
                if (i < np) cmap[i] = k ? (int)pos[u] : -1;
                if (k) {
                    kout[pos[u]] = K[u];
                    cout[pos[u]] = c[u];
                    if (key_is_zero(K[u])) a.id[r] = pos[u];
                }
                in[u] = k && more && commutes(K[u], gn);
                h[u] = key_hash(K[u]) & mask;
                // generations only grow: the slot is ours unless it was this one's
                if (in[u]) old[u] = atomicMax(&a.table[h[u]].tag, gnext);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (!in[u]) continue;
                int p = 0;
                while (old[u] == gnext && ++p < a.probe_limit) {
                    h[u] = (h[u] + 1) & mask;
                    old[u] = atomicMax(&a.table[h[u]].tag, gnext);
                }
                if (old[u] == gnext) {
                    set_status(ctl, ST_HASH_PROBE, 1);
                    continue;
                }
                Slot<W>* sl = a.table + h[u];
#pragma unroll
                for (int w = 0; w < W; ++w) { sl->x[w] = K[u].x[w]; sl->z[w] = K[u].z[w]; }
                sl->c = c[u];
                sl->idx = (uint32_t)pos[u];
            }
            __syncthreads();
        }
        if (first && threadIdx.x == 0) sh->stop[x] = *(volatile int*)&ctl->status;
        if (!team_barrier(team, ctl)) return;
        if (__ldcg(&sh->stop[x])) return;   // uniform
        gen = gnext;
        n = nn;
        rnorm = rnew;
    }
    if (first && threadIdx.x == 0) ctl->gen = gen;
}

// Seed: mu[i] = sum of the weights of the observable strings equal to key i.
template <int W>
__global__ void __launch_bounds__(256)
k_adj_seed(const PKey<W>* keys, uint64_t n, const uint64_t* ox, const uint64_t* oz,
           const double* wsum, const int* tab, int tsize, double* mu) {
    const uint64_t mask = (uint64_t)tsize - 1;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const PKey<W> K = keys[i];
        double v = 0.0;
        uint64_t h = key_hash(K) & mask;
        for (int p = 0; p < tsize; ++p) {
            const int e = tab[h];
            if (e < 0) break;
            PKey<W> o;
            for (int w = 0; w < W; ++w) { o.x[w] = ox[(size_t)e * W + w]; o.z[w] = oz[(size_t)e * W + w]; }
            if (key_eq(o, K)) { v = wsum[e]; break; }
            h = (h + 1) & mask;
        }
        mu[i] = v;
    }
}

// Per distinct observable string (first occurrence), the sum of its weights.
__global__ void k_adj_wsum(const int* first, const double* w, int m, double* wsum) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    for (int j = 0; j < m; ++j) wsum[j] = 0.0;
    for (int j = 0; j < m; ++j) wsum[first[j]] = __dadd_rn(wsum[first[j]], w[j]);
}

// The reverse sweep over a segment by one persistent launch: mu_{s-1} from
// nu_s through the recorded output positions, with the partial sums of
// df/dtheta_s, and of the next step's dot = sum_{j != I} mu[j] u[j] (nu_I =
// -dot / D) from the values just made.  One barrier a step, where
// four launches were.
// The grid and so the order of the sums are fixed by the sizes.
template <int W>
__global__ void __launch_bounds__(kBlock, 4)
k_adj_reverse(const AdjSweep<W> a, double* mu_out, double* mu_in, double* partials, double* gstep) {
    if (a.ctl->status) return;   // maps may be missing
    __shared__ double s[kBlock];
    TeamOf<AdjShared> team{a.sh, blockIdx.x, gridDim.x, 0u, 0u};
    const int G = (int)gridDim.x;
    double* p_dot = partials;           // [2][G]
    double* p_grad = partials + 2 * G;  // [2][G]
    const uint64_t tid = (uint64_t)blockIdx.x * kBlock + threadIdx.x;
    const uint64_t all = (uint64_t)G * kBlock;
    auto sum_of = [&](const double* p) {
        double acc = 0.0;
        for (int i = threadIdx.x; i < G; i += kBlock) acc = __dadd_rn(acc, __ldcg(p + i));
        return block_sum(acc, s);
    };
    const int R = a.n_steps;
    {
        const AdjStep<W>& S = a.steps[R - 1];
        const unsigned long long id = a.id[R];
        const double rr = a.rn[R];
        double acc = 0.0;
        for (uint64_t j = tid; j < S.co; j += all)
            if (j != id) acc = __dadd_rn(acc, __dmul_rn(mu_out[j], __dmul_rn(S.cout[j], rr)));
        const double b = block_sum(acc, s);
        if (threadIdx.x == 0) p_dot[(R & 1) * G + blockIdx.x] = b;
    }
    if (!team_barrier(team, a.ctl)) return;
    for (int r = R; r >= 1; --r) {
        const AdjStep<W> S = a.steps[r - 1];
        const int x = r & 1;
        const double ro = a.rn[r], ri = a.rn[r - 1];
        const long long id = (long long)a.id[r];
        const unsigned long long id_in = r > 1 ? a.id[r - 1] : ~0ULL;
        const double nI = -__dmul_rn(sum_of(p_dot + x * G), ro);
        // nu at an output position of the step (before the term bound)
        auto nu = [&](int pre) -> double {
            if (pre < 0) return 0.0;
            const int c = S.cmap[pre];
            return c < 0 ? 0.0 : (c == id ? nI : __dmul_rn(__ldcg(mu_out + c), ro));
        };
        double acc = 0.0, dot = 0.0;
        for (uint64_t i = tid; i < S.ci; i += all) {
            const PKey<W> K = S.kin[i];
            const double raw = S.cin[i];
            const double vs = nu(S.self_out[i]);
            double m = vs;
            if (commutes(K, S.g)) {
                const double sg = product_negative(K, S.g) ? -1.0 : 1.0;
                int po = S.emit_out[i];
                if (po < 0 && S.part_src[i] >= 0) po = S.self_out[S.part_src[i]];
                const double vp = nu(po);
                m = __dadd_rn(__dmul_rn(S.g.ch, vs), __dmul_rn(sg * S.g.msh, vp));
                const double u = normalised(raw, ri, key_is_zero(K));
                acc = __dadd_rn(acc, __dmul_rn(u, __dsub_rn(__dmul_rn(S.sh, vs),
                                                            __dmul_rn(sg * S.chd, vp))));
            }
            mu_in[i] = m;
            if (i != id_in) dot = __dadd_rn(dot, __dmul_rn(m, __dmul_rn(raw, ri)));
        }
        const double bg = block_sum(acc, s), bd = block_sum(dot, s);
        if (threadIdx.x == 0) {
            p_grad[x * G + blockIdx.x] = bg;
            p_dot[(x ^ 1) * G + blockIdx.x] = bd;
        }
        if (!team_barrier(team, a.ctl)) return;
        if (blockIdx.x == 0) {
            const double g = sum_of(p_grad + x * G);
            if (threadIdx.x == 0) gstep[r - 1] = g;
        }
        double* t = mu_out; mu_out = mu_in; mu_in = t;
    }
}

__global__ void __launch_bounds__(kRB)
k_adj_gsum(const double* partials, int np, double* gstep, long long s) {
    __shared__ double sh[kRB];
    double acc = 0.0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) acc = __dadd_rn(acc, partials[i]);
    const double b = block_sum(acc, sh);
    if (threadIdx.x == 0) gstep[s] = b;
}

template <int W>
__global__ void __launch_bounds__(256)
k_adj_remap_insert(const PKey<W>* keys, const double* mu, uint64_t n, Slot<W>* table,
                   uint64_t alloc_slots, DevCtl* ctl, int probe_limit) {
    const uint64_t mask = table_mask(n, alloc_slots, 50);
    const unsigned gen = ctl->gen;
    int probes = 0;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x)
        if (!table_insert(table, mask, gen, keys[i], mu[i], (uint32_t)i, probe_limit, &probes))
            set_status(ctl, ST_HASH_PROBE, 30);
}

template <int W>
__global__ void __launch_bounds__(256)
k_adj_remap_lookup(const PKey<W>* keys, uint64_t n, uint64_t n_table, double* mu,
                   const Slot<W>* table, uint64_t alloc_slots, DevCtl* ctl, int probe_limit) {
    const uint64_t mask = table_mask(n_table, alloc_slots, 50);
    const unsigned gen = ctl->gen;
    int probes = 0;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        double v = 0.0;
        if (!table_find(table, mask, gen, keys[i], &v, probe_limit, ctl, &probes))
            set_status(ctl, ST_STATE, 31);   // the sets at a boundary must agree
        mu[i] = v;
    }
}

__global__ void k_adj_bump_gen(DevCtl* ctl) {
    if (threadIdx.x == 0) ctl->gen = ctl->gen + 1u;
}

// The adjoint shares the handle's merge table: its generations continue the
// handle's, and the handle continues after the adjoint's, so no stale slot
// ever reads as occupied (the table is cleared first: the forward's selects
// keep lists in its memory).
__global__ void k_adj_gen_copy(DevCtl* dst, const DevCtl* src) {
    if (threadIdx.x == 0) dst->gen = src->gen + 1u;
}

// Frozen forward with other gate weights: one step of the linear map of
// Eq. (ITPP_PropRules) on the kept support recorded by the recompute (the
// output positions of every input's children, and which were kept), before
// the step's normalisation.  Every kept position receives exactly one write.
template <int W>
__global__ void __launch_bounds__(256)
k_frz_step(const PKey<W>* kin, const double* u_in, uint64_t n_in, const int* self_out,
           const int* emit_out, const int* part_src, const int* cmap, GateArg<W> g,
           double* u_out, const DevCtl* ctl) {
    if (ctl->status) return;   // maps may be missing
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_in;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const PKey<W> K = kin[i];
        const double u = u_in[i];
        const int so = self_out[i];
        const int ks = so >= 0 ? cmap[so] : -1;
        if (!commutes(K, g)) {
            if (ks >= 0) u_out[ks] = u;
            continue;
        }
        const double m = product_negative(K, g) ? -g.msh : g.msh;   // s (-sinh)
        const int ps = part_src[i];
        const double a = __dmul_rn(g.ch, u);
        if (ks >= 0) u_out[ks] = ps >= 0 ? __dadd_rn(a, __dmul_rn(m, u_in[ps])) : a;
        const int eo = emit_out[i];
        const int ke = eo >= 0 ? cmap[eo] : -1;
        if (ke >= 0) u_out[ke] = __dmul_rn(m, u);
    }
}

// The step's normalisation: every kept value divided by the identity's (the
// identity then exactly one).  d receives the identity's value first.
__global__ void k_frz_trace(const double* u, const unsigned long long* id_pos, double* d, const DevCtl* ctl) {
    if (threadIdx.x == 0 && blockIdx.x == 0 && !ctl->status) *d = u[*id_pos];
}

__global__ void __launch_bounds__(256)
k_frz_scale(double* u, uint64_t n, const unsigned long long* id_pos, const double* d) {
    const unsigned long long id = *id_pos;
    const double r = __ddiv_rn(1.0, *d);
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x)
        u[i] = i == id ? 1.0 : __dmul_rn(u[i], r);
}

// sum_i mu[i] u[i] (block partials; fixed grid, fixed order).
__global__ void __launch_bounds__(kRB)
k_frz_dot(const double* mu, const double* u, uint64_t n, double* partials) {
    __shared__ double s[kRB];
    double acc = 0.0;
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n;
         j += (uint64_t)gridDim.x * blockDim.x)
        acc = __dadd_rn(acc, __dmul_rn(mu[j], u[j]));
    const double b = block_sum(acc, s);
    if (threadIdx.x == 0) partials[blockIdx.x] = b;
}

// grad_alpha[k] = dtau * sum over layers of df/dtheta at gate k.
__global__ void k_adj_params(const double* gstep, int n_layers, int n_gates, double dtau,
                             double* grad) {
    for (int k = threadIdx.x; k < n_gates; k += blockDim.x) {
        double acc = 0.0;
        for (int l = 0; l < n_layers; ++l)
            acc = __dadd_rn(acc, gstep[(size_t)l * n_gates + k]);
        grad[k] = __dmul_rn(acc, dtau);
    }
}

// CTAs per SM of the two sweeps (which wait for one another's).
template <int W>
int adj_fit(bool recompute) {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &n, recompute ? reinterpret_cast<const void*>(&k_adj_recompute<W>)
                      : reinterpret_cast<const void*>(&k_adj_reverse<W>), kBlock, 0);
    return n > 0 ? n : 1;
}

struct DevBuf {
    void* p = nullptr;
    ~DevBuf() { if (p) cudaFree(p); }
    bool alloc(size_t bytes) { return cudaMalloc(&p, bytes ? bytes : 16) == cudaSuccess; }
    template <class T> T* as() const { return static_cast<T*>(p); }
};

// Weights of a frozen evaluation: per elementary gate of the schedule.
struct FrozenEval {
    std::vector<double> ch, msh;
};

// The adjoint sweep (ev == nullptr), or the frozen forward evaluated with the
// weights of ev on the support the handle's own coefficients produce (ev:
// value receives f, grad_alpha is not written).
template <int W>
itpp_status adjoint_w(itpp_ctx* h, int L, int K, const uint64_t* obs_x, const uint64_t* obs_z,
                      const double* seed, int m, double* grad_alpha, double* value,
                      const FrozenEval* ev = nullptr) {
    DeviceState& s = h->s;
    cudaStream_t st = h->stream;
    const int G = (int)h->gates.size();
    const long long S = (long long)L * G;
    if (K > L) K = L;   // one segment holds them all
    const int n_seg = (L + K - 1) / K;
    const size_t kb = sizeof(PKey<W>);
    const int grid = s.num_sms * 8;
    auto chk = [&](cudaError_t e) { return e == cudaSuccess; };

    // ---- forward from the identity, logging counts, snapshot per segment
    DevBuf log;
    if (!log.alloc((size_t)(S + 1) * 8)) return ITPP_ERR_ALLOC;
    if (!chk(launch_reset_identity(s, st))) return ITPP_ERR_CUDA;
    std::vector<DevBuf> snap((size_t)n_seg);
    std::vector<uint64_t> snap_n((size_t)n_seg);
    for (int j = 0; j < n_seg; ++j) {
        itpp_status stt = itpp_detail_sync_ctl(h);
        if (stt) return stt;
        const uint64_t c = h->h_ctl->count[h->h_ctl->cur];
        snap_n[(size_t)j] = c;
        if (!snap[(size_t)j].alloc((size_t)c * (kb + 8))) return ITPP_ERR_ALLOC;
        PKey<W>* sk = snap[(size_t)j].as<PKey<W>>();
        double* sc = reinterpret_cast<double*>(sk + c);
        if (!chk(itpp_detail_materialize(h))) return ITPP_ERR_CUDA;
        k_adj_snapshot<W><<<grid, 256, 0, st>>>(
            static_cast<const PKey<W>*>(s.keys[0]), s.coef[0],
            static_cast<const PKey<W>*>(s.keys[1]), s.coef[1], s.ctl, sk, sc);
        if (j == 0) k_adj_log<<<1, 32, 0, st>>>(s.ctl, log.as<unsigned long long>(), 0);
        const int l_end = (j + 1) * K < L ? (j + 1) * K : L;
        itpp_status e = itpp_detail_layers(h, l_end - j * K,
                                           log.as<unsigned long long>() + (size_t)j * K * G + 1);
        if (e) return e;
    }
    itpp_status stt = itpp_detail_sync_ctl(h);
    if (stt) return stt;
    std::vector<unsigned long long> cnt_log((size_t)S + 1);
    if (!chk(cudaMemcpy(cnt_log.data(), log.p, (size_t)(S + 1) * 8, cudaMemcpyDeviceToHost)))
        return ITPP_ERR_CUDA;

    // ---- value f and the observable table for the seed
    const size_t tsize = [&] { size_t t = 1; while (t < (size_t)2 * m) t <<= 1; return t; }();
    DevBuf obs;
    if (!obs.alloc((size_t)m * W * 16 + (size_t)m * 8 * 4 + tsize * 4 + (size_t)m * 4 + 64))
        return ITPP_ERR_ALLOC;
    char* op = obs.as<char>();
    uint64_t* d_ox = reinterpret_cast<uint64_t*>(op); op += (size_t)m * W * 8;
    uint64_t* d_oz = reinterpret_cast<uint64_t*>(op); op += (size_t)m * W * 8;
    double* d_w = reinterpret_cast<double*>(op); op += (size_t)m * 8;
    double* d_vals = reinterpret_cast<double*>(op); op += (size_t)m * 8;
    double* d_out = reinterpret_cast<double*>(op); op += (size_t)(m + 1) * 8;
    double* d_wsum = reinterpret_cast<double*>(op); op += (size_t)m * 8;
    int* d_tab = reinterpret_cast<int*>(op); op += tsize * 4;
    int* d_first = reinterpret_cast<int*>(op);
    if (!chk(cudaMemcpyAsync(d_ox, obs_x, (size_t)m * W * 8, cudaMemcpyHostToDevice, st)) ||
        !chk(cudaMemcpyAsync(d_oz, obs_z, (size_t)m * W * 8, cudaMemcpyHostToDevice, st)) ||
        !chk(cudaMemcpyAsync(d_w, seed, (size_t)m * 8, cudaMemcpyHostToDevice, st)))
        return ITPP_ERR_CUDA;
    if (!chk(itpp_detail_materialize(h)) ||
        !chk(launch_expect(s, d_ox, d_oz, d_w, m, (int)tsize, d_tab, d_first, d_vals, d_out, st)))
        return ITPP_ERR_CUDA;
    k_adj_wsum<<<1, 32, 0, st>>>(d_first, d_w, m, d_wsum);
    double fval = 0;
    if (!chk(cudaMemcpyAsync(&fval, d_out + m, 8, cudaMemcpyDeviceToHost, st)) ||
        !chk(cudaStreamSynchronize(st)))
        return ITPP_ERR_CUDA;

    // ---- arena for the largest segment.  Per step r >= 1: its kept terms (the
    // next step's input), the three output-position maps of the inputs and the
    // compaction map of the outputs before the term bound (at most 2 * inputs,
    // one buffer for all steps); region 0 holds the snapshot.
    auto round256 = [](size_t b) { return (b + 255) / 256 * 256; };
    size_t arena_max = 0, reg_max = 1;
    for (int j = 0; j < n_seg; ++j) {
        const long long s0 = (long long)j * K * G;
        const long long s1 = ((long long)(j + 1) * K < L ? (long long)(j + 1) * K : L) * G;
        size_t bytes = 0;
        for (long long q = s0; q <= s1; ++q) {
            const size_t c = cnt_log[(size_t)q];
            bytes += round256(c * kb) + round256(c * 8);
            if (q > s0) {
                const size_t ci = cnt_log[(size_t)(q - 1)];
                bytes += round256(ci * 12) + round256(2 * ci * 4);
                reg_max = 2 * ci > reg_max ? 2 * ci : reg_max;
            }
            reg_max = c > reg_max ? c : reg_max;
        }
        arena_max = bytes > arena_max ? bytes : arena_max;
    }
    const int steps_max = K * G;
    const uint64_t fit_c = (uint64_t)adj_fit<W>(true) * s.num_sms;
    const uint64_t fit_r = (uint64_t)adj_fit<W>(false) * s.num_sms;
    const auto grid_of = [](uint64_t fit, uint64_t want) {
        return (int)(want < 1 ? 1 : want < fit ? want : fit);
    };
    const int grid_c = grid_of(fit_c, (reg_max + 511) / 512);
    // (a tile is 512 inputs or 512 outputs, of which there are at most reg_max)
    const int grid_r = grid_of(fit_r < kRGrid ? fit_r : kRGrid, (reg_max + 511) / 512);
    // beside the arena: the outputs before the bound, the select's list and
    // its ties
    const size_t pre_at = round256(arena_max), prec_at = pre_at + round256(reg_max * kb);
    const size_t cv_at = prec_at + round256(reg_max * 8), ci_at = cv_at + round256(reg_max * 8);
    const size_t tie_at = ci_at + round256(reg_max * 4);
    DevBuf arena, mu0, mu1, musave, ctl2, arrs, part, gst, grad, d_steps, d_sh;
    if (!arena.alloc(tie_at + reg_max * kb) || !mu0.alloc(reg_max * 8) ||
        !mu1.alloc(reg_max * 8) || !musave.alloc(reg_max * 8) || !ctl2.alloc(sizeof(DevCtl)) ||
        !arrs.alloc((size_t)(steps_max + 1) * 8 * 4) || !part.alloc((size_t)kRGrid * 8 * 4) ||
        !gst.alloc((size_t)S * 8) || !grad.alloc((size_t)G * 8) ||
        !d_steps.alloc((size_t)steps_max * sizeof(AdjStep<W>)) || !d_sh.alloc(sizeof(AdjShared)))
        return ITPP_ERR_ALLOC;
    unsigned long long* a_cnt = arrs.as<unsigned long long>();
    double* a_rn = reinterpret_cast<double*>(a_cnt + steps_max + 1);
    unsigned long long* a_id = reinterpret_cast<unsigned long long*>(a_rn + steps_max + 1);
    unsigned long long* a_idpre = a_id + steps_max + 1;   // identity position before the bound
    DevCtl* c2 = ctl2.as<DevCtl>();
    if (!chk(cudaMemsetAsync(c2, 0, sizeof(DevCtl), st))) return ITPP_ERR_CUDA;
    k_adj_gen_copy<<<1, 32, 0, st>>>(c2, s.ctl);
    // the forward may have kept lists in the table's memory: no stale word may
    // read as a tag
    if (!chk(cudaMemsetAsync(s.table, 0, s.table_slots * sizeof(Slot<W>), st)))
        return ITPP_ERR_CUDA;
    double* mu_cur = mu0.as<double>();
    double* mu_prev = mu1.as<double>();

    // frozen evaluation: the state carried across segment boundaries (on
    // the next snapshot's order) and the identity's value of a step
    DevBuf u_snap, d_tr;
    if (ev && (!u_snap.alloc(reg_max * 8) || !d_tr.alloc(64))) return ITPP_ERR_ALLOC;
    if (ev) {
        const double one = 1.0;   // segment 0 starts from the identity alone
        if (!chk(cudaMemcpyAsync(u_snap.p, &one, 8, cudaMemcpyHostToDevice, st)))
            return ITPP_ERR_CUDA;
    }
    for (int jj = 0; jj < n_seg; ++jj) {
        const int j = ev ? jj : n_seg - 1 - jj;
        const long long s0 = (long long)j * K * G;
        const long long s1 = ((long long)(j + 1) * K < L ? (long long)(j + 1) * K : L) * G;
        const int R = (int)(s1 - s0);
        // region layout
        std::vector<AdjStep<W>> steps((size_t)R);
        char* ap = arena.as<char>();
        auto take = [&](size_t bytes) { char* q = ap; ap += round256(bytes); return q; };
        const uint64_t c0 = snap_n[(size_t)j];
        PKey<W>* rk = reinterpret_cast<PKey<W>*>(take(c0 * kb));
        double* rc = reinterpret_cast<double*>(take(c0 * 8));
        PKey<W>* const rk0 = rk;
        double* const rc0 = rc;
        for (int r = 1; r <= R; ++r) {
            AdjStep<W>& q = steps[(size_t)r - 1];
            const HostGate& hg = h->gates[(size_t)((s0 + r - 1) % G)];
            q.ci = r > 1 ? cnt_log[(size_t)(s0 + r - 1)] : c0;
            q.co = cnt_log[(size_t)(s0 + r)];
            q.kin = rk;
            q.cin = rc;
            rk = q.kout = reinterpret_cast<PKey<W>*>(take(q.co * kb));
            rc = q.cout = reinterpret_cast<double*>(take(q.co * 8));
            q.self_out = reinterpret_cast<int*>(take(q.ci * 12));
            q.emit_out = q.self_out + q.ci;
            q.part_src = q.emit_out + q.ci;
            q.cmap = reinterpret_cast<int*>(take(2 * q.ci * 4));
            q.g = gate_arg_of<W>(hg);
            q.sh = hg.sh;
            q.chd = hg.chd;
        }
        // restore the snapshot into region 0 (normalised values, rn = 1)
        const PKey<W>* sk = snap[(size_t)j].as<PKey<W>>();
        const double* sc = reinterpret_cast<const double*>(sk + c0);
        const unsigned long long c0u = c0;
        const double one = 1.0;
        if (!chk(cudaMemcpyAsync(rk0, sk, c0 * kb, cudaMemcpyDeviceToDevice, st)) ||
            !chk(cudaMemcpyAsync(rc0, sc, c0 * 8, cudaMemcpyDeviceToDevice, st)) ||
            !chk(cudaMemcpyAsync(a_cnt, &c0u, 8, cudaMemcpyHostToDevice, st)) ||
            !chk(cudaMemcpyAsync(a_rn, &one, 8, cudaMemcpyHostToDevice, st)) ||
            !chk(cudaMemcpyAsync(d_steps.p, steps.data(), (size_t)R * sizeof(AdjStep<W>),
                                 cudaMemcpyHostToDevice, st)) ||
            !chk(cudaMemsetAsync(d_sh.p, 0, sizeof(AdjShared), st)) ||
            !chk(cudaMemsetAsync(c2->count, 0, sizeof(c2->count), st)))
            return ITPP_ERR_CUDA;
        // recompute the segment, recording output positions
        AdjSweep<W> sw;
        sw.steps = d_steps.as<AdjStep<W>>();
        sw.n_steps = R;
        sw.kpre = reinterpret_cast<PKey<W>*>(arena.as<char>() + pre_at);
        sw.cpre = reinterpret_cast<double*>(arena.as<char>() + prec_at);
        sw.ctl = c2;
        sw.table = static_cast<Slot<W>*>(s.table);
        sw.slots = s.table_slots;
        sw.probe_limit = s.probe_limit;
        sw.cap_policy = s.cap_policy;
        sw.delta = s.delta;
        sw.cap_M = s.cap_M;
        sw.cnt0 = a_cnt;
        sw.rn = a_rn;
        sw.id = a_id;
        sw.id_pre = a_idpre;
        sw.sh = d_sh.as<AdjShared>();
        sw.cand_v = reinterpret_cast<unsigned long long*>(arena.as<char>() + cv_at);
        sw.cand_i = reinterpret_cast<uint32_t*>(arena.as<char>() + ci_at);
        sw.ties = reinterpret_cast<PKey<W>*>(arena.as<char>() + tie_at);
        void* sw_args[1] = {&sw};
        if (!chk(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_adj_recompute<W>),
                                             dim3(grid_c), dim3(kBlock), sw_args, 0, st)))
            return ITPP_ERR_CUDA;
        const size_t cR = cnt_log[(size_t)s1];
        if (ev) {
            // the recorded maps with the evaluation's weights, from the state
            // carried into this segment (on the snapshot's order)
            if (!chk(cudaMemcpyAsync(mu_prev, u_snap.p, c0 * 8, cudaMemcpyDeviceToDevice, st)))
                return ITPP_ERR_CUDA;
            for (int r = 1; r <= R; ++r) {
                const size_t gi = (size_t)((s0 + r - 1) % G);
                const AdjStep<W>& q = steps[(size_t)r - 1];
                GateArg<W> g = q.g;
                g.ch = ev->ch[gi];
                g.msh = ev->msh[gi];
                const size_t co = q.co;
                k_frz_step<W><<<grid, 256, 0, st>>>(q.kin, mu_prev, q.ci, q.self_out, q.emit_out,
                                                    q.part_src, q.cmap, g, mu_cur, c2);
                k_frz_trace<<<1, 32, 0, st>>>(mu_cur, a_id + r, d_tr.as<double>(), c2);
                k_frz_scale<<<grid, 256, 0, st>>>(mu_cur, co, a_id + r, d_tr.as<double>());
                double* t = mu_cur; mu_cur = mu_prev; mu_prev = t;
            }
            // mu_prev: the evaluated state on this segment's last order
            if (j < n_seg - 1) {
                const uint64_t cn = snap_n[(size_t)j + 1];
                const PKey<W>* nk = snap[(size_t)j + 1].as<PKey<W>>();
                k_adj_remap_insert<W><<<grid, 256, 0, st>>>(rk, mu_prev, cR,
                                                            static_cast<Slot<W>*>(s.table),
                                                            s.table_slots, c2, s.probe_limit);
                k_adj_remap_lookup<W><<<grid, 256, 0, st>>>(nk, cn, cR, u_snap.as<double>(),
                                                            static_cast<const Slot<W>*>(s.table),
                                                            s.table_slots, c2, s.probe_limit);
                k_adj_bump_gen<<<1, 32, 0, st>>>(c2);
            } else {
                k_adj_seed<W><<<grid, 256, 0, st>>>(rk, cR, d_ox, d_oz, d_wsum, d_tab,
                                                    (int)tsize, mu_cur);
                k_frz_dot<<<kRGrid, kRB, 0, st>>>(mu_cur, mu_prev, cR, part.as<double>());
                k_adj_gsum<<<1, kRB, 0, st>>>(part.as<double>(), kRGrid, d_tr.as<double>(), 1);
            }
            if (!chk(cudaGetLastError())) return ITPP_ERR_CUDA;
            continue;
        }
        // seed of this segment's last state
        if (j == n_seg - 1) {
            k_adj_seed<W><<<grid, 256, 0, st>>>(rk, cR, d_ox, d_oz, d_wsum, d_tab,
                                                (int)tsize, mu_cur);
        } else {
            // carry mu across the boundary by key: the next segment's snapshot
            const uint64_t cn = snap_n[(size_t)j + 1];
            const PKey<W>* nk = snap[(size_t)j + 1].as<PKey<W>>();
            k_adj_remap_insert<W><<<grid, 256, 0, st>>>(nk, musave.as<double>(), cn,
                                                        static_cast<Slot<W>*>(s.table),
                                                        s.table_slots, c2, s.probe_limit);
            k_adj_remap_lookup<W><<<grid, 256, 0, st>>>(rk, cR, cn, mu_cur,
                                                        static_cast<const Slot<W>*>(s.table),
                                                        s.table_slots, c2, s.probe_limit);
            k_adj_bump_gen<<<1, 32, 0, st>>>(c2);
        }
        // reverse sweep over the segment
        double* gst_seg = gst.as<double>() + s0;
        double* parts = part.as<double>();
        void* rv_args[5] = {&sw, &mu_cur, &mu_prev, &parts, &gst_seg};
        if (!chk(cudaMemsetAsync(d_sh.p, 0, sizeof(AdjShared), st)) ||
            !chk(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_adj_reverse<W>),
                                             dim3(grid_r), dim3(kBlock), rv_args, 0, st)))
            return ITPP_ERR_CUDA;
        if (R & 1) {
            double* t = mu_cur;
            mu_cur = mu_prev;
            mu_prev = t;
        }
        // mu on the snapshot order, for the previous segment
        if (!chk(cudaMemcpyAsync(musave.p, mu_cur, c0 * 8, cudaMemcpyDeviceToDevice, st)))
            return ITPP_ERR_CUDA;
        if (!chk(cudaGetLastError())) return ITPP_ERR_CUDA;
    }
    if (ev) {
        k_adj_gen_copy<<<1, 32, 0, st>>>(s.ctl, c2);
        double fe = 0.0;
        int c2_status = 0;
        if (!chk(cudaMemcpyAsync(&fe, d_tr.as<double>() + 1, 8, cudaMemcpyDeviceToHost, st)) ||
            !chk(cudaMemcpyAsync(&c2_status, &c2->status, sizeof(int), cudaMemcpyDeviceToHost,
                                 st)) ||
            !chk(cudaStreamSynchronize(st)))
            return ITPP_ERR_CUDA;
        if (c2_status) return (itpp_status)c2_status;
        *value = fe;
        return ITPP_OK;
    }
    k_adj_params<<<1, 256, 0, st>>>(gst.as<double>(), L, G, h->dtau, grad.as<double>());
    k_adj_gen_copy<<<1, 32, 0, st>>>(s.ctl, c2);
    int c2_status = 0;
    if (!chk(cudaMemcpyAsync(grad_alpha, grad.p, (size_t)G * 8, cudaMemcpyDeviceToHost, st)) ||
        !chk(cudaMemcpyAsync(&c2_status, &c2->status, sizeof(int), cudaMemcpyDeviceToHost, st)) ||
        !chk(cudaStreamSynchronize(st)))
        return ITPP_ERR_CUDA;
    if (c2_status) return (itpp_status)c2_status;
    if (value) *value = fval;
    return ITPP_OK;
}

}  // namespace

extern "C" itpp_status itpp_adjoint(itpp_handle h, int n_layers, int ckpt_every,
                                    const uint64_t* obs_x, const uint64_t* obs_z,
                                    const double* seed, int m, double* grad_alpha,
                                    double* value) {
    if (!h || n_layers < 1 || ckpt_every < 1 || !obs_x || !obs_z || !seed || !grad_alpha ||
        m < 1 || m > 65536)
        return ITPP_ERR_ARG;
    if (h->gates.empty()) return ITPP_ERR_ARG;
    if (h->sticky) return h->sticky;
    // gradients per elementary gate of the schedule, then folded onto the
    // Hamiltonian's coefficients (d alpha_gate / d alpha = src_scale)
    std::vector<double> g_sched(h->gates.size(), 0.0);
    itpp_status st = h->s.W == 1
        ? adjoint_w<1>(h, n_layers, ckpt_every, obs_x, obs_z, seed, m, g_sched.data(), value)
        : adjoint_w<2>(h, n_layers, ckpt_every, obs_x, obs_z, seed, m, g_sched.data(), value);
    if (st == ITPP_ERR_CUDA) h->sticky = st;
    if (st == ITPP_OK) {
        for (int k = 0; k < h->user_gates; ++k) grad_alpha[k] = 0.0;
        for (size_t j = 0; j < g_sched.size(); ++j)
            grad_alpha[h->src_gate[j]] += g_sched[j] * h->src_scale[j];
    }
    return st;
}

extern "C" itpp_status itpp_frozen_value(itpp_handle h, int n_layers, int ckpt_every,
                                         const double* alpha_eval, const uint64_t* obs_x,
                                         const uint64_t* obs_z, const double* w, int m,
                                         double* value) {
    if (!h || n_layers < 1 || ckpt_every < 1 || !alpha_eval || !obs_x || !obs_z || !w ||
        !value || m < 1 || m > 65536)
        return ITPP_ERR_ARG;
    if (h->gates.empty()) return ITPP_ERR_ARG;
    if (h->sticky) return h->sticky;
    FrozenEval ev;
    ev.ch.resize(h->gates.size());
    ev.msh.resize(h->gates.size());
    for (size_t j = 0; j < h->gates.size(); ++j) {
        const double a = alpha_eval[h->src_gate[j]];
        if (!std::isfinite(a)) return ITPP_ERR_ARG;
        const double theta = (a * h->src_scale[j]) * h->dtau;
        ev.ch[j] = std::cosh(theta);
        ev.msh[j] = -std::sinh(theta);
        if (!std::isfinite(ev.ch[j]) || !std::isfinite(ev.msh[j])) return ITPP_ERR_ARG;
    }
    itpp_status st = h->s.W == 1
        ? adjoint_w<1>(h, n_layers, ckpt_every, obs_x, obs_z, w, m, nullptr, value, &ev)
        : adjoint_w<2>(h, n_layers, ckpt_every, obs_x, obs_z, w, m, nullptr, value, &ev);
    if (st == ITPP_ERR_CUDA) h->sticky = st;
    return st;
}

extern "C" itpp_status itpp_set_alpha(itpp_handle h, const double* alpha) {
    if (!h || !alpha) return ITPP_ERR_ARG;
    for (int k = 0; k < h->user_gates; ++k)
        if (!std::isfinite(alpha[k])) return ITPP_ERR_ARG;
    for (size_t k = 0; k < h->gates.size(); ++k) {   // cosh / sinh overflow
        const double theta = (alpha[h->src_gate[k]] * h->src_scale[k]) * h->dtau;
        if (!std::isfinite(std::cosh(theta)) || !std::isfinite(std::sinh(theta))) return ITPP_ERR_ARG;
    }
    cudaStreamSynchronize(h->stream);
    for (size_t k = 0; k < h->gates.size(); ++k) {
        HostGate& g = h->gates[k];
        const double theta = (alpha[h->src_gate[k]] * h->src_scale[k]) * h->dtau;
        g.ch = std::cosh(theta);
        g.msh = -std::sinh(theta);
        g.sh = std::sinh(theta);
        g.chd = std::cosh(theta);
    }
    return ITPP_OK;
}
