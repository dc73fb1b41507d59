// itpp_part.cu -- a gate of a large state by separate launches: the partitioned
// merge, in place.
//
// A gate's merge only pairs a string K with its partner QK (Sec. II.B: a
// commuting string keeps cosh(theta) of itself and sends -sinh(theta) s to QK).
// Take a window of consecutive gates whose strings act on at most a few
// sites S, and group the state by the key with the sites of S cleared: K, QK
// and every child under any gate of the window share that group.  The state
// is scattered once per window into hash partitions of that masked key (one
// streaming pass, one atomic per term on the partition's cursor), and every
// gate of the window then runs over the partitions where they lie
// (itpp_inplace.cuh): a string keeps its place, its coefficient goes to the
// same place of a second array (zero: no term any more), and the few new
// strings are appended to the partition's stride, so keys are written only
// where they are new and no scatter runs between the gates of a window.  A
// group holds at most 4^|S| terms; a partition above a pass's capacity is
// merged in sub-passes, each taking the pairs of one hash class of the pair
// key, so no partition size forces a re-partition.  A gate
// acting on more sites than a window allows is a window of its own,
// partitioned by its pair key (the member of {K, QK} with the gate's lowest bit
// clear).
//
// The top-M select (Sec. II.C, term bound) is folded into the merge: every
// kept child is compared with a range around the threshold predicted for the
// gate; the merge counts the kept children, lists those inside the range and
// leaves out those below it (they are dropped by the select whenever at least
// cap_M children lie at or above the range; otherwise, and when a stride ran
// out, k_gate_part merges again in full from the unchanged input into a
// contiguous run), and the select (itpp_select.cu) then works on that short
// list instead of passing over every coefficient.
#include <cstring>

#include "itpp_common.cuh"
#include "itpp_gate_body.cuh"
#include "itpp_launch.h"
#include "itpp_stage.cuh"
#include "itpp_inplace.cuh"

namespace itpp {

// Scatter the current state into the partitions of a window (force), or,
// inside a window, only when the state has no partitions, or those of another
// window, or they held for the previous gate alone.  The state is a contiguous
// run, or the partitions of a home; it goes to the other home.
//
// What bounds it: the random stores and cursor claims of 32 different
// partitions a warp, each an access of its own (2.2 ms for 2^26 terms, 1.4 TB/s
// of the bytes it moves, DRAM 29 % busy, a real scatter in 29 of the 64-site
// chain's 128 gates).  More loads or claims in flight, fewer or more CTAs and
// padded cursors leave it as it is at that size; claims before first use help
// where the state sits in L2.
template <int W>
__global__ void __launch_bounds__(256, 4)
k_part_scatter(Bufs<W> B, Homes<W> H, DevCtl* ctl, GateArg<W> g, PartFn<W> f, int force, int win,
               int n_sites, int target, int redo) {
    if (ctl->status) return;
    // the second launch of a gate's scatter runs only when the first one
    // found a partition's stride too small for the groups hashed to it; it
    // scatters by the gate's pair key (pairs always fit) into cleared cursors
    if (redo && !ctl->scatter_over) return;
    if (redo) f.pair = 1;
    const int cur = ctl->cur;
    const bool run = force || redo || ctl->need_scatter || !ctl->home || ctl->part_win != win;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        // the next merge's counters
        ctl->count[cur ^ 1] = 0ULL;
        ctl->alloc = 0ULL;
        ctl->sp_ovf = 0;
        ctl->over = 0;
        ctl->scattered = run;
    }
    if (!run) return;
    const uint64_t n = live_count(ctl, cur);
    const bool fallback = redo || (!f.pair && !window_fits(n_sites, f.sites, n));
    if (fallback) f.pair = 1;
    PartPlan pl = part_plan(n, H.cap, H.part_max, target);
    if (!f.pair) {
        // a partition's stride holds a whole group (up to 4^sites strings,
        // the terms with one pattern outside the window), however the terms
        // fall, where that keeps partitions near the target; larger windows
        // rely on the second scatter by pair key when a stride overflows
        const uint64_t gmax = 1ULL << (2 * f.sites);
        if (pl.R < gmax && gmax <= 2ULL * (uint64_t)target) {
            const uint64_t P = H.cap / gmax;
            pl.P = (uint32_t)(P > 0 ? P : 1);
            pl.R = H.cap / pl.P;
        }
    }
    const bool home = ctl->home != 0;
    const int a = home ? ctl->ha : cur;
    const int to_b = home ? ctl->hb ^ 1 : 0, to_x = home ? ctl->hx ^ 1 : 0;
    const int to_c = next3(ctl->hc);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->to_b = to_b;
        ctl->to_x = to_x;
        ctl->to_c = to_c;
        ctl->to_P = pl.P;
        ctl->to_R = pl.R;
        ctl->to_win = win;
        if (!home) ctl->ha = cur;
        ctl->stat_scatters += 1;
        ctl->part_over = f.pair;   // such partitions hold for this gate only
    }
    const Pending<W> pd = pending_of<W>(ctl);
    // one loop for both layouts (a single copy of the scatter body): each
    // partition by one CTA, or the contiguous run by the whole grid
    const StateRuns<W> r = state_runs(ctl, B, H);
    for (uint32_t s = r.cnt ? blockIdx.x : 0u; s < r.P; s += r.cnt ? gridDim.x : 1u) {
        const uint64_t off = (uint64_t)s * r.R;
        const uint64_t cnt = r.cnt ? (r.cnt[s] < r.R ? (uint64_t)r.cnt[s] : r.R) : r.n;
        const uint64_t first = r.cnt ? 0ULL : (uint64_t)blockIdx.x * blockDim.x;
        const uint64_t stride = r.cnt ? (uint64_t)blockDim.x : (uint64_t)gridDim.x * blockDim.x;
        scatter_run(r.keys + off, r.coef + off, cnt, first, stride, pd, ctl,
                    H.keys(B, a, to_b), H.coef(B, a, to_x), H.cursors(to_c), pl, g, f,
                    [&] {
                        if (!f.pair) ctl->scatter_over = 1;   // again by the pair key
                        else set_status(ctl, ST_CAPACITY, 40);
                    });
    }
    if (redo) return;
    // when a stride was too small, the last CTA clears the cursors for the
    // second launch
    __shared__ int s_clear;
    __syncthreads();
    if (threadIdx.x == 0) s_clear = last_cta(ctl) && *(volatile int*)&ctl->scatter_over;
    __syncthreads();
    if (s_clear)
        for (uint32_t i = threadIdx.x; i < H.part_max; i += blockDim.x)
            H.cursors(__ldcg(&ctl->to_c))[i] = 0u;   // (read again: one register less over the loop)
}

// After a merge that left children out: with at least cap_M kept, the select
// keeps cap_M of them and every one left out lay below them all; with fewer
// they are needed.  Then, and when a partition's stride ran out, the gate's
// merge is done again in full (its input is still in place).  One thread.
__device__ __forceinline__ void merge_check(DevCtl* ctl, uint64_t cap_M) {
    const int nxt = ctl->cur ^ 1;
    ctl->retry = 0;
    ctl->scatter_over = 0;   // the gate's scatters are done
    if (__ldcg(&ctl->over) || (__ldcg(&ctl->drop_on) && __ldcg(&ctl->count[nxt]) < cap_M)) {
        ctl->retry = 1;
        ctl->count[nxt] = 0ULL;
        ctl->alloc = 0ULL;
        ctl->sp_ovf = 0;
        ctl->cand_regions = 0;
        ctl->out_max = 0ULL;
        ctl->stat_retry += 1ULL;
    }
    ctl->drop_on = 0;
}

// Where this gate's input partitions are: where its scatter put them, or
// where the previous gate left them.
struct GateInput {
    int a, b, x, c;
    uint32_t P;
    uint64_t R;
};

__device__ __forceinline__ GateInput gate_input(const DevCtl* ctl) {
    GateInput in;
    const bool s = ctl->scattered != 0;
    in.a = ctl->ha;
    in.b = s ? ctl->to_b : ctl->hb;
    in.x = s ? ctl->to_x : ctl->hx;
    in.c = s ? ctl->to_c : ctl->hc;
    in.P = s ? ctl->to_P : ctl->part_P;
    in.R = s ? ctl->to_R : ctl->part_R;
    return in;
}

// The gate's merge, in place (itpp_inplace.cuh): persistent CTAs, one
// partition at a time, a later partition of the same CTA prefetched into L2
// by bulk (TMA) requests.  With a top-M bound the children at or
// below the select's lower limit are left out; merge_check then keeps the
// result when at least cap_M were kept and no partition's stride ran out, and
// otherwise k_gate_part merges the gate again in full from the same input.
template <int W, int BLOCK>
__global__ void __launch_bounds__(BLOCK, (InOcc<W, BLOCK>::kMin))
k_gate_inplace(Bufs<W> B, Homes<W> H, DevCtl* ctl, GateArg<W> g, double delta, CandRegions cd,
               uint64_t cap_M) {
    constexpr uint32_t C = InPass<W, kLargeBits>::C;
    __shared__ unsigned long long s_T, s_thr, s_kept;
    __shared__ PKey<W> s_tk;
    __shared__ double s_rnorm;
    __shared__ uint32_t s_long, s_n, s_app, s_rare;
    __shared__ int s_stop, s_ties, s_over;
    const int cur = ctl->cur, nxt = cur ^ 1;
    const GateInput in = gate_input(ctl);
    const uint64_t R = in.R;
    if (threadIdx.x == 0) {
        // one read of the status for the whole CTA (another CTA may set it
        // meanwhile, and every thread must leave at the same point)
        s_stop = ctl->status;
        const Pending<W> pd = pending_of<W>(ctl);
        s_T = pd.T;
        s_ties = pd.all_ties;
        s_tk = pd.tk;
        s_rnorm = ctl->rnorm[cur];
        g_cn = 0u;
        g_range[0] = ctl->sp_lo;
        g_range[1] = ctl->sp_hi;
        s_kept = 0ULL;
        s_long = 0u;
        s_over = 0;
        s_app = s_rare = 0u;
        const unsigned long long dbits = (unsigned long long)__double_as_longlong(delta);
        const unsigned long long thr = ctl->sp_hi && ctl->sp_thr > dbits ? ctl->sp_thr : dbits;
        s_thr = thr;
        g_delta = dbits;
        if (blockIdx.x == 0 && !ctl->status) {
            ctl->drop_on = thr != dbits;
            ctl->cand_regions = gridDim.x;
        }
    }
    inplace_init<W, BLOCK, kLargeBits>();
    __syncthreads();
    if (s_stop) return;
    // the third cursor array (the previous gate's input) is the next scatter's
    {
        unsigned int* spare = H.cursors(next3(next3(in.c)));
        for (uint32_t i = blockIdx.x * BLOCK + threadIdx.x; i < H.part_max; i += gridDim.x * BLOCK)
            spare[i] = 0u;
    }
    PKey<W>* keys = H.keys(B, in.a, in.b);
    const double* cin = H.coef(B, in.a, in.x);
    double* cout = H.coef(B, in.a, in.x ^ 1);
    const unsigned int* cnt_in = H.cursors(in.c);
    unsigned int* cnt_out = H.cursors(next3(in.c));
    const uint32_t p_id = identity_part<W>(in.P);
    auto push = [&](bool hit, unsigned long long v, uint64_t idx) {
        cand_push(hit, v, idx, cd, &g_cn);
    };
    InStats st{0u, 0u};
    uint32_t tag = 0;
    InRows<W, BLOCK> rows;
    auto stored = [&](uint32_t p) -> uint32_t {
        const uint32_t c = p < in.P ? cnt_in[p] : 0u;
        return c < R ? c : (uint32_t)R;
    };
    auto load = [&](uint32_t p, uint32_t n) {   // (a longer one is gathered later)
        if (n && n <= C) load_rows<W, BLOCK, false>(rows, keys + (uint64_t)p * R, cin + (uint64_t)p * R, n);
    };
    uint32_t np = stored(blockIdx.x), np2 = stored(blockIdx.x + gridDim.x);
    load(blockIdx.x, np);
    for (uint32_t p = blockIdx.x; p < in.P; p += gridDim.x) {
        InPlace<W> io;
        io.n = np;
        io.room = (uint32_t)(R < 0xffffffffULL ? R : 0xffffffffULL);
        io.first = (uint64_t)p * R;
        io.keys = keys + io.first;
        io.cin = cin + io.first;
        io.cout = cout + io.first;
        io.s_app = &s_app;
        io.s_rare = &s_rare;
        io.over = &s_over;
        // warm L2 with the partition after the next
        const uint32_t pn = p + gridDim.x, pf = pn + gridDim.x;
        np = np2;
        np2 = stored(pf);
        if (threadIdx.x == 0 && np2) {
            l2_prefetch_bulk(keys + (uint64_t)pf * R, np2 * sizeof(PKey<W>));
            l2_prefetch_bulk(cin + (uint64_t)pf * R, np2 * sizeof(double));
        }
        const bool subs = inplace_partition<W, BLOCK, kLargeBits>(g, s_T, s_ties != 0, s_tk, s_rnorm, s_thr,
                                                      p == p_id, ctl, nxt, &tag, io, st,
                                                      g_range[1], &s_n, rows, push,
                                                      [&] { load(pn, np); });
        if (threadIdx.x == 0) {
            // (the others use these again only after the next pass's barrier)
            const uint64_t c = (uint64_t)io.n + s_app;
            cnt_out[p] = (unsigned int)(c < R ? c : R);
            s_app = s_rare = 0u;
            if (subs) s_long += 1u;
        }
        if (tag >= kHeadTagMax - 65536u) {   // tags start again
            inplace_init<W, BLOCK, kLargeBits>();
            tag = 0;
            __syncthreads();
        }
    }
    // one atomic per warp for the largest pattern, one per CTA for the term
    // count
    const uint32_t hm = __reduce_max_sync(0xffffffffu, st.hi_max);
    const uint32_t kept = __reduce_add_sync(0xffffffffu, st.kept);
    if ((threadIdx.x & 31) == 0) {
        if (hm) atomicMax(&ctl->out_max, ((unsigned long long)hm << 32) | 0xffffffffULL);
        if (kept) atomicAdd(&s_kept, (unsigned long long)kept);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_kept) atomicAdd(&ctl->count[nxt], s_kept);
        if (s_long) atomicAdd(&ctl->stat_long, (unsigned long long)s_long);
        if (s_over) ctl->over = 1;
        const uint32_t c = g_cn;
        cd.cnt[blockIdx.x] = c < cd.region ? c : (uint32_t)cd.region;
        if (c > cd.region) ctl->sp_ovf = 1;
        if (last_cta(ctl)) merge_check(ctl, cap_M);
    }
}

// The gate's merge again, in full, into a contiguous run of the free buffer:
// one partition at a time per CTA, its children counted, then claimed (one
// atomic a partition) and written.  Lists no candidates: the select passes
// over the state.
template <int W, int BLOCK>
__global__ void __launch_bounds__(BLOCK, (PartOcc<W, BLOCK>::kMin))
k_gate_part(Bufs<W> B, Homes<W> H, DevCtl* ctl, GateArg<W> g, double delta, uint64_t cap_out) {
    using A = PassArgs<W>;
    __shared__ unsigned long long s_at;
    __shared__ uint32_t s_n;
    __shared__ int s_stop;
    __shared__ Pending<W> s_pd;
    __shared__ double s_rnorm;
    const int cur = ctl->cur, nxt = cur ^ 1;
    if (threadIdx.x == 0) {
        s_stop = ctl->status || !ctl->retry;
        s_pd = pending_of<W>(ctl);
        s_rnorm = ctl->rnorm[cur];
    }
    __syncthreads();
    if (s_stop) return;
    pass_init<W, BLOCK>();
    __syncthreads();
    const GateInput in = gate_input(ctl);
    const unsigned long long dbits = (unsigned long long)__double_as_longlong(delta);
    const PKey<W>* keys = H.keys(B, in.a, in.b);
    const double* cin = H.coef(B, in.a, in.x);
    PKey<W>* kout = B.key(in.a);
    double* cout = B.coef(in.a);
    const uint32_t p_id = identity_part<W>(in.P);
    {   // the first try's cursors: the next scatter's
        unsigned int* spare = H.cursors(next3(in.c));
        for (uint32_t i = blockIdx.x * BLOCK + threadIdx.x; i < H.part_max; i += gridDim.x * BLOCK)
            spare[i] = 0u;
    }
    auto room = [&](uint32_t n_out) -> unsigned long long {
        if (threadIdx.x == 0) {
            unsigned long long at = n_out ? atomicAdd(&ctl->alloc, (unsigned long long)n_out) : 0ULL;
            if (at + n_out > cap_out) {
                set_status(ctl, ST_CAPACITY, 2);
                at = ~0ULL;
            }
            s_at = at;
        }
        __syncthreads();
        return s_at;
    };
    SelStats st{0ULL};
    uint32_t pass = 0;
    for (uint32_t p = blockIdx.x; p < in.P; p += gridDim.x) {
        uint64_t np = H.cursors(in.c)[p];
        if (np > in.R) np = in.R;
        const PKey<W>* kp = keys + (uint64_t)p * in.R;
        const double* cp = cin + (uint64_t)p * in.R;
        if (np <= (uint64_t)Stage<W>::C) {
            ++pass;   // (merge_long numbers its own: consecutive passes alternate)
            for (uint32_t i = threadIdx.x; i < np; i += BLOCK) {
                A::keys()[i] = load_key_stream(kp + i);
                A::vals()[i] = __ldcs(cp + i);
            }
            __syncthreads();
            stage_pass<W, BLOCK, PassRoom::kExact>((uint32_t)np, g, s_pd, s_rnorm, dbits,
                                                   p == p_id, ctl, nxt, pass, kout, cout, st, room);
        } else {
            merge_long<W, BLOCK>(kp, cp, np, g, s_pd, s_rnorm, dbits, p == p_id, ctl, nxt, &pass,
                                 kout, cout, st, room, &s_n);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        st.out_max = max(st.out_max, __shfl_xor_sync(0xffffffffu, st.out_max, o));
    if ((threadIdx.x & 31) == 0 && st.out_max) atomicMax(&ctl->out_max, st.out_max);
}

// After the merge: where the state is now, then the buffer switch, normaliser,
// statistics and bound of every gate (post_one), and the way to the top-M
// threshold (itpp_select.cu): the merge's candidates when the cap_M-th largest
// value lies among them, else passes over the state.
__global__ void __launch_bounds__(256)
k_part_post(DevCtl* ctl, CandRegions cd, uint64_t cap_M, int cap_policy, uint64_t cand_cap,
            unsigned long long delta_bits) {
    __shared__ uint32_t s_scan[256 / 32];
    if (ctl->status) return;
    const uint32_t nreg = ctl->cand_regions < 1024u ? ctl->cand_regions : 1024u;
    uint32_t c = 0, tot;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const uint32_t r = u * 256u + threadIdx.x;
        c += r < nreg ? cd.cnt[r] : 0u;
    }
    block_exclusive_scan<256>(c, &tot, s_scan);
    unsigned int* team = reinterpret_cast<unsigned int*>(&ctl->sel);
    for (uint32_t b = threadIdx.x; b < sizeof(SelTeam) / 4; b += 256u) team[b] = 0u;
    if (threadIdx.x == 0) {
        if (ctl->scattered) {
            ctl->home = 1;
            ctl->hb = ctl->to_b;
            ctl->hx = ctl->to_x;
            ctl->hc = ctl->to_c;
            ctl->part_P = ctl->to_P;
            ctl->part_R = ctl->to_R;
            ctl->part_win = ctl->to_win;
        }
        if (ctl->retry) {
            ctl->home = 0;
            ctl->count[ctl->cur ^ 1] = ctl->alloc;
            ctl->alloc = 0ULL;
        } else {
            ctl->hx ^= 1;
            ctl->hc = next3(ctl->hc);
        }
        const int active = post_one(ctl, cap_M, cap_policy);
        const int cur = ctl->cur, a = ctl->ha;
        const unsigned long long kept = ctl->count[cur];
        if (!ctl->home && cur != a) {   // the run is in buffer a
            ctl->count[a] = kept;
            ctl->norm[a] = ctl->norm[cur];
            ctl->rnorm[a] = ctl->rnorm[cur];
            ctl->cur = a;
        }
        if (active) {
            // kept children above the range: all that were not listed
            const unsigned long long above = kept - tot;
            const int reason = ctl->sp_hi == 0ULL ? 1
                               : (ctl->sp_ovf || tot > cand_cap) ? 2
                               : above >= cap_M ? 3
                               : above + tot < cap_M ? 4 : 0;
            const bool fast = reason == 0;
            const unsigned long long range = ctl->sp_hi - ctl->sp_lo;
            ctl->sel_fast = fast ? 1 : 0;
            ctl->sp_reason = reason;
            ctl->sel_prefix = 0ULL;
            ctl->sel_mask = 0ULL;
            ctl->sel_lo = fast ? ctl->sp_lo : delta_bits;
            ctl->sel_cand_n = fast ? tot : 0ULL;
            if (fast) {
                ctl->sel_top = range ? 64 - __clzll((long long)range) : 0;
                ctl->sel_k = cap_M - above;
            } else {
                ctl->stat_sel_full += 1;
            }
        } else if (ctl->retry) {
            // the state has fallen below its bound: with the old limit every
            // gate from here on would be merged twice
            ctl->sp_thr = ctl->sp_lo = ctl->sp_hi = ctl->sp_tprev = 0ULL;
        }
    }
}

// ---------------------------------------------------------------------------
// Launcher
// ---------------------------------------------------------------------------
template <int W>
static Bufs<W> pbufs_of(const DeviceState& s) {
    Bufs<W> b;
    for (int i = 0; i < 2; ++i) {
        b.k[i] = reinterpret_cast<PKey<W>*>(s.keys[i]);
        b.c[i] = s.coef[i];
    }
    return b;
}

template <int W>
static GateArg<W> gate_of(const HostGate& h) {
    GateArg<W> g;
    for (int w = 0; w < W; ++w) { g.qx[w] = h.qx[w]; g.qz[w] = h.qz[w]; }
    g.ch = h.ch;
    g.msh = h.msh;
    g.qyy = h.qyy;
    g.maxw = h.maxw;
    return g;
}

template <int W>
static PartFn<W> part_fn_of(const HostGate& h) {
    PartFn<W> f;
    for (int w = 0; w < W; ++w) { f.kx[w] = h.keep_x[w]; f.kz[w] = h.keep_z[w]; }
    f.pair = h.pair_mode;
    f.sites = h.win_sites;
    bool found = false;
    for (int w = 0; w < 2 * W; ++w) {
        const uint64_t m = w < W ? h.qx[w] : h.qz[w - W];
        const uint64_t bit = (!found && m) ? (m & (~m + 1)) : 0ULL;
        if (w < W) f.px[w] = bit; else f.pz[w - W] = bit;
        found = found || m;
    }
    return f;
}

template <int W>
static Homes<W> homes_of(const DeviceState& s) {
    Homes<W> h;
    h.kp = reinterpret_cast<PKey<W>*>(s.part_keys);
    h.cp = s.part_coef;
    h.cnt = s.part_cursor;
    h.part_max = s.part_max;
    h.cap = s.part_cap < s.buf_cap ? s.part_cap : s.buf_cap;
    return h;
}

template <int W>
static cudaError_t scatter_w(const DeviceState& s, const HostGate& h, cudaStream_t st) {
    uint64_t gs = (s.buf_cap + 255) / 256;
    const uint64_t lim = (uint64_t)s.num_sms * 8;
    if (gs > lim) gs = lim;
    if (gs < 1) gs = 1;
    for (int redo = 0; redo < 2; ++redo) {
        k_part_scatter<W><<<(int)gs, 256, 0, st>>>(pbufs_of<W>(s), homes_of<W>(s), s.ctl,
                                                   gate_of<W>(h), part_fn_of<W>(h), h.win_start,
                                                   h.win, s.n, s.part_target, redo);
    }
    return cudaGetLastError();
}

template <int W, int BLOCK>
static cudaError_t merge_wb(const DeviceState& s, const GateArg<W>& g, cudaStream_t st) {
    static int per_sm = 0, per_sm_full = 0;
    constexpr size_t smem = InPass<W, kLargeBits>::kBytes, smem_full = Stage<W>::kBytes;
    if (!per_sm) {
        // shared memory for every resident CTA's staging rather than L1
        cudaFuncSetAttribute(k_gate_inplace<W, BLOCK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
        cudaFuncSetAttribute(k_gate_inplace<W, BLOCK>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             (int)cudaSharedmemCarveoutMaxShared);
        cudaFuncSetAttribute(k_gate_part<W, BLOCK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem_full);
        cudaFuncSetAttribute(k_gate_part<W, BLOCK>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             (int)cudaSharedmemCarveoutMaxShared);
        int n = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gate_part<W, BLOCK>, BLOCK, smem_full);
        per_sm_full = n > 0 ? n : 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gate_inplace<W, BLOCK>, BLOCK, smem);
        per_sm = n > 0 ? n : 1;
    }
    int grid = s.num_sms * per_sm;
    if (grid > s.max_ctas) grid = s.max_ctas;   // one candidate region per CTA
    k_gate_inplace<W, BLOCK><<<grid, BLOCK, smem, st>>>(pbufs_of<W>(s), homes_of<W>(s), s.ctl, g,
                                                        s.delta, s.cand, s.cap_M);
    k_gate_part<W, BLOCK><<<s.num_sms * per_sm_full, BLOCK, smem_full, st>>>(
        pbufs_of<W>(s), homes_of<W>(s), s.ctl, g, s.delta, s.buf_cap);
    return cudaGetLastError();
}

// The partitioned merge's CTA size (threads loop over a partition's staged
// strings, so there is no items-per-thread parameter on this path).
template <int W>
static cudaError_t merge_w(const DeviceState& s, const HostGate& h, cudaStream_t st) {
    const GateArg<W> g = gate_of<W>(h);
    switch (s.block) {
        case 128: return merge_wb<W, 128>(s, g, st);
        case 256: return merge_wb<W, 256>(s, g, st);
        case 512: return merge_wb<W, 512>(s, g, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_part_scatter(const DeviceState& s, const HostGate& h, cudaStream_t st) {
    return s.W == 1 ? scatter_w<1>(s, h, st) : scatter_w<2>(s, h, st);
}

cudaError_t launch_part_post(const DeviceState& s, cudaStream_t st) {
    unsigned long long dbits;
    std::memcpy(&dbits, &s.delta, sizeof dbits);   // delta >= +0: it bounds every kept pattern
    k_part_post<<<1, 256, 0, st>>>(s.ctl, s.cand, s.cap_M, s.cap_policy, select_list_cap(s), dbits);
    return cudaGetLastError();
}

cudaError_t launch_part_merge(const DeviceState& s, const HostGate& h, cudaStream_t st) {
    return s.W == 1 ? merge_w<1>(s, h, st) : merge_w<2>(s, h, st);
}

void plan_windows(int W, std::vector<HostGate>& gates) {
    const int max_sites = W == 1 ? PartGeom<1>::kWinSites : PartGeom<2>::kWinSites;
    auto sites = [](const uint64_t* m) {
        return __builtin_popcountll(m[0]) + __builtin_popcountll(m[1]);
    };
    size_t k = 0;
    while (k < gates.size()) {
        uint64_t S[2] = {gates[k].qx[0] | gates[k].qz[0], gates[k].qx[1] | gates[k].qz[1]};
        if (sites(S) > max_sites) {
            // a wide gate: a window of its own, partitioned by its pair key
            HostGate& h = gates[k];
            h.pair_mode = 1;
            h.win_start = 1;
            h.win = (int)k;
            for (int w = 0; w < 2; ++w) { h.keep_x[w] = ~0ULL; h.keep_z[w] = ~0ULL; }
            ++k;
            continue;
        }
        size_t e = k + 1;
        while (e < gates.size()) {
            const uint64_t T[2] = {S[0] | gates[e].qx[0] | gates[e].qz[0],
                                   S[1] | gates[e].qx[1] | gates[e].qz[1]};
            if (sites(T) > max_sites) break;
            S[0] = T[0];
            S[1] = T[1];
            ++e;
        }
        for (size_t j = k; j < e; ++j) {
            HostGate& h = gates[j];
            h.pair_mode = 0;
            h.win_sites = sites(S);
            h.win_start = j == k;
            h.win = (int)k;
            for (int w = 0; w < 2; ++w) { h.keep_x[w] = ~S[w]; h.keep_z[w] = ~S[w]; }
        }
        k = e;
    }
}

int partition_target_default(int W) {
    return W == 1 ? PartGeom<1>::kTarget : PartGeom<2>::kTarget;
}

uint32_t partition_max(uint64_t cap_M, int target) {
    const uint64_t t = (uint64_t)target;
    return (uint32_t)((cap_M + t - 1) / t + 1);
}

}  // namespace itpp
