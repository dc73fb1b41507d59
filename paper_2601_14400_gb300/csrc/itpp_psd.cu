// itpp_psd.cu -- the positive-semidefinite-restored observable (Sec. II.C):
//
//   <O>_{2 tau} ~= Tr[(O rho) rho] / Tr[rho^2],   rho = sum_P c_P P, c_I = 1,
//
// for O = sum_j w_j O_j.  With Tr(P_a P_b) = 2^n delta_ab the purity is
// Tr[rho^2] / 2^n = sum_P c_P^2 (the squared l2 norm of the coefficients),
// and Tr[(O_j P) R] is nonzero only for R = O_j.P.  When O_j and P
// anticommute the product carries a factor +-i and the pair (P, O_j.P) is
// met again as (O_j.P, P) with the opposite factor, so those terms cancel;
// when they commute O_j P = s O_j.P with s = +-1 (the sign of the
// propagation rule), so
//
//   Tr[(O rho) rho] / 2^n = sum_j w_j sum_{P : [P, O_j] = 0} s(O_j, P) c_P c_{O_j.P}.
//
// That is a partner lookup: every term of the state goes into the merge
// table (under a generation of its own), then one pass over the state
// looks up O_j.P for every commuting observable string.  Sums are
// compensated per thread, then reduced in a fixed order, so the result does
// not depend on scheduling.  Few of the strings O_j.P are in the state (a few in
// a hundred for the chains), so a bitmap of the state's hashes, about 8 to 16
// bits a term, is asked first: a 4-byte read that mostly hits L1 instead of a
// random 32- or 64-byte table slot.  What
// passes it goes on a queue per warp and is looked up and summed 32 at a time: a
// warp holds the double-precision pipe for every instruction however few of its
// lanes have a pair (448 us for 2^18 terms and 63 strings when each lane did its
// own, 185 us this way).  Each pair {P, O_j.P} is taken once, from the member without O_j's
// lowest bit, and counts twice.
#include "itpp_common.cuh"
#include "itpp_gate_body.cuh"
#include "itpp_launch.h"

namespace itpp {

namespace {

constexpr int kPB = 256;

template <int W>
static Bufs<W> psd_bufs(const DeviceState& s) {
    Bufs<W> b;
    for (int i = 0; i < 2; ++i) {
        b.k[i] = reinterpret_cast<PKey<W>*>(s.keys[i]);
        b.c[i] = s.coef[i];
    }
    return b;
}

// A fresh table generation for the state's terms (never equal to a gate's).
// Clears the filter.
template <int W>
__global__ void k_psd_begin(Bufs<W> B, DevCtl* ctl, size_t fbytes) {
    if (ctl->status) return;
    uint4* f = reinterpret_cast<uint4*>(B.key(ctl->cur ^ 1));
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < fbytes / 16;
         i += (size_t)gridDim.x * blockDim.x)
        f[i] = make_uint4(0u, 0u, 0u, 0u);
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    ctl->gen = ctl->gen + 1u;
    if (ctl->gen == 0u) set_status(ctl, ST_STATE, 60);
}

// Bits of the filter for n terms: the power of two between 8 and 16 a term.
__device__ __forceinline__ uint32_t filter_shift(uint64_t n) {
    int b = 64 - __clzll((long long)(n | 7ULL));   // n < 2^b
    b += 3;
    return 32u - (uint32_t)(b < 31 ? b : 31);        // the hash's top bits
}

template <int W>
__device__ __forceinline__ uint32_t filter_hash(const PKey<W>& K) {
    uint32_t h = 0x51ed270bu;
#pragma unroll
    for (int w = 0; w < W; ++w)
        h = h * 0x2c1b3c6du + (uint32_t)K.x[w] * 0x9e3779b1u + (uint32_t)(K.x[w] >> 32) * 0x85ebca77u +
            (uint32_t)K.z[w] * 0xc2b2ae3du + (uint32_t)(K.z[w] >> 32) * 0x27d4eb2fu;
    return h;
}

// Every term of the state, normalised, into the table and the filter.
template <int W>
__global__ void __launch_bounds__(kPB)
k_psd_build(Bufs<W> B, DevCtl* ctl, Slot<W>* table, uint64_t slots, int load_pct,
            int probe_limit) {
    if (ctl->status) return;
    const int cur = ctl->cur;
    uint32_t* filter = reinterpret_cast<uint32_t*>(B.key(cur ^ 1));
    const uint64_t n = live_count(ctl, cur);
    const double rnorm = ctl->rnorm[cur];
    const unsigned gen = ctl->gen;
    const uint64_t mask = table_mask(n, slots, load_pct);
    const uint32_t fs = filter_shift(n);
    int probes = 0;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const PKey<W> K = load_key(B.key(cur) + i);
        const uint32_t fb = filter_hash(K) >> fs;
        atomicOr(filter + (fb >> 5), 1u << (fb & 31u));
        const double c = normalised(B.coef(cur)[i], rnorm, key_is_zero(K));
        if (!table_insert(table, mask, gen, K, c, (uint32_t)i, probe_limit, &probes))
            set_status(ctl, ST_HASH_PROBE, 61);
    }
}

__device__ __forceinline__ void kahan_add(double& s, double& comp, double v) {
    const double y = __dsub_rn(v, comp);
    const double t = __dadd_rn(s, y);
    comp = __dsub_rn(__dsub_rn(t, s), y);
    s = t;
}

constexpr int kObs = 8;   // observable strings looked up together

template <int W>
__device__ __forceinline__ bool obs_is_identity(const GateArg<W>& o) {
    uint64_t q = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) q |= o.qx[w] | o.qz[w];
    return q == 0ULL;
}

// Of the pair {P, O.P}: the member without O's lowest bit (any P for O = I,
// which is its own partner).
template <int W>
__device__ __forceinline__ bool first_of_pair(const PKey<W>& P, const GateArg<W>& o) {
    uint64_t bit = 0;
    bool found = false;
#pragma unroll
    for (int w = 0; w < 2 * W; ++w) {
        const uint64_t q = w < W ? o.qx[w] : o.qz[w - W];
        const uint64_t k = w < W ? P.x[w] : P.z[w - W];
        if (!found) bit = k & q & (~q + 1ULL);
        found = found || q != 0ULL;
    }
    return bit == 0ULL;
}

template <int W>
__device__ __forceinline__ GateArg<W> obs_gate(const uint64_t* __restrict__ ox,
                                               const uint64_t* __restrict__ oz, int j) {
    GateArg<W> o;
    int yy = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        o.qx[w] = __ldg(ox + (size_t)j * W + w);
        o.qz[w] = __ldg(oz + (size_t)j * W + w);
        yy += __popcll(o.qx[w] & o.qz[w]);
    }
    o.qyy = yy & 3;
    return o;
}

// One pass over the state: purity and the commuting-pair overlap; per-block
// partials (numerator, purity) in a fixed-order tree.
template <int W>
__global__ void __launch_bounds__(kPB)
k_psd_pairs(Bufs<W> B, DevCtl* ctl, const Slot<W>* table, uint64_t slots, int load_pct,
            int probe_limit, const uint64_t* __restrict__ ox, const uint64_t* __restrict__ oz,
            const double* __restrict__ ow, int m, double* partials) {
    __shared__ double s_num[kPB], s_den[kPB];
    __shared__ uint32_t s_qi[kPB / 32][64];   // queue: term, string
    __shared__ uint32_t s_qj[kPB / 32][64];
    double num = 0.0, cn = 0.0, den = 0.0, cd = 0.0;
    if (!ctl->status) {
        const int cur = ctl->cur;
        const uint64_t n = live_count(ctl, cur);
        const double rnorm = ctl->rnorm[cur];
        const unsigned gen = ctl->gen;
        const uint64_t mask = table_mask(n, slots, load_pct);
        const uint32_t* __restrict__ filter = reinterpret_cast<const uint32_t*>(B.key(cur ^ 1));
        const uint32_t fs = filter_shift(n);
        const uint32_t lane = threadIdx.x & 31u;
        const unsigned int lt = (1u << lane) - 1u;
        uint32_t* qi = s_qi[threadIdx.x >> 5];
        uint32_t* qj = s_qj[threadIdx.x >> 5];
        uint32_t qn = 0;   // queued, the same on every lane
        int probes = 0;
        // the first `take` entries of the queue, one per lane
        auto drain = [&](uint32_t take) {
            __syncwarp();
            if (lane < take) {
                const uint64_t i = qi[lane];
                const int j = (int)qj[lane];
                const GateArg<W> o = obs_gate<W>(ox, oz, j);
                const PKey<W> P = load_key(B.key(cur) + i);
                double cr;
                if (table_find(table, mask, gen, key_xor(P, o), &cr, probe_limit, ctl, &probes)) {
                    const double cp = normalised(B.coef(cur)[i], rnorm, key_is_zero(P));
                    // twice the product, not twice the weight, which may have no
                    // double (the identity is its own partner)
                    const double w = __dmul_rn(__ldg(ow + j), __dmul_rn(cp, cr));
                    const double v = obs_is_identity(o) ? w : w + w;
                    kahan_add(num, cn, product_negative(P, o) ? -v : v);
                }
            }
            __syncwarp();
            if (lane + take < qn) {
                qi[lane] = qi[lane + take];   // take is 32 here: the halves are apart
                qj[lane] = qj[lane + take];
            }
            __syncwarp();
            qn -= take;
        };
        // whole warps iterate together
        for (uint64_t i0 = (uint64_t)blockIdx.x * kPB + (threadIdx.x & ~31u); i0 < n;
             i0 += (uint64_t)gridDim.x * kPB) {
            const uint64_t i = i0 + lane;
            PKey<W> P;
#pragma unroll
            for (int w = 0; w < W; ++w) { P.x[w] = 0; P.z[w] = 0; }
            if (i < n) {
                P = load_key(B.key(cur) + i);
                const double cp = normalised(B.coef(cur)[i], rnorm, key_is_zero(P));
                kahan_add(den, cd, __dmul_rn(cp, cp));
            }
            for (int j0 = 0; j0 < m; j0 += kObs) {
                // the filter's words of a group of strings, all in flight
                uint32_t word[kObs];
#pragma unroll
                for (int u = 0; u < kObs; ++u) {
                    const GateArg<W> o = obs_gate<W>(ox, oz, j0 + u < m ? j0 + u : m - 1);
                    const uint32_t fb = filter_hash(key_xor(P, o)) >> fs;
                    const bool ask = i < n && j0 + u < m && first_of_pair(P, o) && commutes(P, o);
                    word[u] = ask ? __ldg(filter + (fb >> 5)) >> (fb & 31u) : 0u;
                }
#pragma unroll
                for (int u = 0; u < kObs; ++u) {
                    const bool hit = word[u] & 1u;
                    const unsigned int h = __ballot_sync(0xffffffffu, hit);
                    if (!h) continue;
                    if (hit) {
                        qi[qn + __popc(h & lt)] = (uint32_t)i;
                        qj[qn + __popc(h & lt)] = (uint32_t)(j0 + u);
                    }
                    qn += __popc(h);
                    if (qn >= 32u) drain(32u);
                }
            }
        }
        if (qn) drain(qn);
    }
    s_num[threadIdx.x] = num;
    s_den[threadIdx.x] = den;
    __syncthreads();
    for (int o = kPB / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            s_num[threadIdx.x] = __dadd_rn(s_num[threadIdx.x], s_num[threadIdx.x + o]);
            s_den[threadIdx.x] = __dadd_rn(s_den[threadIdx.x], s_den[threadIdx.x + o]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = s_num[0];
        partials[2 * blockIdx.x + 1] = s_den[0];
    }
}

// The blocks' partials, compensated per thread over a fixed stride, then in a
// fixed tree (one thread adding 1,216 of them in turn took 376 us: every step
// of a compensated sum waits for the last); the ratio; the next gate gets a
// fresh table generation.
__global__ void __launch_bounds__(kPB)
k_psd_final(DevCtl* ctl, const double* partials, int n_part, double* out) {
    __shared__ double s_s[2][kPB], s_c[2][kPB];
    double num = 0.0, cn = 0.0, den = 0.0, cd = 0.0;
    for (int b = threadIdx.x; b < n_part; b += kPB) {
        kahan_add(num, cn, partials[2 * b]);
        kahan_add(den, cd, partials[2 * b + 1]);
    }
    s_s[0][threadIdx.x] = num;
    s_c[0][threadIdx.x] = cn;
    s_s[1][threadIdx.x] = den;
    s_c[1][threadIdx.x] = cd;
    __syncthreads();
    for (int o = kPB / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                // add (sum_b - comp_b) into (sum_a, comp_a), one compensated step
                const double a = s_s[k][threadIdx.x];
                const double y = __dsub_rn(s_s[k][threadIdx.x + o],
                                           __dadd_rn(s_c[k][threadIdx.x], s_c[k][threadIdx.x + o]));
                const double t = __dadd_rn(a, y);
                s_c[k][threadIdx.x] = __dsub_rn(__dsub_rn(t, a), y);
                s_s[k][threadIdx.x] = t;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    out[0] = __ddiv_rn(s_s[0][0], s_s[1][0]);
    out[1] = s_s[0][0];
    out[2] = s_s[1][0];
    if (!ctl->status) {
        ctl->gen = ctl->gen + 1u;
        if (ctl->gen == 0u) set_status(ctl, ST_STATE, 62);
    }
}

template <int W>
static cudaError_t psd_w(const DeviceState& s, const uint64_t* d_ox, const uint64_t* d_oz,
                         const double* d_ow, int m, double* d_partials, int n_part,
                         double* d_out, cudaStream_t st) {
    // stale contents (the top-M select borrows this memory) must not read as
    // tags: clear the table first
    const size_t slot = W == 1 ? 32 : 64;
    cudaError_t e = cudaMemsetAsync(s.table, 0, (size_t)s.table_slots * slot, st);
    if (e != cudaSuccess) return e;
    // the filter lies in the other buffer's keys, free between gates: two bytes
    // a term at most, and those hold 16 or more (which of the two is the other
    // one the device knows)
    const size_t fbytes = ((size_t)s.cap_M * 2 + 15) / 16 * 16;
    k_psd_begin<<<s.num_sms * 4, 256, 0, st>>>(psd_bufs<W>(s), s.ctl, fbytes);
    Slot<W>* table = static_cast<Slot<W>*>(s.table);
    k_psd_build<W><<<s.num_sms * 8, kPB, 0, st>>>(psd_bufs<W>(s), s.ctl, table, s.table_slots,
                                                 s.load_pct, s.probe_limit);
    k_psd_pairs<W><<<n_part, kPB, 0, st>>>(psd_bufs<W>(s), s.ctl, table, s.table_slots,
                                          s.load_pct, s.probe_limit, d_ox, d_oz, d_ow, m,
                                          d_partials);
    k_psd_final<<<1, kPB, 0, st>>>(s.ctl, d_partials, n_part, d_out);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_expect_psd(const DeviceState& s, const uint64_t* d_ox, const uint64_t* d_oz,
                              const double* d_ow, int m, double* d_partials, int n_part,
                              double* d_out, cudaStream_t st) {
    return s.W == 1 ? psd_w<1>(s, d_ox, d_oz, d_ow, m, d_partials, n_part, d_out, st)
                    : psd_w<2>(s, d_ox, d_oz, d_ow, m, d_partials, n_part, d_out, st);
}

}  // namespace itpp
