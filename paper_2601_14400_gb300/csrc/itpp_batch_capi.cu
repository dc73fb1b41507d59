// itpp_batch_capi.cu -- C ABI of the batched propagation (include/itpp.h):
// many independent ITPP instances advanced together: a team of CTAs per
// instance in one launch (merge_path 0), or shared launches replayed as one CUDA
// graph per Trotter layer (merge_path 2).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "itpp.h"
#include "itpp_common.cuh"
#include "itpp_launch.h"
#include "itpp_run.cuh"

using namespace itpp;

struct itpp_batch_ctx {
    BatchState s;
    std::vector<int> n;        // sites per instance
    std::vector<int> n_gates;  // gates per layer per instance
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    cudaGraphExec_t layer = nullptr;
    std::vector<int> h_status;          // [B] of a probed shape
    itpp_status sticky = ITPP_OK;
    void* obs_mem = nullptr;
    size_t obs_bytes = 0;
    uint64_t launches = 0;
    std::vector<unsigned char> h_ctl;   // one DevCtl head, for reads
    int load_floor = 50;                // lowest table load the allocation allows
    // run kernel: gates, sites, teams, their shared blocks, threshold drifts
    void* run_gates = nullptr;          // RunGate<W>[B * max_gates]
    int* run_sites = nullptr;           // [B]
    uint4* run_teams = nullptr;         // [grid]
    void* run_shared = nullptr;
    long long* run_drift = nullptr;     // [B * (max_gates + 1)]
    int run_grid = 0, run_n_teams = 0, run_fit_ctas = 0;
    bool run_wide = false;
    int max_weight = 0;
    bool target_fixed = false;          // partition size given by the caller
};

namespace {

constexpr size_t kHead = offsetof(DevCtl, sel_hist);
constexpr int kTargetMin = 150;   // smallest mean partition size the autotuner tries
constexpr int kMinPartMin = 64;   // smallest lower limit of it

uint64_t next_pow2(uint64_t v) {
    uint64_t s = 1;
    while (s < v) s <<= 1;
    return s;
}

bool bits_ok(int n, int W, const uint64_t* x) {
    for (int w = 0; w < W; ++w) {
        const int lo = 64 * w;
        if (n >= lo + 64) continue;
        const uint64_t top = (n <= lo) ? ~0ULL : (~0ULL << (n - lo));
        if (x[w] & top) return false;
    }
    return true;
}

void free_batch(itpp_batch_ctx* h) {
    BatchState& s = h->s;
    for (int i = 0; i < 2; ++i) {
        if (s.keys[i]) cudaFree(s.keys[i]);
        if (s.coef[i]) cudaFree(s.coef[i]);
    }
    if (s.table) cudaFree(s.table);
    if (s.part_keys) cudaFree(s.part_keys);
    if (s.part_coef) cudaFree(s.part_coef);
    if (s.part_cursor) cudaFree(s.part_cursor);
    if (h->run_gates) cudaFree(h->run_gates);
    if (h->run_sites) cudaFree(h->run_sites);
    if (h->run_teams) cudaFree(h->run_teams);
    if (h->run_shared) cudaFree(h->run_shared);
    if (h->run_drift) cudaFree(h->run_drift);
    if (s.ctls) cudaFree(s.ctls);
    if (s.gates) cudaFree(s.gates);
    if (s.n_gates) cudaFree(s.n_gates);
    if (s.item_prefix) cudaFree(s.item_prefix);
    if (h->obs_mem) cudaFree(h->obs_mem);
    if (h->layer) cudaGraphExecDestroy(h->layer);
    if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
}

// Single-propagation view of instance b (for export, expectation, import).
DeviceState view(const itpp_batch_ctx* h, int b) {
    const BatchState& s = h->s;
    DeviceState d;
    d.n = h->n[(size_t)b];
    d.W = s.W;
    const size_t kb = (size_t)s.buf_cap * 16 * s.W;
    for (int i = 0; i < 2; ++i) {
        d.keys[i] = static_cast<char*>(s.keys[i]) + (size_t)b * kb;
        d.coef[i] = s.coef[i] + (size_t)b * s.buf_cap;
    }
    d.table = static_cast<char*>(s.table) + (size_t)b * s.table_slots * (s.W == 1 ? 32 : 64);
    d.table_slots = s.table_slots;
    d.ctl = s.ctls + b;
    d.cap_M = s.cap_M;
    d.buf_cap = s.buf_cap;
    d.cap_policy = s.cap_policy;
    d.delta = s.delta;
    d.num_sms = s.num_sms;
    d.load_pct = s.load_pct;
    d.probe_limit = s.probe_limit;
    return d;
}

template <int W>
void fill_gate(void* dst, const uint64_t* qx, const uint64_t* qz, double alpha, double dtau,
               int max_weight) {
    GateArg<W> g;
    std::memset(&g, 0, sizeof(g));
    int yy = 0;
    for (int w = 0; w < W; ++w) {
        g.qx[w] = qx[w];
        g.qz[w] = qz[w];
        uint64_t v = qx[w] & qz[w];
        while (v) { v &= v - 1; ++yy; }
    }
    const double theta = alpha * dtau;
    g.ch = std::cosh(theta);
    g.msh = -std::sinh(theta);
    g.qyy = yy & 3;
    g.maxw = max_weight ? max_weight : (1 << 30);
    std::memcpy(dst, &g, sizeof(g));
}

itpp_status read_head(itpp_batch_ctx* h, int b, DevCtl* out) {
    if (cudaMemcpyAsync(out, h->s.ctls + b, kHead, cudaMemcpyDeviceToHost, h->stream) !=
            cudaSuccess ||
        cudaStreamSynchronize(h->stream) != cudaSuccess) {
        h->sticky = ITPP_ERR_CUDA;
        return ITPP_ERR_CUDA;
    }
    return ITPP_OK;
}

// Reset every instance to the identity (statistics cleared).
itpp_status reset_all(itpp_batch_ctx* h) {
    const BatchState& s = h->s;
    for (int b = 0; b < s.B; ++b)
        if (launch_reset_identity(view(h, b), h->stream) != cudaSuccess) return ITPP_ERR_CUDA;
    return ITPP_OK;
}

// Which CTAs work on which instance: every instance its team, of a size in
// proportion to its gates (a layer ends with the slowest team), at most one
// CTA per smallest partition; with more instances than CTAs every CTA is a
// team and takes one instance after another.
itpp_status plan_teams(itpp_batch_ctx* h) {
    const BatchState& s = h->s;
    const int per_sm = s.team_ctas > 0 && s.team_ctas < h->run_fit_ctas ? s.team_ctas : h->run_fit_ctas;
    const long long ctas = (long long)s.num_sms * per_sm;
    std::vector<uint4> t;
    if ((long long)s.B >= ctas) {
        for (long long c = 0; c < ctas; ++c)
            t.push_back(make_uint4((unsigned)c, 0u, 1u, (unsigned)ctas));
        h->run_n_teams = (int)ctas;
    } else {
        long long sum = 0;
        for (int g : h->n_gates) sum += g;
        const long long most = (long long)(s.cap_M / (uint64_t)s.min_part) + 1;
        for (int b = 0; b < s.B; ++b) {
            long long size = 1 + (sum ? (ctas - s.B) * h->n_gates[(size_t)b] / sum : 0);
            size = std::min(size, most);
            for (long long r = 0; r < size; ++r)
                t.push_back(make_uint4((unsigned)b, (unsigned)r, (unsigned)size, (unsigned)s.B));
        }
        h->run_n_teams = s.B;
    }
    h->run_grid = (int)t.size();
    return cudaMemcpyAsync(h->run_teams, t.data(), t.size() * sizeof(uint4), cudaMemcpyHostToDevice,
                           h->stream) == cudaSuccess &&
                   cudaStreamSynchronize(h->stream) == cudaSuccess
               ? ITPP_OK : ITPP_ERR_CUDA;
}

// n_layers layers of every instance in one launch.
template <int W>
itpp_status run_batch(itpp_batch_ctx* h, int n_layers) {
    const BatchState& s = h->s;
    RunArgs<W> a{};
    for (int i = 0; i < 2; ++i) {
        a.k[i] = static_cast<PKey<W>*>(s.keys[i]);
        a.c[i] = s.coef[i];
    }
    a.kp = static_cast<PKey<W>*>(s.part_keys);
    a.cp = s.part_coef;
    a.cnt = s.part_cursor;
    a.ctl = s.ctls;
    a.scratch = s.table;
    a.shared = h->run_shared;
    a.drift = h->run_drift;
    a.n = h->run_sites;
    a.gates = static_cast<const RunGate<W>*>(h->run_gates);
    a.n_gates = s.n_gates;
    a.team_of = h->run_teams;
    a.buf_stride = s.buf_cap;
    a.part_stride = s.part_cap;
    a.scratch_stride = s.table_slots * (W == 1 ? 32 : 64);
    a.shared_stride = run_shared_bytes();
    a.buf_cap = s.buf_cap;
    a.home_cap = std::min(s.part_cap, s.buf_cap);
    a.cand_cap = run_list_cap<W>(a.scratch_stride, a.home_cap);
    a.tie_off = run_tie_off(a.cand_cap);
    a.cap_M = s.cap_M;
    a.cand_hi = std::max<uint64_t>(1024, s.cap_M / 16);
    std::memcpy(&a.delta_bits, &s.delta, sizeof a.delta_bits);
    a.part_max = s.part_max;
    a.drift_stride = s.max_gates + 1;
    a.drift_gates = s.max_gates;
    a.B = s.B;
    a.max_gates = s.max_gates;
    a.n_layers = n_layers;
    a.target = s.part_target;
    a.min_part = s.min_part;
    a.cap_policy = s.cap_policy;
    a.maxw = h->max_weight ? h->max_weight : (1 << 30);
    static const RunChunk<W> none{};
    if (cudaMemset2DAsync(h->run_shared, a.shared_stride, 0, run_shared_head(),
                          (size_t)h->run_n_teams, h->stream) != cudaSuccess ||
        launch_run<W>(a, none, h->run_grid, h->run_wide, h->stream) != cudaSuccess) {
        cudaGetLastError();
        return ITPP_ERR_CUDA;
    }
    h->launches += 1;
    return ITPP_OK;
}

itpp_status run_layers(itpp_batch_ctx* h, int n_layers) {
    // at most a few thousand gates a launch (it holds the GPU's CTA slots)
    const int most = std::max(1, 4096 / std::max(1, h->s.max_gates));
    for (int l = 0; l < n_layers && h->s.max_gates > 0; l += most) {
        const int nl = std::min(most, n_layers - l);
        const itpp_status st = h->s.W == 1 ? run_batch<1>(h, nl) : run_batch<2>(h, nl);
        if (st) return st;
    }
    return ITPP_OK;
}

// The gates of every instance with the windows that start at each.
template <int W>
void fill_run_gates(RunGate<W>* dst, int max_g, const GateArg<W>* src, const std::vector<int>& n) {
    for (size_t b = 0; b < n.size(); ++b) {
        RunGate<W>* g = dst + b * (size_t)max_g;
        for (int j = 0; j < n[b]; ++j) {
            const GateArg<W>& q = src[b * (size_t)max_g + (size_t)j];
            for (int w = 0; w < W; ++w) {
                g[j].qx[w] = q.qx[w];
                g[j].qz[w] = q.qz[w];
            }
            g[j].ch = q.ch;
            g[j].msh = q.msh;
        }
        plan_run_windows(g, n[b]);
    }
}

// Capture one Trotter layer (every gate step, all instances per launch) as
// the handle's graph, if it has none.
itpp_status capture_layer(itpp_batch_ctx* h) {
    if (h->layer || h->s.merge_path == 0) return ITPP_OK;
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
        return ITPP_ERR_CUDA;
    cudaError_t e = cudaSuccess;
    for (int step = 0; step < h->s.max_gates && e == cudaSuccess; ++step)
        e = launch_batch_step(h->s, step, h->stream);
    cudaError_t e2 = cudaStreamEndCapture(h->stream, &g);
    if (e != cudaSuccess || e2 != cudaSuccess || !g) {
        if (g) cudaGraphDestroy(g);
        cudaGetLastError();
        return ITPP_ERR_CUDA;
    }
    e = cudaGraphInstantiate(&h->layer, g, 0);
    cudaGraphDestroy(g);
    return e == cudaSuccess ? ITPP_OK : ITPP_ERR_CUDA;
}

// Time probe_layers layers from the identity with the current shape; *failed
// counts the instances that ended with an error (and may have stopped early).
itpp_status time_shape(itpp_batch_ctx* h, int probe_layers, double* ms, int* failed) {
    if (h->layer) {
        cudaGraphExecDestroy(h->layer);
        h->layer = nullptr;
    }
    if (reset_all(h) != ITPP_OK || cudaStreamSynchronize(h->stream) != cudaSuccess)
        return ITPP_ERR_CUDA;
    // capture the layer graph outside the timed region
    if (capture_layer(h) != ITPP_OK) return ITPP_ERR_CUDA;
    cudaEvent_t a, b;
    if (cudaEventCreate(&a) != cudaSuccess) return ITPP_ERR_CUDA;
    if (cudaEventCreate(&b) != cudaSuccess) { cudaEventDestroy(a); return ITPP_ERR_CUDA; }
    cudaEventRecord(a, h->stream);
    bool ok = true;
    if (h->s.merge_path == 0) ok = run_layers(h, probe_layers) == ITPP_OK;
    else for (int l = 0; l < probe_layers && ok; ++l) ok = cudaGraphLaunch(h->layer, h->stream) == cudaSuccess;
    cudaEventRecord(b, h->stream);
    float f = 0.f;
    ok = cudaEventSynchronize(b) == cudaSuccess && cudaEventElapsedTime(&f, a, b) == cudaSuccess && ok;
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (!ok) return ITPP_ERR_CUDA;
    *ms = f;
    if (cudaMemcpy2DAsync(h->h_status.data(), sizeof(int), &h->s.ctls->status, sizeof(DevCtl),
                          sizeof(int), (size_t)h->s.B, cudaMemcpyDeviceToHost, h->stream) !=
            cudaSuccess ||
        cudaStreamSynchronize(h->stream) != cudaSuccess)
        return ITPP_ERR_CUDA;
    *failed = 0;
    for (int v : h->h_status) *failed += v != 0;
    return ITPP_OK;
}

}  // namespace

extern "C" {

itpp_status itpp_batch_create(int B, const int* n, const int* n_gates, const uint64_t* gate_x,
                              const uint64_t* gate_z, const double* alpha, double dtau,
                              const itpp_params* p, void* cuda_stream, itpp_batch_handle* out) {
    if (!out || !p || !n || !n_gates || B < 1 || B > 65535) return ITPP_ERR_ARG;
    if (!std::isfinite(dtau) || !(p->delta >= 0.0) || !std::isfinite(p->delta)) return ITPP_ERR_ARG;
    if (p->cap_M < 1 || p->cap_M > (1ULL << 31)) return ITPP_ERR_ARG;
    if (p->cap_policy != 0 && p->cap_policy != 1) return ITPP_ERR_ARG;
    if (p->merge_path != 0 && p->merge_path != 2) return ITPP_ERR_ARG;
    if (p->partition_target != 0 && (p->partition_target < 64 || p->partition_target > 2048))
        return ITPP_ERR_ARG;
    if (p->max_weight < 0 || p->max_weight > 128) return ITPP_ERR_ARG;
    int max_n = 0, max_g = 0;
    long long total_g = 0;
    for (int b = 0; b < B; ++b) {
        if (n[b] < 1 || n[b] > 128 || n_gates[b] < 0) return ITPP_ERR_ARG;
        max_n = n[b] > max_n ? n[b] : max_n;
        max_g = n_gates[b] > max_g ? n_gates[b] : max_g;
        total_g += n_gates[b];
    }
    if (total_g > 0 && (!gate_x || !gate_z || !alpha)) return ITPP_ERR_ARG;
    const int W = (max_n + 63) / 64;
    {
        long long k = 0;
        for (int b = 0; b < B; ++b)
            for (int j = 0; j < n_gates[b]; ++j, ++k) {
                if (!std::isfinite(alpha[k])) return ITPP_ERR_ARG;
                if (!std::isfinite(std::cosh(alpha[k] * dtau)) ||
                    !std::isfinite(std::sinh(alpha[k] * dtau)))
                    return ITPP_ERR_ARG;   // the gate's weights overflow
                if (!bits_ok(n[b], W, gate_x + k * W) || !bits_ok(n[b], W, gate_z + k * W))
                    return ITPP_ERR_ARG;
            }
    }
    itpp_batch_ctx* h = new (std::nothrow) itpp_batch_ctx;
    if (!h) return ITPP_ERR_ALLOC;
    h->n.assign(n, n + B);
    h->n_gates.assign(n_gates, n_gates + B);
    h->stream = static_cast<cudaStream_t>(cuda_stream);
    if (!h->stream) {
        if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete h;
            return ITPP_ERR_CUDA;
        }
        h->own_stream = true;
    }
    BatchState& s = h->s;
    s.B = B;
    s.W = W;
    s.max_gates = max_g;
    s.cap_M = p->cap_M;
    s.buf_cap = 2 * p->cap_M;
    s.cap_policy = p->cap_policy;
    h->max_weight = p->max_weight;
    s.merge_path = p->merge_path;
    s.delta = p->delta + 0.0;   // -0 becomes +0 (the threshold compares bit patterns)
    s.load_pct = p->table_load_pct ? p->table_load_pct : 50;
    if (s.load_pct < 10 || s.load_pct > 75) { free_batch(h); delete h; return ITPP_ERR_ARG; }
    if (s.merge_path == 0) {
        // a home per instance, and cursors for the smallest partition sizes the
        // autotuner tries
        h->target_fixed = p->partition_target != 0;
        s.part_target = p->partition_target ? p->partition_target : partition_target_default(W);
        s.min_part = run_min_part(s.part_target);
        s.part_cap = 2 * p->cap_M + p->cap_M / 2 + 4096;
        s.part_cap += s.part_cap & 1ULL;
        const int t_min = std::min(h->target_fixed ? s.part_target : kTargetMin, s.part_target);
        s.part_max = partition_max(p->cap_M, t_min) + 1;
        h->run_wide = (uint64_t)B * p->cap_M > kRunWide;
        h->run_fit_ctas = run_fit(W, h->run_wide);
    }
    // auto sizing leaves room for the autotuner to try loads down to 25 %
    const int load_for_size = p->table_load_pct ? (s.load_pct < 50 ? s.load_pct : 50) : 25;
    h->load_floor = load_for_size;
    const uint64_t need = (p->cap_M * 100 + load_for_size - 1) / load_for_size;
    s.table_slots = next_pow2(need < 256 ? 256 : need);
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    s.num_sms = sms;
    if (s.merge_path == 0)   // a partition for every CTA of a team
        s.part_max = (uint32_t)std::max<uint64_t>(
            s.part_max, std::min<uint64_t>((uint64_t)sms * h->run_fit_ctas,
                                           p->cap_M / (uint64_t)kMinPartMin + 1) + 1);

    const size_t gsz = W == 1 ? sizeof(GateArg<1>) : sizeof(GateArg<2>);
    std::vector<unsigned char> gates((size_t)B * (max_g > 0 ? max_g : 1) * gsz, 0);
    {
        long long k = 0;
        for (int b = 0; b < B; ++b)
            for (int j = 0; j < n_gates[b]; ++j, ++k) {
                void* dst = gates.data() + ((size_t)b * max_g + j) * gsz;
                if (W == 1) fill_gate<1>(dst, gate_x + k * W, gate_z + k * W, alpha[k], dtau, p->max_weight);
                else fill_gate<2>(dst, gate_x + k * W, gate_z + k * W, alpha[k], dtau, p->max_weight);
            }
    }
    const size_t slot = W == 1 ? 32 : 64;
    bool ok = true;
    for (int i = 0; i < 2 && ok; ++i) {
        ok &= cudaMalloc(&s.keys[i], (size_t)B * s.buf_cap * 16 * W) == cudaSuccess;
        ok &= ok && cudaMalloc(reinterpret_cast<void**>(&s.coef[i]), (size_t)B * s.buf_cap * 8) ==
                        cudaSuccess;
    }
    ok &= ok && cudaMalloc(&s.table, (size_t)B * s.table_slots * slot) == cudaSuccess;
    if (s.merge_path == 0) {
        ok &= ok && cudaMalloc(&s.part_keys, (size_t)B * s.part_cap * 16 * W) == cudaSuccess;
        ok &= ok && cudaMalloc(reinterpret_cast<void**>(&s.part_coef),
                               ((size_t)B * s.part_cap + 2) * 8) == cudaSuccess;
        ok &= ok && cudaMalloc(reinterpret_cast<void**>(&s.part_cursor),
                               (size_t)B * 3 * s.part_max * kRunPad * sizeof(unsigned int)) ==
                        cudaSuccess;
        const size_t ctas = (size_t)sms * h->run_fit_ctas;
        const size_t rg = W == 1 ? sizeof(RunGate<1>) : sizeof(RunGate<2>);
        const size_t nd = (size_t)B * (max_g + 1) * sizeof(long long);
        ok &= ok && cudaMalloc(&h->run_gates, (size_t)B * (max_g > 0 ? max_g : 1) * rg) == cudaSuccess;
        ok &= ok && cudaMalloc(reinterpret_cast<void**>(&h->run_sites), (size_t)B * sizeof(int)) ==
                        cudaSuccess;
        ok &= ok && cudaMalloc(reinterpret_cast<void**>(&h->run_teams), ctas * sizeof(uint4)) ==
                        cudaSuccess;
        ok &= ok && cudaMalloc(&h->run_shared, std::min<size_t>(ctas, (size_t)B) *
                                                   run_shared_bytes()) == cudaSuccess;
        ok &= ok && cudaMalloc(reinterpret_cast<void**>(&h->run_drift), nd) == cudaSuccess;
        ok &= ok && cudaMemsetAsync(h->run_drift, 0, nd, h->stream) == cudaSuccess;
    }
    ok &= ok && cudaMalloc(reinterpret_cast<void**>(&s.ctls), (size_t)B * sizeof(DevCtl)) == cudaSuccess;
    ok &= ok && cudaMalloc(&s.gates, gates.size()) == cudaSuccess;
    ok &= ok && cudaMalloc(reinterpret_cast<void**>(&s.n_gates), (size_t)B * sizeof(int)) == cudaSuccess;
    ok &= ok && cudaMalloc(reinterpret_cast<void**>(&s.item_prefix),
                           4 * (size_t)(B + 1) * sizeof(unsigned long long)) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        free_batch(h);
        delete h;
        return ITPP_ERR_ALLOC;
    }
    s.tile_prefix = s.item_prefix + (B + 1);
    s.cap_prefix = s.tile_prefix + (B + 1);
    s.ccap_prefix = s.cap_prefix + (B + 1);
    ok &= cudaMemcpyAsync(s.gates, gates.data(), gates.size(), cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
    ok &= cudaMemcpyAsync(s.n_gates, n_gates, (size_t)B * sizeof(int), cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
    ok &= cudaMemsetAsync(s.table, 0, (size_t)B * s.table_slots * slot, h->stream) == cudaSuccess;
    ok &= cudaMemsetAsync(s.ctls, 0, (size_t)B * sizeof(DevCtl), h->stream) == cudaSuccess;
    ok &= cudaMemsetAsync(s.item_prefix, 0, 4 * (size_t)(B + 1) * sizeof(unsigned long long), h->stream) == cudaSuccess;
    std::vector<unsigned char> rgates;
    if (s.merge_path == 0 && ok) {
        const size_t rg = W == 1 ? sizeof(RunGate<1>) : sizeof(RunGate<2>);
        rgates.assign((size_t)B * (max_g > 0 ? max_g : 1) * rg, 0);
        if (W == 1)
            fill_run_gates<1>(reinterpret_cast<RunGate<1>*>(rgates.data()), max_g,
                              reinterpret_cast<const GateArg<1>*>(gates.data()), h->n_gates);
        else
            fill_run_gates<2>(reinterpret_cast<RunGate<2>*>(rgates.data()), max_g,
                              reinterpret_cast<const GateArg<2>*>(gates.data()), h->n_gates);
        ok &= cudaMemcpyAsync(h->run_gates, rgates.data(), rgates.size(), cudaMemcpyHostToDevice,
                              h->stream) == cudaSuccess;
        ok &= cudaMemcpyAsync(h->run_sites, n, (size_t)B * sizeof(int), cudaMemcpyHostToDevice,
                              h->stream) == cudaSuccess;
        ok &= plan_teams(h) == ITPP_OK;
    }
    for (int b = 0; b < B && ok; ++b) {
        DeviceState d = view(h, b);
        ok &= cudaMemcpyAsync(&d.ctl->buf_cap, &s.buf_cap, sizeof(s.buf_cap),
                              cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
        ok &= launch_reset_identity(d, h->stream) == cudaSuccess;
    }
    ok &= cudaStreamSynchronize(h->stream) == cudaSuccess;
    if (!ok) {
        free_batch(h);
        delete h;
        return ITPP_ERR_CUDA;
    }
    h->h_ctl.resize(sizeof(DevCtl));
    h->h_status.resize((size_t)B);
    *out = h;
    return ITPP_OK;
}

itpp_status itpp_batch_destroy(itpp_batch_handle h) {
    if (!h) return ITPP_OK;
    cudaStreamSynchronize(h->stream);
    free_batch(h);
    delete h;
    return ITPP_OK;
}

itpp_status itpp_batch_apply_trotter_layer(itpp_batch_handle h, int n_layers) {
    if (!h || n_layers < 0) return ITPP_ERR_ARG;
    if (h->sticky) return h->sticky;
    if (h->s.merge_path == 0) {
        const itpp_status st = run_layers(h, n_layers);
        return st == ITPP_OK ? ITPP_OK : h->sticky = st;
    }
    // one layer (every gate step, all instances per launch) as a graph
    if (n_layers > 0 && capture_layer(h) != ITPP_OK) return h->sticky = ITPP_ERR_CUDA;
    for (int l = 0; l < n_layers; ++l) {
        if (cudaGraphLaunch(h->layer, h->stream) != cudaSuccess) return h->sticky = ITPP_ERR_CUDA;
        h->launches += (uint64_t)h->s.max_gates * batch_step_launches(h->s);
    }
    return ITPP_OK;
}

itpp_status itpp_batch_autotune(itpp_batch_handle h, int probe_layers, itpp_tune_result* out) {
    if (!h || probe_layers < 1) return ITPP_ERR_ARG;
    if (h->sticky) return h->sticky;
    BatchState& s = h->s;
    const bool part = s.merge_path == 0;
    // a shape: block, CTAs per SM (partitioned: 0 = what fits) or of the
    // branch-emit kernel, CTAs per SM of the table build or (partitioned) the
    // smallest mean partition in units of 16 terms, table load (global table)
    // or mean partition size (partitioned)
    struct Shape { int mb, mg, ig, load, target; };
    auto install = [&](const Shape& c) -> itpp_status {
        s.main_block = c.mb;
        if (part) {
            s.team_ctas = c.mg;
            s.min_part = h->target_fixed ? std::min(16 * c.ig, c.target) : 16 * c.ig;
            s.part_target = c.target;
            return plan_teams(h);
        }
        s.main_grid = c.mg;
        s.insert_grid = c.ig;
        s.load_pct = c.load;
        return ITPP_OK;
    };
    Shape best = part ? Shape{256, 0, 8, 0, s.part_target}
                      : Shape{256, 4, 8, 50 < h->load_floor ? h->load_floor : 50, 0};
    double best_ms = 0, default_ms = 0;
    int tried = 0, best_failed = 0;
    itpp_status st = install(best);
    if (!st) st = time_shape(h, probe_layers, &best_ms, &best_failed);
    if (st) return h->sticky = st;
    default_ms = best_ms;
    ++tried;
    // an instance that stops on an error is fast: a shape with more of them than
    // the best one so far is not better, whatever its time
    auto try_shape = [&](Shape c) -> itpp_status {
        double ms = 0;
        int failed = 0;
        itpp_status e = install(c);
        if (!e) e = time_shape(h, probe_layers, &ms, &failed);
        if (e) return e;
        ++tried;
        if (failed < best_failed || (failed == best_failed && ms < best_ms)) {
            best_ms = ms;
            best_failed = failed;
            best = c;
        }
        return ITPP_OK;
    };
    // one parameter at a time, each from the best shape so far
    const int blocks[3] = {128, 256, 512};
    if (!part) for (int v : blocks) if (v != best.mb) { Shape c = best; c.mb = v; if ((st = try_shape(c))) return h->sticky = st; }
    if (part) {
        const int mgs[4] = {1, 2, 3, 0}, sgs[3] = {4, 8, 16};
        const int t1[4] = {350, 500, 700, 1000}, t2[3] = {150, 300, 450};
        for (int v : mgs) if (v != best.mg) { Shape c = best; c.mg = v; if ((st = try_shape(c))) return h->sticky = st; }
        for (int v : sgs) if (v != best.ig) { Shape c = best; c.ig = v; if ((st = try_shape(c))) return h->sticky = st; }
        if (!h->target_fixed) {
            const int* ts = s.W == 1 ? t1 : t2;
            const int nt = s.W == 1 ? 4 : 3;
            for (int k = 0; k < nt; ++k)
                if (ts[k] != best.target) { Shape c = best; c.target = ts[k]; if ((st = try_shape(c))) return h->sticky = st; }
        }
    } else {
        const int grids[3] = {2, 4, 8}, igrids[3] = {4, 8, 16};
        const int loads[4] = {25, 35, 50, 65};
        for (int v : grids) if (v != best.mg) { Shape c = best; c.mg = v; if ((st = try_shape(c))) return h->sticky = st; }
        for (int v : igrids) if (v != best.ig) { Shape c = best; c.ig = v; if ((st = try_shape(c))) return h->sticky = st; }
        for (int v : loads)
            if (v != best.load && v >= h->load_floor) { Shape c = best; c.load = v; if ((st = try_shape(c))) return h->sticky = st; }
    }
    if ((st = install(best))) return h->sticky = st;
    if (h->layer) {
        cudaGraphExecDestroy(h->layer);
        h->layer = nullptr;
    }
    // the chosen shape's layer graph, ready for the next apply
    if (reset_all(h) != ITPP_OK || capture_layer(h) != ITPP_OK ||
        cudaStreamSynchronize(h->stream) != cudaSuccess)
        return h->sticky = ITPP_ERR_CUDA;
    if (out) {
        std::memset(out, 0, sizeof(*out));
        out->main_block = best.mb;
        out->main_grid = part ? (best.mg ? best.mg : h->run_fit_ctas) : best.mg;
        out->insert_grid = best.ig;
        out->table_load_pct = part ? 0 : best.load;
        out->partition_target = part ? best.target : 0;
        out->ms_per_probe = best_ms;
        out->ms_per_probe_default = default_ms;
        out->candidates = tried;
    }
    return ITPP_OK;
}

itpp_status itpp_batch_get_counts(itpp_batch_handle h, uint64_t* counts, int* statuses) {
    if (!h || !counts) return ITPP_ERR_ARG;
    DevCtl* c = reinterpret_cast<DevCtl*>(h->h_ctl.data());
    itpp_status first = ITPP_OK;
    for (int b = 0; b < h->s.B; ++b) {
        itpp_status st = read_head(h, b, c);
        if (st) return st;
        counts[b] = c->count[c->cur];
        if (statuses) statuses[b] = c->status;
        if (!first && c->status) first = (itpp_status)c->status;
    }
    return first;
}

itpp_status itpp_batch_synchronize(itpp_batch_handle h) {
    if (!h) return ITPP_ERR_ARG;
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) return h->sticky = ITPP_ERR_CUDA;
    std::vector<uint64_t> counts((size_t)h->s.B);
    return itpp_batch_get_counts(h, counts.data(), nullptr);
}

itpp_status itpp_batch_get_stats(itpp_batch_handle h, int b, itpp_stats* o) {
    if (!h || !o || b < 0 || b >= h->s.B) return ITPP_ERR_ARG;
    DevCtl* c = reinterpret_cast<DevCtl*>(h->h_ctl.data());
    itpp_status st = read_head(h, b, c);
    if (st) return st;
    o->gates_applied = c->stat_gates;
    o->terms_in = c->stat_in;
    o->terms_out = c->stat_out;
    o->peak_terms = c->stat_peak;
    o->cap_events = c->stat_cap;
    o->count = c->count[c->cur];
    o->table_probes = c->stat_probes;
    o->repartitions = c->stat_scatters;
    o->select_candidates = c->stat_cands;
    o->select_range = c->stat_range;
    o->select_full = c->stat_sel_full;
    o->long_partitions = c->stat_long;
    o->merge_retries = c->stat_retry;
    o->error_site = c->status ? c->err_info : 0;
    o->kernel_launches = h->launches;
    return (itpp_status)c->status;
}

itpp_status itpp_batch_get_terms(itpp_batch_handle h, int b, uint64_t* x, uint64_t* z, double* cc,
                                 uint64_t capacity, uint64_t* count) {
    if (!h || !count || b < 0 || b >= h->s.B) return ITPP_ERR_ARG;
    DevCtl* c = reinterpret_cast<DevCtl*>(h->h_ctl.data());
    itpp_status st = read_head(h, b, c);
    if (st) return st;
    if (c->status) return (itpp_status)c->status;
    const uint64_t n = c->count[c->cur];
    *count = n;
    if (capacity < n) return ITPP_ERR_CAPACITY;
    if (n == 0) return ITPP_OK;
    if (!x || !z || !cc) return ITPP_ERR_ARG;
    DeviceState d = view(h, b);
    const int o = c->cur ^ 1;
    uint64_t* dx = static_cast<uint64_t*>(d.keys[o]);
    uint64_t* dz = dx + n * d.W;
    double* dc = d.coef[o];
    const size_t kb = (size_t)n * d.W * 8;
    if (launch_export(d, dx, dz, dc, h->stream) != cudaSuccess ||
        cudaMemcpyAsync(x, dx, kb, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess ||
        cudaMemcpyAsync(z, dz, kb, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess ||
        cudaMemcpyAsync(cc, dc, (size_t)n * 8, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess ||
        cudaStreamSynchronize(h->stream) != cudaSuccess)
        return h->sticky = ITPP_ERR_CUDA;
    return ITPP_OK;
}

itpp_status itpp_batch_expect(itpp_batch_handle h, int b, const uint64_t* obs_x,
                              const uint64_t* obs_z, const double* obs_w, int m, double* out) {
    if (!h || b < 0 || b >= h->s.B || !obs_x || !obs_z || !obs_w || !out || m < 1 || m > 65536)
        return ITPP_ERR_ARG;
    if (h->sticky) return h->sticky;
    const int W = h->s.W;
    for (int j = 0; j < m; ++j)
        if (!bits_ok(h->n[(size_t)b], W, obs_x + (size_t)j * W) ||
            !bits_ok(h->n[(size_t)b], W, obs_z + (size_t)j * W))
            return ITPP_ERR_ARG;
    const size_t tsize = next_pow2((uint64_t)2 * m);
    const size_t need = (size_t)m * W * 16 + (size_t)m * 8 * 2 + (size_t)(m + 1) * 8 + tsize * 4 +
                        (size_t)m * 4 + 256;
    if (need > h->obs_bytes) {
        if (h->obs_mem) cudaFree(h->obs_mem);
        h->obs_mem = nullptr;
        h->obs_bytes = 0;
        if (cudaMalloc(&h->obs_mem, need) != cudaSuccess) return ITPP_ERR_ALLOC;
        h->obs_bytes = need;
    }
    char* p = static_cast<char*>(h->obs_mem);
    uint64_t* ox = reinterpret_cast<uint64_t*>(p); p += (size_t)m * W * 8;
    uint64_t* oz = reinterpret_cast<uint64_t*>(p); p += (size_t)m * W * 8;
    double* ow = reinterpret_cast<double*>(p); p += (size_t)m * 8;
    double* vals = reinterpret_cast<double*>(p); p += (size_t)m * 8;
    double* res = reinterpret_cast<double*>(p); p += (size_t)(m + 1) * 8;
    int* tab = reinterpret_cast<int*>(p); p += tsize * 4;
    int* first = reinterpret_cast<int*>(p);
    std::vector<double> buf((size_t)m + 1);
    DeviceState d = view(h, b);
    if (cudaMemcpyAsync(ox, obs_x, (size_t)m * W * 8, cudaMemcpyHostToDevice, h->stream) != cudaSuccess ||
        cudaMemcpyAsync(oz, obs_z, (size_t)m * W * 8, cudaMemcpyHostToDevice, h->stream) != cudaSuccess ||
        cudaMemcpyAsync(ow, obs_w, (size_t)m * 8, cudaMemcpyHostToDevice, h->stream) != cudaSuccess ||
        launch_expect(d, ox, oz, ow, m, (int)tsize, tab, first, vals, res, h->stream) != cudaSuccess ||
        cudaMemcpyAsync(buf.data(), res, ((size_t)m + 1) * 8, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess ||
        cudaStreamSynchronize(h->stream) != cudaSuccess)
        return h->sticky = ITPP_ERR_CUDA;
    DevCtl* c = reinterpret_cast<DevCtl*>(h->h_ctl.data());
    itpp_status st = read_head(h, b, c);
    if (st) return st;
    if (c->status) return (itpp_status)c->status;
    *out = buf[(size_t)m];
    return ITPP_OK;
}

}  // extern "C"
