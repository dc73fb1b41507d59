// itpp_ctx.h -- the handle behind itpp_handle (internal; shared by the C ABI
// translation units).
#pragma once

#include <cstddef>
#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

#include "itpp.h"
#include "itpp_common.cuh"
#include "itpp_launch.h"

namespace itpp_detail {

constexpr int kKinds = 4;
constexpr size_t kCtlHead = offsetof(itpp::DevCtl, sel_hist);

struct EventPair {
    cudaEvent_t a, b;
};

}  // namespace itpp_detail

using itpp_detail::EventPair;
using itpp_detail::kKinds;
using itpp_detail::kCtlHead;

struct itpp_ctx {
    itpp::DeviceState s;
    std::vector<itpp::HostGate> gates;   // the elementary gates of one layer
    // gate j of the layer is Hamiltonian term src_gate[j] with coefficient
    // alpha * src_scale[j] (the first-order product: j, 1; Strang: halves)
    std::vector<int> src_gate;
    std::vector<double> src_scale;
    int user_gates = 0;
    double dtau = 0;
    itpp_params p{};
    cudaStream_t stream = nullptr;
    int device = 0;
    itpp_status sticky = ITPP_OK;
    itpp::DevCtl* h_ctl = nullptr;   // pinned mirror of the control block head
    // expectation scratch
    void* obs_mem = nullptr;
    size_t obs_bytes = 0;
    // PSD-restored observable: block partials and the result
    double* psd_mem = nullptr;
    // sorted merge scratch
    void* sort_mem = nullptr;
    uint64_t sort_bytes = 0;
    uint64_t launches = 0;   // kernels launched by this handle
    // gates run in one launch (itpp_run_impl.cuh): bounds up to kRunMax terms; the
    // team's shared block and the partition cursors
    bool run_ok = false;
    int run_grid = 0;
    uint32_t run_part_max = 0;
    void* run_shared = nullptr;
    unsigned int* run_cnt = nullptr;
    // profiling
    bool prof = false;
    std::vector<EventPair> ev[kKinds];
    size_t ev_used[kKinds] = {0, 0, 0, 0};
    double prof_ms[kKinds] = {0, 0, 0, 0};
    uint64_t prof_n[kKinds] = {0, 0, 0, 0};
};


// Helpers of the C ABI used by more than one translation unit.
itpp_status itpp_detail_sync_ctl(itpp_ctx* h);
// n_layers whole layers; log (device, or null) receives the term count after
// every gate.
itpp_status itpp_detail_layers(itpp_ctx* h, int n_layers, unsigned long long* log);
cudaError_t itpp_detail_materialize(itpp_ctx* h);
