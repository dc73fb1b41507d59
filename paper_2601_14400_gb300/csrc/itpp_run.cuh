// itpp_run.cuh -- arguments of the run kernel (itpp_run.cu): a layer's gates
// in one launch.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "itpp_common.cuh"

namespace itpp {

// One gate as the run reads it.
template <int W>
struct RunGate {
    uint64_t qx[W], qz[W];
    uint64_t win[W];     // sites of its window
    double ch, msh;
    int pair, sites;     // pair-key mode; sites of the window
    int start, pad;      // first gate of its window
};

// The gates of a launch as a kernel argument: the host keeps no device copy
// of them that a change of the coefficients or a captured launch could race.
constexpr int kRunChunk = 256;
// Smallest mean partition a scatter aims for to give every CTA one.
constexpr int kRunMinPart = 128;
template <int W>
struct RunChunk {
    RunGate<W> g[kRunChunk];
};

template <int W>
struct RunArgs {
    PKey<W>* k[2];
    double* c[2];
    PKey<W>* kp;
    double* cp;
    unsigned int* cnt;            // [B][2][part_max]
    DevCtl* ctl;                  // [B]
    void* scratch;                // [B] candidates and ties (the merge table's memory)
    void* shared;                 // [teams] RunShared
    long long* drift;             // [B][drift_stride]
    unsigned long long* log;      // terms after every gate, or null
    const int* n;                 // [B] sites, or null: one_n
    const RunGate<W>* gates;      // [B][max_gates], or null: the chunk argument
    const int* n_gates;           // [B]
    const uint4* team_of;         // [grid] (team, rank, size, teams), or null: one team
    uint64_t buf_stride, part_stride, scratch_stride, shared_stride;
    uint64_t buf_cap, home_cap;   // terms a run / a home holds
    uint64_t cand_cap, tie_off, cap_M, cand_hi;
    unsigned long long delta_bits;
    uint32_t part_max;
    int drift_stride, drift_gates;
    int B, max_gates, one_gates, one_n, gate0, n_layers;
    int target, min_part, cap_policy, maxw;
};

// Bytes of one team's shared block, and of its head that a launch clears.
size_t run_shared_bytes();
size_t run_shared_head();
// CTAs per SM that fit.
int run_fit(int W);
// A cooperative launch (the CTAs of a team wait for one another).
template <int W>
cudaError_t launch_run(const RunArgs<W>& a, const RunChunk<W>& chunk, int grid, cudaStream_t st);

}  // namespace itpp
