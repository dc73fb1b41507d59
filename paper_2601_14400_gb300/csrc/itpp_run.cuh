// itpp_run.cuh -- arguments of the run kernel (itpp_run_impl.cuh): a layer's
// gates in one launch.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "itpp_common.cuh"

namespace itpp {

// One gate as the run reads it, with the windows a scatter at this gate can
// prepare: the gates from here on that act on at most so many sites (level 0:
// the longest windows, level 1: three sites), len 0 when this gate alone acts
// on more.
template <int W>
struct RunGate {
    uint64_t qx[W], qz[W];
    uint64_t win[2][W];
    double ch, msh;
    uint8_t len[2], sites[2];
    uint8_t pad[4];
};

// Sites of the two window levels.
constexpr int run_sites(int W, int level) { return level ? 3 : (W == 1 ? 5 : 4); }

// The windows that start at each of n gates of a schedule (which repeats).
template <int W>
void plan_run_windows(RunGate<W>* g, int n) {
    for (int lv = 0; lv < 2; ++lv)
        for (int k = 0; k < n; ++k) {
            uint64_t s[W] = {};
            int len = 0, sites = 0;
            for (int j = 0; j < n && len < 255; ++j) {
                const RunGate<W>& q = g[(k + j) % n];
                uint64_t t[W];
                int c = 0;
                for (int w = 0; w < W; ++w) {
                    t[w] = s[w] | q.qx[w] | q.qz[w];
                    c += __builtin_popcountll(t[w]);
                }
                if (c > run_sites(W, lv)) break;
                for (int w = 0; w < W; ++w) s[w] = t[w];
                sites = c;
                ++len;
            }
            g[k].len[lv] = (uint8_t)len;
            g[k].sites[lv] = (uint8_t)sites;
            for (int w = 0; w < W; ++w) g[k].win[lv][w] = s[w];
        }
}

// The gates of a launch as a kernel argument: the host keeps no device copy
// of them that a change of the coefficients or a captured launch could race.
constexpr int kRunChunk = 256;
// Smallest mean partition a scatter aims for to give every CTA one, unless the
// caller asks for smaller ones.
constexpr int kRunMinPart = 128;
constexpr int run_min_part(int target) { return target < kRunMinPart ? target : kRunMinPart; }
// Distance of two partition cursors (words).
constexpr int kRunPad = 32;
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
    unsigned int* cnt;            // [B][3][part_max], kRunPad apart
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

// Entries of the candidate list, and where the ties lie behind it, in `bytes` of
// scratch (values, then indices; the ties on a 256-byte boundary).  A select
// without a range lists every child of one digit of |c|, and a digit may hold
// all of them: 2 cap_M.  The table's memory has room for that at every bound
// (64 cap_M bytes at one mask word, 128 at two, 256 slots at least): it is not
// to be cut further.
template <int W>
constexpr uint64_t run_list_cap(uint64_t bytes, uint64_t home_cap) {
    const uint64_t n = (bytes - 255) / (12 + sizeof(PKey<W>));
    return n < home_cap ? n : home_cap;
}
constexpr uint64_t run_tie_off(uint64_t cand_cap) { return (cand_cap * 12 + 255) / 256 * 256; }

// Bytes of one team's shared block, and of its head that a launch clears.
size_t run_shared_bytes();
size_t run_shared_head();
// The kernel with few CTAs per SM (3; 2 with two mask words), or the wide one
// with one more.  The register file is shared out: the first spills less (844
// bytes of stores against 1,184, with two words 132 against 1,004), the second
// hides more latency.  For
// one propagation of 2^16 or 2^18 terms a layer takes 3.21 and 3.14 ms with the
// first, 3.55 and 3.45 with the second; at 2^20 both 9.3.  Batches of 4 x 2^16
// and 16 x 2^14: 64.1 and 39.8 ms with the first, 68.1 and 41.6 with the second;
// 8 x 2^16 and 64 x 2^14: 77.2 and 69.4 against 72.1 and 60.7.
template <int W, bool kWide> int run_fit_as();
template <int W, bool kWide>
cudaError_t launch_run_as(const RunArgs<W>& a, const RunChunk<W>& chunk, int grid, cudaStream_t st);
extern template int run_fit_as<1, true>();
extern template int run_fit_as<2, true>();
extern template cudaError_t launch_run_as<1, true>(const RunArgs<1>&, const RunChunk<1>&, int, cudaStream_t);
extern template cudaError_t launch_run_as<2, true>(const RunArgs<2>&, const RunChunk<2>&, int, cudaStream_t);
// A batch of more terms than this runs on the wide one.
constexpr uint64_t kRunWide = 1ULL << 18;

// CTAs per SM that fit.
int run_fit(int W, bool wide);
// A cooperative launch (the CTAs of a team wait for one another).
template <int W>
cudaError_t launch_run(const RunArgs<W>& a, const RunChunk<W>& chunk, int grid, bool wide,
                       cudaStream_t st);

}  // namespace itpp
