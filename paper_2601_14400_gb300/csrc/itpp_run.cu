// itpp_run.cu -- the run kernel with few CTAs per SM, and the choice.
#include "itpp_run_impl.cuh"

namespace itpp {

size_t run_shared_bytes() { return (sizeof(RunShared) + 255) / 256 * 256; }
size_t run_shared_head() { return offsetof(RunShared, pub); }

int run_fit(int W, bool wide) {
    if (wide) return W == 1 ? run_fit_as<1, true>() : run_fit_as<2, true>();
    return W == 1 ? run_fit_as<1, false>() : run_fit_as<2, false>();
}

template <int W>
cudaError_t launch_run(const RunArgs<W>& a, const RunChunk<W>& chunk, int grid, bool wide,
                       cudaStream_t st) {
    return wide ? launch_run_as<W, true>(a, chunk, grid, st)
                : launch_run_as<W, false>(a, chunk, grid, st);
}

template int run_fit_as<1, false>();
template int run_fit_as<2, false>();
template cudaError_t launch_run<1>(const RunArgs<1>&, const RunChunk<1>&, int, bool, cudaStream_t);
template cudaError_t launch_run<2>(const RunArgs<2>&, const RunChunk<2>&, int, bool, cudaStream_t);

}  // namespace itpp
