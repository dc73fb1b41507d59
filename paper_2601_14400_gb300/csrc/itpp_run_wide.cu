// itpp_run_wide.cu -- the run kernel with one more CTA per SM (a translation
// unit of its own: each takes the compiler half a minute).
#include "itpp_run_impl.cuh"

namespace itpp {

template int run_fit_as<1, true>();
template int run_fit_as<2, true>();
template cudaError_t launch_run_as<1, true>(const RunArgs<1>&, const RunChunk<1>&, int, cudaStream_t);
template cudaError_t launch_run_as<2, true>(const RunArgs<2>&, const RunChunk<2>&, int, cudaStream_t);

}  // namespace itpp
