// Instantiations of the decode kernel's fp16 form (see gemv.cuh).
#include "gemv.cuh"

namespace btc {
namespace gv {
int launch_half(const Batch &b, const Pick &k, int grid, int cluster, int *fit, cudaStream_t s) { return dispatch<true, false>(b, k, grid, cluster, fit, s); }
}  // namespace gv
}  // namespace btc
