// Instantiations of the decode kernel's fp16 form with the passes over K shared in a cluster (see gemv.cuh).
#include "gemv.cuh"

namespace btc {
namespace gv {
int launch_half_split(const Batch &b, const Pick &k, int grid, int cluster, int *fit, cudaStream_t s) { return dispatch<true, true>(b, k, grid, cluster, fit, s); }
}  // namespace gv
}  // namespace btc
