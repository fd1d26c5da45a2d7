// Instantiations of the decode kernel's integer form (see gemv.cuh).
#include "gemv.cuh"

namespace btc {
namespace gv {
int launch_int(const Batch &b, const Pick &k, int grid, int cluster, int *fit, cudaStream_t s) { return dispatch<false, false>(b, k, grid, cluster, fit, s); }
}  // namespace gv
}  // namespace btc
