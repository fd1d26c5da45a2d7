// Instantiations of the decode kernel's integer form (see gemv.cuh).
#include "gemv.cuh"

namespace btc {
namespace gv {
int launch_int(const Batch &b, int ncls, int tab, int ib, int nw, bool x32, int grid, cudaStream_t s) { return dispatch<false>(b, ncls, tab, ib, nw, x32, grid, s); }
}  // namespace gv
}  // namespace btc
