// Instantiations of the decode kernel's fp16 form (see gemv.cuh).
#include "gemv.cuh"

namespace btc {
namespace gv {
int launch_half(const Batch &b, int ncls, int tab, int ib, int nw, bool x32, int grid, cudaStream_t s) { return dispatch<true>(b, ncls, tab, ib, nw, x32, grid, s); }
}  // namespace gv
}  // namespace btc
