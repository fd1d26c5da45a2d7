// Internal declarations shared by the translation units of the library (not installed).
#pragma once
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include "btc.h"

namespace btc {

struct LinearArgs {
    const void *x;
    const uint16_t *idx;
    const uint32_t *Cp;
    const __half *alpha;
    const __half *mu;      // may be nullptr
    void *y;
    void *workspace;
    size_t workspace_bytes;
    int x_dt, y_dt;
    int M, N, K, v, Kc, Kb;   // Kb = K / v
    // dense-packed indices (idx_bits > 0): idx is unused, idx_packed holds rows of idx_pitch bytes, idx_bits bits per index
    const void *idx_packed = nullptr;
    size_t idx_pitch = 0;
    int idx_bits = 0;
    // a term of a sum of layers: x / idx may be column ranges of wider matrices (row strides in elements, 0 = dense),
    // and the result may be added to y (fp32) instead of overwriting it
    int x_stride = 0;
    int idx_stride = 0;
    int accumulate = 0;
};

// Records a CUDA error for btc_last_cuda_error() and maps it to BTC_ERR_CUDA.
int cuda_fail(cudaError_t e);
// SMs of the current device, which size the launches.
int device_sms();
inline int cuda_check_launch() {
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? BTC_OK : cuda_fail(e);
}

// gemv_generic.cu: any v / Kc / M (M is tiled by 8 over grid.y), plain CUDA cores.
int launch_linear_generic(const LinearArgs &a, cudaStream_t s);

// gemv_decode.cu: decode path for rows of indices that are not a whole number of 16-byte pieces (M <= 8, v a multiple of 4).
// Returns BTC_ERR_UNSUPPORTED when the shape is outside what it covers, in which case the caller falls back to the generic kernel.
int launch_gemv_decode(const LinearArgs &a, cudaStream_t s);

// gemm_tcgen05.cu: tensor-core path; `transformed`: x comes from the activation transform, run in front of it.  Same UNSUPPORTED convention.
int launch_gemm_tcgen05(const LinearArgs &a, bool transformed, cudaStream_t s);
size_t gemm_tcgen05_workspace_bytes(int M);   // row sums of x (a split of K sums in distributed shared memory)

// gemv.cu: the decode path; runs up to IM_MAXP independent layers (M <= 8 each), one launch for those that share a kernel.
// Returns BTC_ERR_UNSUPPORTED when some layer is outside what it covers (nothing is launched then).
constexpr int IM_MAXP = 8;
int launch_gemv(const LinearArgs *problems, int count, cudaStream_t s);
int gemv_status_read(int *out);
int gemv_status_reset();
int gemv_selftest_wait(cudaStream_t s);

// pack.cu: debug check of the index range (BTC_DEBUG_CHECK_INDICES=1) and its status word.
bool debug_check_indices_enabled();
int launch_index_check(const uint16_t *idx, size_t count, int Kc, cudaStream_t s);
int index_status_read(int *out);
int index_status_reset();

// codebook_kmeans.cu: status word of its grid barrier.
int km_status_read(int *out);
int km_status_reset();

// gemv_lut.cu: the paper's two-stage lookup scheme (alternative route, own entry point).
int launch_gemv_lut(const LinearArgs &a, cudaStream_t s);
size_t gemv_lut_workspace_bytes(int M, int N, int K, int v);

// transform.cu: x' = x * D * (P1 (x) P2) into xt (same shape as x, dtype out_dt).
int launch_transform(const void *x, int x_dt, const btc_transform &T, void *xt, int out_dt, int M, int K,
                     cudaStream_t s);

// ---- small device helpers ------------------------------------------------------------------
__device__ __forceinline__ float load_as_float(const void *p, int dt, size_t i) {
    if (dt == BTC_F16) return __half2float(reinterpret_cast<const __half *>(p)[i]);
    if (dt == BTC_BF16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(p)[i]);
    return reinterpret_cast<const float *>(p)[i];
}
__device__ __forceinline__ void store_from_float(void *p, int dt, size_t i, float f) {
    if (dt == BTC_F32) reinterpret_cast<float *>(p)[i] = f;
    else if (dt == BTC_F16) reinterpret_cast<__half *>(p)[i] = __float2half_rn(f);
    else reinterpret_cast<__nv_bfloat16 *>(p)[i] = __float2bfloat16_rn(f);
}
// Activations in a kernel that starts before the one in front of it has ended: that one may be writing them while this one runs, so
// they are not read-only for its lifetime as ld.global.nc (__ldg, const __restrict__) demands, and a line of them that an
// SM's L1 still holds from a pass before would not have to be given up.  Plain loads, which griddepcontrol.wait orders; volatile, so that none
// moves in front of it.
__device__ __forceinline__ uint4 ld_x128(const void *p) {
    uint4 q;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w) : "l"(p));
    return q;
}
__device__ __forceinline__ uint2 ld_x64(const void *p) {
    uint2 q;
    asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(q.x), "=r"(q.y) : "l"(p));
    return q;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

}  // namespace btc
