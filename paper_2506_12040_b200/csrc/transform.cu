// Online activation transform  x' = x * D * (P1 (x) P2),  D = diag(sigma), sigma in {+1,-1}
// (paper Section 4.2 "Transformation Pair": learnable sign flips and a Kronecker-factored matrix, applied
// at inference as X <- X T).  With a row of x viewed row-major as a k1 x k2 matrix X (k1 * k2 = K):
//     X' = P1^T (X o sigma) P2,     X'[c][d] = sum_a sum_b P1[a][c] * sigma[a k2 + b] * X[a][b] * P2[b][d]
// computed as two small products with fp32 accumulation: Y = (X o sigma) P2, then X' = P1^T Y.
// The result is written as fp32 for the decode path (which quantises or rounds the activations itself, so no intermediate
// 16-bit rounding is added) and in the dtype of x for the tensor-core path.
// transform_kernel (fp32 activations, factor sizes that the other two do not take): a CTA owns a tile of TR_DT output
// columns d and a group of rows of x: it stages the k2 x TR_DT slab of P2 and all of P1 in shared memory once, then for each of
// its rows loads X (K values) and produces X'[:, d-tile]; a decode step with one row of x therefore spreads over k2 / TR_DT
// SMs instead of one.
#include <atomic>
#include <type_traits>
#include "btc_internal.cuh"

namespace btc {

constexpr int TR_THREADS = 256;
constexpr int TR_DT = 8;            // output columns d per CTA

__global__ void __launch_bounds__(TR_THREADS)
transform_kernel(const void *x, int x_dt, const uint32_t *__restrict__ sigma_bits,
                 const float *__restrict__ P1, const float *__restrict__ P2, int k1, int k2, void *__restrict__ xt, int out_dt,
                 int M, int rows_per_cta)
{
    extern __shared__ float tr_smem[];
    // (the layer kernel that follows may start right away and prefetch its indices; it reads x' only after this grid
    // has completed)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int K = k1 * k2;
    const int d0 = blockIdx.x * TR_DT, nd = min(TR_DT, k2 - d0);
    const int xp = k2 + 4;                 // X row pitch: four words of padding put the 8 rows x 4 lanes of a warp on 32 banks
    const int kp = k1 + 8;                 // P1 row pitch, for the same reason
    float *X = tr_smem;                    // [k1][xp]   (sign-flipped activations of the current row)
    float *Pd = X + ((k1 * xp + 3) & ~3);                     // [k2][TR_DT] slab of P2
    float *Y = Pd + k2 * TR_DT;            // [k1][TR_DT]
    float *Q1 = Y + k1 * TR_DT;            // [k1][kp]   P1, staged once per CTA
    for (int i = threadIdx.x; i < k2 * TR_DT; i += TR_THREADS) {
        const int b = i / TR_DT, d = i - b * TR_DT;
        Pd[i] = d < nd ? __ldg(P2 + (size_t)b * k2 + d0 + d) : 0.f;
    }
    for (int i = threadIdx.x; i < k1 * k1; i += TR_THREADS) Q1[(i / k1) * kp + (i % k1)] = __ldg(P1 + i);
    // the factors are parameters of the layer, complete before the call was enqueued: they were staged while the kernel
    // before this one may still be running; x is read only once that kernel has completed
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int m0 = blockIdx.y * rows_per_cta, m1 = min(M, m0 + rows_per_cta);
    for (int m = m0; m < m1; ++m) {
        const size_t row = (size_t)m * K;
        __syncthreads();                   // (previous row's X and Y are no longer read; P slabs are in place)
        if (x_dt != BTC_F32 && (k2 & 7) == 0) {
            // 16-bit activations, eight per 16-byte load (rows are 16-byte aligned when 8 divides K)
            const uint4 *src = reinterpret_cast<const uint4 *>(reinterpret_cast<const uint16_t *>(x) + row);
            for (int i = threadIdx.x; i < K / 8; i += TR_THREADS) {
                const uint4 q = ld_x128(src + i);
                const uint32_t sg = __ldg(sigma_bits + (i >> 2)) >> ((i & 3) * 8);
                const uint32_t w[4] = {q.x, q.y, q.z, q.w};
                const int rr = 4 * ((8 * i) / k2);     // the eight elements share a row of X (8 divides k2 here)
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    float lo, hi;
                    if (x_dt == BTC_F16) {
                        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&w[h]));
                        lo = f.x; hi = f.y;
                    } else {
                        lo = __uint_as_float(w[h] << 16); hi = __uint_as_float(w[h] & 0xffff0000u);
                    }
                    const int e0 = 8 * i + 2 * h;                                    // element e of row r sits at e + 4 r
                    X[e0 + rr] = ((sg >> (2 * h)) & 1u) ? -lo : lo;
                    X[e0 + 1 + rr] = ((sg >> (2 * h + 1)) & 1u) ? -hi : hi;
                }
            }
        } else {
            for (int i = threadIdx.x; i < K; i += TR_THREADS) {
                float v = load_as_float(x, x_dt, row + i);
                if ((__ldg(sigma_bits + (i >> 5)) >> (i & 31)) & 1u) v = -v;
                X[i + 4 * (i / k2)] = v;
            }
        }
        __syncthreads();
        // Y[a][d] = sum_b X[a][b] * P2[b][d0 + d]: four lanes share a row a, each sums a quarter of b for all TR_DT columns
        // (one X value and one slab row per 8 FMAs), then the quad adds up
        for (int w0 = 0; w0 < k1 * 4; w0 += TR_THREADS) {
            const int w = w0 + threadIdx.x, a = w >> 2, q = w & 3;
            float acc[TR_DT];
#pragma unroll
            for (int d = 0; d < TR_DT; ++d) acc[d] = 0.f;
            if (a < k1) {
                const float *xa = X + (size_t)a * xp;
                for (int b = q; b < k2; b += 4) {                      // (interleaved quarters: the quad reads four neighbouring slab rows)
                    const float xv = xa[b];
                    const float4 p0 = *reinterpret_cast<const float4 *>(Pd + b * TR_DT), p1 = *reinterpret_cast<const float4 *>(Pd + b * TR_DT + 4);
                    acc[0] = fmaf(xv, p0.x, acc[0]); acc[1] = fmaf(xv, p0.y, acc[1]); acc[2] = fmaf(xv, p0.z, acc[2]); acc[3] = fmaf(xv, p0.w, acc[3]);
                    acc[4] = fmaf(xv, p1.x, acc[4]); acc[5] = fmaf(xv, p1.y, acc[5]); acc[6] = fmaf(xv, p1.z, acc[6]); acc[7] = fmaf(xv, p1.w, acc[7]);
                }
            }
#pragma unroll
            for (int d = 0; d < TR_DT; ++d) {
                acc[d] += __shfl_xor_sync(0xffffffffu, acc[d], 1);
                acc[d] += __shfl_xor_sync(0xffffffffu, acc[d], 2);
            }
            if (a < k1 && q == 0) {
                *reinterpret_cast<float4 *>(Y + a * TR_DT) = make_float4(acc[0], acc[1], acc[2], acc[3]);
                *reinterpret_cast<float4 *>(Y + a * TR_DT + 4) = make_float4(acc[4], acc[5], acc[6], acc[7]);
            }
        }
        __syncthreads();
        // X'[c][d0 + d] = sum_a P1[a][c] * Y[a][d]: the same split, quarters of a
        for (int w0 = 0; w0 < k1 * 4; w0 += TR_THREADS) {
            const int w = w0 + threadIdx.x, c = w >> 2, q = w & 3;
            float acc[TR_DT];
#pragma unroll
            for (int d = 0; d < TR_DT; ++d) acc[d] = 0.f;
            if (c < k1) {
                for (int a = q; a < k1; a += 4) {
                    const float pv = Q1[a * kp + c];
                    const float4 y0 = *reinterpret_cast<const float4 *>(Y + a * TR_DT), y1 = *reinterpret_cast<const float4 *>(Y + a * TR_DT + 4);
                    acc[0] = fmaf(pv, y0.x, acc[0]); acc[1] = fmaf(pv, y0.y, acc[1]); acc[2] = fmaf(pv, y0.z, acc[2]); acc[3] = fmaf(pv, y0.w, acc[3]);
                    acc[4] = fmaf(pv, y1.x, acc[4]); acc[5] = fmaf(pv, y1.y, acc[5]); acc[6] = fmaf(pv, y1.z, acc[6]); acc[7] = fmaf(pv, y1.w, acc[7]);
                }
            }
#pragma unroll
            for (int d = 0; d < TR_DT; ++d) {
                acc[d] += __shfl_xor_sync(0xffffffffu, acc[d], 1);
                acc[d] += __shfl_xor_sync(0xffffffffu, acc[d], 2);
            }
            if (c < k1 && q == 0) {
#pragma unroll
                for (int d = 0; d < TR_DT; ++d)
                    if (d < nd) store_from_float(xt, out_dt, row + (size_t)c * k2 + d0 + d, acc[d]);
            }
        }
    }
}

// ---- up to eight rows of 16-bit activations, k2 = 64 or 128, k1 up to 128 ------------------------------------------------
// A CTA owns eight output columns d of one row of x.  Four lanes share a row a of X and read it from global memory straight into
// registers, each every fourth piece of eight; Y (k1 x 8) goes through shared memory; four lanes share an output row c, each with
// every fourth a.  Lanes that share a sum hand over halves of their columns, so that four sums over four lanes take three shuffles
// and leave one in each.
// Bound: latency, of the chain behind the kernel before it: wait, x from L2, two products of K2 / 4 and k1 / 4 steps with one
// barrier between them, store; P1 waits in L1.  A CTA asks for more than half of an SM's shared memory, so that no two share one: small
// CTAs, up to eight on an SM, all went to the few SMs that a layer in front of them left first, worked there side by side, and kept
// those SMs from the layer behind, which has CTAs for all of them.  That layer is let in when the wait is over: it has the transform's time
// to fetch its first indices, needs no more, and takes no SM from transforms that wait.
// us a call, transform and one or three 4096 x K layers behind it (v = 16), of transform_kernel, of small CTAs that let the layer in at
// once, and of this one:
//             one row: one layer    three layers          eight rows: one layer    three layers
//   32 x 64    7.1 /  6.9 /  5.9     8.8 /  8.7 /  7.4     10.0 / 10.2 /  9.5     14.0 / 20.2 / 11.6
//   64 x 64    8.3 /  7.9 /  7.6    11.1 /  9.4 /  9.1     20.5 / 17.2 / 13.1     22.8 / 25.4 / 15.2
//   40 x 128  10.3 /  9.5 /  9.4    15.6 / 14.9 / 12.6     25.0 / 24.0 / 18.6     28.6 / 28.1 / 22.9
//   86 x 128  16.9 / 15.9 / 15.1    21.6 / 26.0 / 20.3     29.2 / 33.0 / 29.2     39.9 / 50.6 / 35.4
// (The small ones were the faster only beside the integer decode kernel at 64 x 64 and less, three layers of 11008: 13.0 and now 13.5.)
constexpr int TS_D = 8;             // columns per CTA
constexpr int TS_ALONE = 115 * 1024; // bytes of dynamic shared memory, unused: half of an SM's and more

// acc[i] summed over the four lanes that differ in bits 0 and 1; lane q gets column q
__device__ __forceinline__ float ts_quad(const float *acc, int q) {
    const float k0 = q & 2 ? acc[2] : acc[0], k1 = q & 2 ? acc[3] : acc[1];
    const float s0 = k0 + __shfl_xor_sync(0xffffffffu, q & 2 ? acc[0] : acc[2], 2);
    const float s1 = k1 + __shfl_xor_sync(0xffffffffu, q & 2 ? acc[1] : acc[3], 2);
    return (q & 1 ? s1 : s0) + __shfl_xor_sync(0xffffffffu, q & 1 ? s0 : s1, 1);
}
__device__ __forceinline__ void ts_fma(float (&acc)[TS_D], float f, const float *row) {
    const float4 p = *reinterpret_cast<const float4 *>(row), r = *reinterpret_cast<const float4 *>(row + 4);
    acc[0] = fmaf(f, p.x, acc[0]); acc[1] = fmaf(f, p.y, acc[1]); acc[2] = fmaf(f, p.z, acc[2]); acc[3] = fmaf(f, p.w, acc[3]);
    acc[4] = fmaf(f, r.x, acc[4]); acc[5] = fmaf(f, r.y, acc[5]); acc[6] = fmaf(f, r.z, acc[6]); acc[7] = fmaf(f, r.w, acc[7]);
}

// AP: passes of 64 rows a, and c; K2: k2.  (The second bound is there for the registers that it has the compiler spend, which keep more loads
// in flight: 64 where it takes 44 to 51 by itself; 128 x 64, one row, alone 6.7 us, and 7.5)
template <int AP, int K2>
__global__ void __launch_bounds__(TR_THREADS, AP == 1 && K2 == 64 ? 8 : 4)
transform_few_kernel(const uint16_t *x, int f16, const uint32_t *__restrict__ sigma_bits, const float *__restrict__ P1,
                     const float *__restrict__ P2, int k1, void *__restrict__ xt, int out_dt)
{
    constexpr int PIECES = K2 / 32;                      // of eight activations, of a lane
    __shared__ __align__(16) float s_p2[K2 / 8][8 * TS_D + 4];           // (four lanes read pieces next to each other: on different banks)
    __shared__ __align__(16) float s_y[64 * AP][TS_D];
    const int tid = threadIdx.x, q = tid & 3, d0 = blockIdx.x * TS_D;
    const size_t row = (size_t)blockIdx.y * k1 * K2;
    for (int i = tid; i < K2 * TS_D; i += TR_THREADS) {
        const int b = i / TS_D, d = i % TS_D;
        s_p2[b / 8][b % 8 * TS_D + d] = __ldg(P2 + (size_t)b * K2 + d0 + d);
    }
    for (int i = 8 * tid; i < k1 * k1; i += 8 * TR_THREADS) {            // (a word of every 32 bytes, into L1)
        float f;
        asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(f) : "l"(P1 + i));
    }
    uint32_t sg[PIECES];                                 // sign bits of a piece
    auto load_signs = [&](int a) {
#pragma unroll
        for (int j = 0; j < PIECES; ++j) {
            const int e = min(a, k1 - 1) * K2 + 8 * (q + 4 * j);
            sg[j] = __ldg(sigma_bits + (e >> 5)) >> (e & 31);
        }
    };
    load_signs(tid >> 2);
    __syncthreads();
    // (the factors are parameters of the layer, complete before the call was enqueued; x is read, and x' written, once the kernel
    // before this one has completed)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#pragma unroll 1
    for (int ap = 0; ap < AP; ++ap) {
        const int a = 64 * ap + (tid >> 2);
        uint4 w[PIECES];
#pragma unroll
        for (int j = 0; j < PIECES; ++j)
            w[j] = a < k1 ? ld_x128(x + row + (size_t)a * K2 + 8 * (q + 4 * j)) : make_uint4(0u, 0u, 0u, 0u);
        float acc[TS_D] = {};
#pragma unroll
        for (int j = 0; j < PIECES; ++j) {
            const uint32_t h[4] = {w[j].x, w[j].y, w[j].z, w[j].w};
            const float *p = s_p2[q + 4 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t u = h[i] ^ (((sg[j] >> (2 * i)) & 1u) << 15) ^ (((sg[j] >> (2 * i + 1)) & 1u) << 31);
                const float2 f = f16 ? __half22float2(*reinterpret_cast<const __half2 *>(&u)) : make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
                ts_fma(acc, f.x, p + 2 * i * TS_D);
                ts_fma(acc, f.y, p + (2 * i + 1) * TS_D);
            }
        }
        const float y0 = ts_quad(acc, q), y1 = ts_quad(acc + 4, q);
        s_y[a][q] = a < k1 ? y0 : 0.f;                   // (not 0 times what P2 holds)
        s_y[a][4 + q] = a < k1 ? y1 : 0.f;
        if (AP > 1) load_signs(a + 64);
    }
    __syncthreads();
#pragma unroll 1
    for (int cp = 0; cp < AP; ++cp) {
        const int c = 64 * cp + (tid >> 2);
        float acc[TS_D] = {};
        int i0 = 0;
#pragma unroll 1
        do {
            float pv[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int a = q + 4 * (i0 + i);
                pv[i] = c < k1 && a < k1 ? __ldg(P1 + (size_t)a * k1 + c) : 0.f;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) ts_fma(acc, pv[i], s_y[q + 4 * (i0 + i)]);
            i0 += 8;
        } while (4 * i0 < k1);
        const float r0 = ts_quad(acc, q), r1 = ts_quad(acc + 4, q);
        if (c < k1) {
            store_from_float(xt, out_dt, row + (size_t)c * K2 + d0 + q, r0);
            store_from_float(xt, out_dt, row + (size_t)c * K2 + d0 + 4 + q, r1);
        }
    }
}

template <int AP, int K2>
static int launch_transform_few(const void *x, int x_dt, const btc_transform &T, void *xt, int out_dt, int M, cudaStream_t s)
{
    auto kern = transform_few_kernel<AP, K2>;
    static std::atomic<uint64_t> done{0};                          // (the attribute, once per device)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e);
    if (dev >= 64 || !((done.load(std::memory_order_relaxed) >> dev) & 1u)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, TS_ALONE);
        if (e != cudaSuccess) return cuda_fail(e);
        if (dev < 64) done.fetch_or(uint64_t(1) << dev, std::memory_order_relaxed);
    }
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(K2 / TS_D, (unsigned)M);
    cfg.blockDim = dim3(TR_THREADS);
    cfg.dynamicSmemBytes = TS_ALONE;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kern, static_cast<const uint16_t *>(x), x_dt == BTC_F16 ? 1 : 0, T.sigma_bits, T.P1, T.P2, T.k1, xt, out_dt);
    return e == cudaSuccess ? BTC_OK : cuda_fail(e);
}

// ---- 16-bit activations, k2 a multiple of 16, k1 up to 128: the two products on the warp-level tensor cores ---------------
// bf16 operands, fp32 accumulation; a factor, and Y between the products, is a sum of TERMS bf16 numbers (two hold 16 bits of
// a value, three all 24 of an fp32), and of the products of terms only those below the last term's own rounding are left out.
// An f16 activation is the sum of two bf16 numbers, a bf16 one is its own operand: loaded, sign bits flipped, multiplied.
// An item of work is one row of x, sixteen output columns d (a slice) and a share of the output rows c, and belongs to one
// warp: Y^T of the slice (16 x k1) stays in registers, where the accumulators of the first product, rounded to terms, are B
// fragments of the second.  Only the factors go through shared memory, split into terms and laid out as A fragments, once
// per CTA and before x is waited for; rows then cost no barrier.
// A lane's columns of x are four neighbours (both products may take their inner index in any order, as long as A and B agree),
// so x is read from global memory straight into fragments, 8 bytes a load; the warps of a CTA take the slices of the same
// rows, so all but the first read from L1.  Likewise a lane's results are four neighbouring columns.
// Bound: instruction issue and, for a few rows, the set-up (factors from L2, split) and one item's chain of MMAs; DRAM is
// under a tenth busy.  A form with both products through shared memory and two barriers a row (tf32; fp32 FMAs below 64 rows)
// took 12.6 us for 512 rows of 64 x 64 and 21.4 for 63, now 8.3 and 4.8; 86 x 128, 2048 rows: 134.6 -> 80.8, 63 rows: 41.1 ->
// 14.9.
constexpr int TM_WARPS = 8;

__device__ __forceinline__ uint32_t tm_pack(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ float tm_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float tm_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ void tm_mma(float (&c)[4], const uint4 &a, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
// the next term of a pair: taken off what is left of it
__device__ __forceinline__ uint32_t tm_term(float &lo, float &hi) {
    const uint32_t w = tm_pack(lo, hi);
    lo -= tm_lo(w); hi -= tm_hi(w);
    return w;
}

// One A fragment (16 rows x 16 of the inner index) of P^T as TERMS x 32 lanes x 16 bytes.  f[2 i], f[2 i + 1]: register i.
template <int TERMS>
__device__ __forceinline__ void tm_put(uint4 *dst, float (&f)[8]) {
#pragma unroll
    for (int u = 0; u < TERMS; ++u) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = tm_term(f[2 * i], f[2 * i + 1]);
        dst[u * 32] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

struct TmPlan { int ds, cg, rw, p2_frags, mask_off; };       // slices, shares of c and rows per CTA (ds * cg * rw warps); A fragments of P2

// NA: 8-wide tiles of a (even; k1 rounded up to 16, and beyond to a size instantiated; at least LO of them are full).  F16:
// activations f16, else bf16.  K2: k2 where it is one of the usual sizes (addresses become immediates), else 0.  DW: 16-wide
// parts of a slice; two use every activation and every fragment of P1 twice.
template <int NA, int TERMS, bool F16, int K2, int DW>
__global__ void __launch_bounds__(TM_WARPS * 32, 1)
transform_mma_kernel(const uint16_t *x, const uint32_t *__restrict__ sigma_bits, const float *__restrict__ P1,
                     const float *__restrict__ P2, int k1, int k2_arg, void *__restrict__ xt, int out_dt, int M, TmPlan plan)
{
    constexpr int LO = NA == 2 ? 0 : NA <= 8 ? NA - 2 : NA - 4, U = 8;
    extern __shared__ __align__(16) uint4 tm_smem[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int k2 = K2 ? K2 : k2_arg;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int K = k1 * k2, ks2 = k2 / 16, nc = (k1 + 15) / 16;
    uint4 *f2 = tm_smem, *f1 = tm_smem + (size_t)plan.p2_frags * TERMS * 32;
    uint2 *mask = reinterpret_cast<uint2 *>(reinterpret_cast<char *>(tm_smem) + plan.mask_off);
    // column of a 16-wide part of a slice that rows g and g + 8 of a fragment of P2, and columns 2t, 2t + 1 of the two result
    // tiles, stand for
    const int dg = 4 * (g >> 1) + (g & 1);
    // ---- the factors as fragments, eight loads of eight in flight per thread; the signs as masks of a lane's four activations
    {
        const int part0 = blockIdx.y * plan.ds * DW, nf = plan.p2_frags + nc * (NA / 2), nw = blockDim.x >> 5;
        for (int i0 = warp; i0 < NA * ks2; i0 += 2 * U * nw) {           // [k][tile of a][lane]
            uint32_t w[2 * U];
#pragma unroll
            for (int u = 0; u < 2 * U; ++u) {
                const int i = i0 + u * nw, k = i / NA, a = 8 * (i - k * NA) + g, e = a * k2 + 16 * k;
                w[u] = i < NA * ks2 && a < k1 ? __ldg(sigma_bits + (e >> 5)) >> ((e & 31) + 4 * t) : 0u;
            }
#pragma unroll
            for (int u = 0; u < 2 * U; ++u) {
                const uint32_t sb = w[u] & 15u;
                if (i0 + u * nw < NA * ks2) mask[(i0 + u * nw) * 32 + lane] = make_uint2((sb * 0x40008000u) & 0x80008000u, (sb * 0x10002000u) & 0x80008000u);
            }
        }
        for (int i0 = warp; i0 < nf; i0 += U * nw) {
            float f[U][8];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = i0 + u * nw;
                const bool second = i >= plan.p2_frags;
                const int j = second ? i - plan.p2_frags : i, per = second ? NA / 2 : ks2, q = j / per, k = j - q * per;
                // element (inner, outer) of the factor: rows b of P2 and its columns d, rows a of P1 and its columns c
                const int n = second ? k1 : k2, in0 = 16 * k + (second ? 2 * t : 4 * t), in1 = in0 + (second ? 8 : 2);
                const int out0 = 16 * (second ? q : part0 + q) + (second ? g : dg), out1 = out0 + (second ? 8 : 2);
                const float *src = (second ? P1 : P2) + (size_t)in0 * n + out0;
#pragma unroll
                for (int r = 0; r < 8; ++r) {            // (register r / 2, half r % 2)
                    const int in = (r & 4 ? in1 : in0) + (r & 1), out = r & 2 ? out1 : out0;
                    f[u][r] = i < nf && in < n && out < n ? __ldg(src + (size_t)(in - in0) * n + (out - out0)) : 0.f;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + u * nw < nf) tm_put<TERMS>(tm_smem + (size_t)(i0 + u * nw) * TERMS * 32 + lane, f[u]);
        }
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const int cs = warp % plan.cg, sl = (warp / plan.cg) % plan.ds, rw = warp / (plan.cg * plan.ds);
    const int d0 = 16 * DW * (blockIdx.y * plan.ds + sl);
    if (d0 >= k2) return;
    const int c_per = (nc + plan.cg - 1) / plan.cg, ct0 = cs * c_per, ct1 = min(nc, ct0 + c_per);
    if (ct0 >= ct1) return;
    const uint4 *A2 = f2 + (size_t)sl * DW * ks2 * TERMS * 32 + lane, *A1 = f1 + lane;
    mask += lane;
    // (an MMA cuts its sum off where an fp32 addition rounds: with three terms each step of the inner index is summed from zero, its
    // smallest products first, and added to the accumulator as an fp32)
    auto part = [](float (&step)[4], float (&sum)[4]) -> float (&)[4] { return TERMS > 2 ? step : sum; };
    constexpr int PF = NA <= 4 ? 4 : 2;                  // loads ahead, in steps of the first product
    for (int m = blockIdx.x * plan.rw + rw; m < M; m += gridDim.x * plan.rw) {
        const uint16_t *xr = x + (size_t)m * K + (size_t)g * k2 + 4 * t;
        uint2 q[PF][NA];
        auto load = [&](int k, uint2 (&dst)[NA]) {
#pragma unroll
            for (int at = 0; at < NA; ++at)
                dst[at] = at < LO || 8 * at + g < k1 ? ld_x64(xr + (size_t)(8 * at) * k2 + 16 * k) : make_uint2(0u, 0u);
        };
#pragma unroll
        for (int u = 0; u < PF; ++u)
            if (u < ks2) load(u, q[u]);
        // ---- Y^T[d][a] = sum_b P2[b][d] X[a][b]
        float y[DW][NA][4];
#pragma unroll
        for (int p = 0; p < DW; ++p)
#pragma unroll
            for (int at = 0; at < NA; ++at)
#pragma unroll
                for (int i = 0; i < 4; ++i) y[p][at][i] = 0.f;
        for (int k0 = 0; k0 < ks2; k0 += PF) {
#pragma unroll
            for (int u = 0; u < PF; ++u) {
                const int k = k0 + u;
                if (k < ks2) {
                    uint4 w[DW][TERMS];
#pragma unroll
                    for (int p = 0; p < DW; ++p)
#pragma unroll
                        for (int i = 0; i < TERMS; ++i) w[p][i] = A2[(size_t)((p * ks2 + k) * TERMS + i) * 32];
                    // a few tiles of a at a time, term by term: MMAs on one accumulator are never neighbours
                    constexpr int G = 4 / DW;
#pragma unroll
                    for (int a0 = 0; a0 < NA; a0 += G) {
                        uint32_t xb[G][2], xl[G][2];
                        float step[DW][G][4] = {};
#pragma unroll
                        for (int n = 0; n < G; ++n) {
                            const uint2 sg = mask[(k * NA + a0 + n) * 32];
                            xb[n][0] = q[u][a0 + n].x ^ sg.x;
                            xb[n][1] = q[u][a0 + n].y ^ sg.y;
                            if constexpr (F16) {
#pragma unroll
                                for (int i = 0; i < 2; ++i) {
                                    float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&xb[n][i]));
                                    xb[n][i] = tm_term(f.x, f.y);
                                    xl[n][i] = tm_pack(f.x, f.y);
                                }
                            }
                        }
#pragma unroll
                        for (int i = TERMS - 1; i >= 0; --i) {
                            if (F16 && i < TERMS - 1)
#pragma unroll
                                for (int n = 0; n < G; ++n)
#pragma unroll
                                    for (int p = 0; p < DW; ++p) tm_mma(part(step[p][n], y[p][a0 + n]), w[p][i], xl[n][0], xl[n][1]);
#pragma unroll
                            for (int n = 0; n < G; ++n)
#pragma unroll
                                for (int p = 0; p < DW; ++p) tm_mma(part(step[p][n], y[p][a0 + n]), w[p][i], xb[n][0], xb[n][1]);
                        }
                        if (TERMS > 2)
#pragma unroll
                            for (int n = 0; n < G; ++n)
#pragma unroll
                                for (int p = 0; p < DW; ++p)
#pragma unroll
                                    for (int i = 0; i < 4; ++i) y[p][a0 + n][i] += step[p][n][i];
                    }
                    if (k + PF < ks2) load(k + PF, q[u]);
                }
            }
        }
        uint32_t yb[DW][NA][2][TERMS];                   // (rows d of the tiles' lower and upper half; terms)
#pragma unroll
        for (int p = 0; p < DW; ++p)
#pragma unroll
            for (int at = 0; at < NA; ++at)
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int i = 0; i < TERMS; ++i) yb[p][at][h][i] = tm_term(y[p][at][2 * h], y[p][at][2 * h + 1]);
        // ---- X'[c][d] = sum_a P1[a][c] Y[a][d]
        for (int ct = ct0; ct < ct1; ++ct) {
            float acc[DW][2][4];
#pragma unroll
            for (int p = 0; p < DW; ++p)
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[p][i >> 2][i & 3] = 0.f;
#pragma unroll
            for (int k = 0; k < NA / 2; ++k) {
                uint4 w[TERMS];
                float step[DW][2][4] = {};
#pragma unroll
                for (int i = 0; i < TERMS; ++i) w[i] = A1[(size_t)((ct * (NA / 2) + k) * TERMS + i) * 32];
#pragma unroll
                for (int i = TERMS - 1; i >= 0; --i)     // term i of P1 with the terms of Y that leave 8 TERMS bits
#pragma unroll
                    for (int j = TERMS - 1 - i; j >= 0; --j)
#pragma unroll
                        for (int p = 0; p < DW; ++p)
#pragma unroll
                            for (int h = 0; h < 2; ++h) tm_mma(part(step[p][h], acc[p][h]), w[i], yb[p][2 * k][h][j], yb[p][2 * k + 1][h][j]);
                if (TERMS > 2)
#pragma unroll
                    for (int p = 0; p < DW; ++p)
#pragma unroll
                        for (int i = 0; i < 8; ++i) acc[p][i >> 2][i & 3] += step[p][i >> 2][i & 3];
            }
#pragma unroll
            for (int p = 0; p < DW; ++p)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int c = 16 * ct + g + 8 * h;
                    if (c < k1 && (DW == 1 || d0 + 16 * p < k2)) {
                        const size_t o = (size_t)m * K + (size_t)c * k2 + d0 + 16 * p + 4 * t;
                        const float4 r = make_float4(acc[p][0][2 * h], acc[p][0][2 * h + 1], acc[p][1][2 * h], acc[p][1][2 * h + 1]);
                        if (out_dt == BTC_F32) *reinterpret_cast<float4 *>(reinterpret_cast<float *>(xt) + o) = r;
                        else if (out_dt == BTC_BF16) *reinterpret_cast<uint2 *>(reinterpret_cast<uint16_t *>(xt) + o) = make_uint2(tm_pack(r.x, r.y), tm_pack(r.z, r.w));
                        else {
                            const __half2 lo = __floats2half2_rn(r.x, r.y), hi = __floats2half2_rn(r.z, r.w);
                            *reinterpret_cast<uint2 *>(reinterpret_cast<uint16_t *>(xt) + o) = make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
                        }
                    }
                }
        }
    }
}

template <int NA, int TERMS, bool F16, int K2, int DW>
static int launch_transform_mma(const void *x, const btc_transform &T, void *xt, int out_dt, int M, cudaStream_t s)
{
    auto kern = transform_mma_kernel<NA, TERMS, F16, K2, DW>;
    const int ks2 = T.k2 / 16, slices = (ks2 + DW - 1) / DW, nc = (T.k1 + 15) / 16;
    // Shares of c: as long as every quadrant of every SM gets at most one warp (each share computes Y again).  Slices per CTA:
    // as many as there are warps left, so that they read the same rows of x.
    const long long items = (long long)M * slices;
    const int sms = device_sms();
    int cg = 1;
    while (cg < 4 && 2 * cg <= nc && items * 2 * cg <= 4 * sms) cg *= 2;
    const int warps = items * cg <= 4 * sms ? 4 : TM_WARPS;
    TmPlan p;
    p.cg = cg;
    p.ds = 1;
    while (2 * p.ds <= warps / cg && p.ds < slices) p.ds *= 2;
    size_t smem;
    for (;; p.ds /= 2) {
        p.p2_frags = p.ds * DW * ks2;
        p.mask_off = (p.p2_frags + nc * (NA / 2)) * TERMS * 512;
        smem = p.mask_off + (size_t)NA * ks2 * 256;
        if (smem <= 227u * 1024u) break;
        if (p.ds == 1) return BTC_ERR_UNSUPPORTED;
    }
    p.rw = warps / (cg * p.ds);
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e);
    if (dev >= 64 || !((done.load(std::memory_order_relaxed) >> dev) & 1u)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return cuda_fail(e);
        if (dev < 64) done.fetch_or(uint64_t(1) << dev, std::memory_order_relaxed);
    }
    // as many CTAs as the SMs hold at once, each taking rows in turn
    const int gy = (slices + p.ds - 1) / p.ds;
    int gx = (M + p.rw - 1) / p.rw, most = sms / gy;
    if (most < 1) most = 1;
    if (gx > most) gx = most;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)gx, (unsigned)gy);
    cfg.blockDim = dim3(warps * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kern, static_cast<const uint16_t *>(x), T.sigma_bits, T.P1, T.P2, T.k1, T.k2, xt, out_dt, M, p);
    return e == cudaSuccess ? BTC_OK : cuda_fail(e);
}

template <int TERMS, bool F16, int K2, int DW>
static int launch_transform_k2(const void *x, const btc_transform &T, void *xt, int out_dt, int M, cudaStream_t s)
{
    if (T.k1 <= 16) return launch_transform_mma<2, TERMS, F16, K2, DW>(x, T, xt, out_dt, M, s);
    if (T.k1 <= 32) return launch_transform_mma<4, TERMS, F16, K2, DW>(x, T, xt, out_dt, M, s);
    if (T.k1 <= 48) return launch_transform_mma<6, TERMS, F16, K2, DW>(x, T, xt, out_dt, M, s);
    if (T.k1 <= 64) return launch_transform_mma<8, TERMS, F16, K2, DW>(x, T, xt, out_dt, M, s);
    if (T.k1 <= 96) return launch_transform_mma<12, TERMS, F16, K2, DW>(x, T, xt, out_dt, M, s);
    return launch_transform_mma<16, TERMS, F16, K2, DW>(x, T, xt, out_dt, M, s);
}

// k2 = 64 and 128 compiled in: 64 x 64, 16 / 63 / 64 / 512 / 2048 rows 4.0 / 4.8 / 4.0 / 8.4 / 19.6 us, with k2 an argument 4.0 / 5.1 /
// 4.2 / 9.3 / 21.4; 86 x 128 8.4 / 14.8 / 8.7 / 27.0 / 79.9 and 8.9 / 16.0 / 9.3 / 28.4 / 85.7; 40 x 128, 16 rows 4.2 and 5.1.
// Slices of 32 columns (half the instructions per product) where they give every quadrant of every SM more than one warp,
// else slices of 16: 86 x 128 at 200 rows, with a 2048-wide layer behind it, 38.9 -> 35.3 us, but at 130 rows 33.5 -> 37.5.
template <int TERMS, bool F16>
static int launch_transform_terms(const void *x, const btc_transform &T, void *xt, int out_dt, int M, cudaStream_t s)
{
    if constexpr (TERMS == 2) {
        const bool wide = (long long)M * (T.k2 / 32) > 4 * device_sms();
        if (wide && T.k2 == 64) return launch_transform_k2<TERMS, F16, 64, 2>(x, T, xt, out_dt, M, s);
        if (wide && T.k2 == 128) return launch_transform_k2<TERMS, F16, 128, 2>(x, T, xt, out_dt, M, s);
    }
    if (T.k2 == 64) return launch_transform_k2<TERMS, F16, 64, 1>(x, T, xt, out_dt, M, s);
    if (T.k2 == 128) return launch_transform_k2<TERMS, F16, 128, 1>(x, T, xt, out_dt, M, s);
    return launch_transform_k2<TERMS, F16, 0, 1>(x, T, xt, out_dt, M, s);
}

int launch_transform(const void *x, int x_dt, const btc_transform &T, void *xt, int out_dt, int M, int K, cudaStream_t s)
{
    if ((long long)T.k1 * T.k2 != K) return BTC_ERR_SHAPE;
    // (up to 8 rows the forms in fp32 have the shorter chain: with three layers of 4096 behind it, 64 x 64, one row 9.1 us where this one
    // took 11.5, eight rows 15.2 and 18.3, 86 x 128 35.4 and 42.3.  Below 64 rows three terms: the precision of the fp32 form; above, two carry more than 16-bit x.)
    if (x_dt != BTC_F32 && M > 8 && T.k2 % 16 == 0 && T.k1 <= 128) {
        const bool f16 = x_dt == BTC_F16;
        const int rc = M >= 64 ? (f16 ? launch_transform_terms<2, true>(x, T, xt, out_dt, M, s) : launch_transform_terms<2, false>(x, T, xt, out_dt, M, s))
                               : (f16 ? launch_transform_terms<3, true>(x, T, xt, out_dt, M, s) : launch_transform_terms<3, false>(x, T, xt, out_dt, M, s));
        if (rc != BTC_ERR_UNSUPPORTED) return rc;
    }
    // (k2 as compiled in; k1 up to two passes of 64 rows.  Up to 16 rows of X most of a pass is empty and a CTA of transform_kernel is small
    // too: 16 x 64, three rows, two layers of 4096 behind it 8.5 us, and 8.9 with this one; 32 x 64 9.4 and 9.0, 86 x 128 29.5 and 25.6.)
    if (x_dt != BTC_F32 && M <= 8 && T.k1 > 16 && T.k1 <= 128 && (T.k2 == 64 || T.k2 == 128)) {
        if (T.k2 == 64) return T.k1 <= 64 ? launch_transform_few<1, 64>(x, x_dt, T, xt, out_dt, M, s) : launch_transform_few<2, 64>(x, x_dt, T, xt, out_dt, M, s);
        return T.k1 <= 64 ? launch_transform_few<1, 128>(x, x_dt, T, xt, out_dt, M, s) : launch_transform_few<2, 128>(x, x_dt, T, xt, out_dt, M, s);
    }
    const size_t smem = ((size_t)K + 4 * T.k1 + 4 + (size_t)T.k2 * TR_DT + (size_t)T.k1 * TR_DT + (size_t)T.k1 * (T.k1 + 8)) * sizeof(float);
    if (smem > 200 * 1024) return BTC_ERR_UNSUPPORTED;
    cudaError_t e = cudaFuncSetAttribute(transform_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e);
    // rows per CTA: about two CTAs per SM in all (the P slabs are staged once per CTA and serve all its rows)
    const int tiles = (T.k2 + TR_DT - 1) / TR_DT;
    int groups = (2 * device_sms() + tiles - 1) / tiles;
    if (groups > M) groups = M;
    const int rows = (M + groups - 1) / groups;
    groups = (M + rows - 1) / rows;
    if (groups > 65535) return BTC_ERR_UNSUPPORTED;
    // programmatic launch: the kernel may start (and stage the factors) before its predecessor on the stream has finished
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)tiles, (unsigned)groups);
    cfg.blockDim = dim3(TR_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, transform_kernel, x, x_dt, T.sigma_bits, T.P1, T.P2, T.k1, T.k2, xt, out_dt, M, rows);
    return e == cudaSuccess ? BTC_OK : cuda_fail(e);
}

}  // namespace btc
