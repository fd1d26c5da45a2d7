// Tensor-core path: y[M,N] = x[M,K] * W^[N,K]^T with W^ = alpha * C[idx] (+ mu), for large M.
//
// The contraction runs on the 5th-generation tensor cores (tcgen05.mma, kind::f16, fp32 accumulators in tensor
// memory).  The weight tile is the A operand (128 rows = UMMA M), x is the B operand (BM rows = UMMA N, loaded by TMA
// with the 128-byte swizzle), so the accumulator holds y^T: tensor-memory lane = output feature n, column = activation
// row m, and a warp stores 32 consecutive n for one m (coalesced).  The decoded tile is pure +-1 and the row scale is
// applied in the fp32 epilogue, which is exact for a row-wise alpha.
//
// Two kernels: gemm_ts_kernel (even v from 8 to 24; decoded weights go straight into tensor memory, see its header) and
// gemm_tcgen05_kernel (any v; one thread per weight row writes the +-1 tile into shared memory):
//   warp 0     TMA producer: x tiles [BM rows x 64 k] -> shared memory
//   warp 1     MMA issuer: one elected thread issues tcgen05.mma for every 64-wide k step
//   warp 2     allocates / frees tensor memory
//   warps 4-7  decode producers: thread r expands the indices of weight row n0+r for the current 64-wide k step into
//              +-1 bf16 (or fp16) in the swizzled K-major layout the MMA reads; afterwards the same warps run the
//              epilogue: tcgen05.ld, scale by alpha_n in fp32 (+ mu_n * sum_k x[m,k]), store y.
//
// Every mbarrier wait is bounded: after ~2 s of polling the CTA raises a status word, stops waiting and runs to
// completion (the output is then undefined and btc_device_status reports the timeout).
#include <cuda.h>
#include <atomic>
#include "btc_internal.cuh"

namespace btc {

constexpr int G_BN = 128;          // weight rows per tile (UMMA M)
constexpr int G_BK = 64;           // k per stage: 64 x 2 bytes = one 128-byte swizzle row
constexpr int G_THREADS = 256;
constexpr uint32_t G_A_BYTES = G_BN * G_BK * 2;

__device__ int g_gemm_status = 0;  // 0 = ok, 7 = a bounded wait ran out

// ------------------------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait.  Returns false (and latches *abort_flag) when the deadline passes.  BACKOFF: sleep between polls;
// every role but the MMA issuer uses it, because a warp that spins takes issue slots from the one thread whose
// instruction stream paces the tensor core.
template <bool BACKOFF = true>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    const long long t0 = clock64();
    int spins = 0;
    while (!mbar_try_wait(bar, parity)) {
        if (BACKOFF) __nanosleep(spins < 8 ? 32 : 128);
        if ((++spins & 63) == 0) {
            if (*abort_flag) return false;
            if (clock64() - t0 > 4000000000LL) {   // ~2 s at 2 GHz
                *abort_flag = 1;
                atomicExch(&g_gemm_status, (int)BTC_ERR_TIMEOUT);
                return false;
            }
        }
    }
    return true;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar) : "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// K-major, 128-byte-swizzled operand tile whose rows are 128 bytes: 8-row groups are 1024 bytes apart.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);          // start address, 16-byte units
    d |= (uint64_t)1 << 16;                            // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;                  // stride byte offset between 8-row groups
    d |= (uint64_t)1 << 46;                            // descriptor version for sm_100
    d |= (uint64_t)2 << 61;                            // SWIZZLE_128B
    return d;
}

struct GemmParams {
    LinearArgs a;
    const float *sumx;       // [M] row sums of x (only read when mu != nullptr)
    int k_tiles;             // ceil(K / 64)
};

// sum_k x[m,k] in fp32 (needed only for the mean term), a CTA per row.  The contraction that follows starts right away and
// waits for the sums in its epilogue.
__global__ void __launch_bounds__(256)
rowsum_kernel(const void *x, int x_dt, int K, float *out)
{
    __shared__ float s_part[8];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");      // (after the wait: x is complete for the contraction too)
    const int m = blockIdx.x, lane = threadIdx.x & 31;
    float s = 0.f;
    const uint4 *row = reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(x) + (size_t)m * K);   // (K is a multiple of 8)
#pragma unroll 4
    for (int i = threadIdx.x; i < K / 8; i += 256) {
        const uint4 q = ld_x128(row + i);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 f = x_dt == BTC_F16 ? __half22float2(*reinterpret_cast<const __half2 *>(&w[j]))
                                             : make_float2(__uint_as_float(w[j] << 16), __uint_as_float(w[j] & 0xffff0000u));
            s += f.x + f.y;
        }
    }
    s = warp_sum(s);
    if (lane == 0) s_part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < 8; ++w) t += s_part[w];
        out[m] = t;
    }
}

template <int BM, int STAGES>
__global__ void __launch_bounds__(G_THREADS, 1)
gemm_tcgen05_kernel(const __grid_constant__ CUtensorMap tmap_x, const GemmParams p)
{
    constexpr uint32_t B_BYTES = BM * G_BK * 2;
    constexpr uint32_t STAGE_BYTES = G_A_BYTES + B_BYTES;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // carve: stages (1024-byte aligned), then barriers
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char *smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_gen + (size_t)STAGES * STAGE_BYTES);
    // bars: [0,S) full_x, [S,2S) full_w, [2S,3S) empty, [3S] accum
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(bars + 3 * STAGES + 1);
    volatile int *s_abort = reinterpret_cast<volatile int *>(s_tmem + 1);

    const LinearArgs &a = p.a;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n0 = blockIdx.x * G_BN;
    const int m0 = blockIdx.y * BM;
    const int KT = p.k_tiles;
    const bool is_bf16 = (a.x_dt == BTC_BF16);

    auto bar_full_x = [&](int s) { return smem_u32(bars + s); };
    auto bar_full_w = [&](int s) { return smem_u32(bars + STAGES + s); };
    auto bar_empty = [&](int s) { return smem_u32(bars + 2 * STAGES + s); };
    const uint32_t bar_accum = smem_u32(bars + 3 * STAGES);

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(bar_full_x(s), 1);
            mbar_init(bar_full_w(s), 128);
            mbar_init(bar_empty(s), 1);
        }
        mbar_init(bar_accum, 1);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) tmem_alloc(smem_u32(s_tmem), BM);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_d = *s_tmem;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (x tiles)
        if (lane == 0) {
            for (int kt = 0; kt < KT; ++kt) {
                const int s = kt % STAGES;
                const uint32_t ph = (kt / STAGES) & 1;
                if (kt >= STAGES) mbar_wait(bar_empty(s), ph ^ 1, s_abort);
                mbar_expect_tx(bar_full_x(s), B_BYTES);
                const uint32_t dst = smem_base + s * STAGE_BYTES + G_A_BYTES;
                tma_load_2d(dst, &tmap_x, kt * G_BK, m0, bar_full_x(s));
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            // kind::f16 instruction descriptor: D = f32, A/B = bf16 or f16, both K-major, M = 128, N = BM
            uint32_t idesc = (1u << 4) | ((uint32_t)(BM >> 3) << 17) | ((uint32_t)(G_BN >> 4) << 24);
            if (is_bf16) idesc |= (1u << 7) | (1u << 10);
            for (int kt = 0; kt < KT; ++kt) {
                const int s = kt % STAGES;
                const uint32_t ph = (kt / STAGES) & 1;
                mbar_wait<false>(bar_full_x(s), ph, s_abort);
                mbar_wait<false>(bar_full_w(s), ph, s_abort);
                tc_fence_after();
                const uint32_t a_addr = smem_base + s * STAGE_BYTES;
                const uint64_t adesc = make_smem_desc(a_addr);
                const uint64_t bdesc = make_smem_desc(a_addr + G_A_BYTES);
#pragma unroll
                for (int k = 0; k < G_BK / 16; ++k)      // +32 bytes per 16-wide k step inside the swizzle row
                    umma_f16(tmem_d, adesc + 2 * k, bdesc + 2 * k, idesc, (kt | k) ? 1u : 0u);
                umma_commit(bar_empty(s));               // frees the stage when these MMAs have read it
            }
            umma_commit(bar_accum);                      // accumulator complete
        }
    } else if (warp >= 4) {
        // ------------------------------------------------------------ decode producers (weights -> A tile)
        const int r = tid - 128;                          // row inside the tile, also the TMEM lane
        const int n = min(n0 + r, a.N - 1);
        const uint16_t *irow = a.idx + (size_t)n * a.Kb;
        const uint32_t one2 = is_bf16 ? 0x3F803F80u : 0x3C003C00u;
        const int v = a.v;
        for (int kt = 0; kt < KT; ++kt) {
            const int s = kt % STAGES;
            const uint32_t ph = (kt / STAGES) & 1;
            // 64 weight bits of this row for k in [k0, k0+64), gathered from the public codeword words
            const int k0 = kt * G_BK;
            const int jf = k0 / v;
            const int jl = min((k0 + G_BK - 1) / v, a.Kb - 1);
            uint64_t win = 0;
            for (int j = jf; j <= jl; ++j) {
                const uint64_t w = __ldg(a.Cp + __ldg(irow + j));
                const int off = j * v - k0;
                win |= (off >= 0) ? (w << off) : (w >> (-off));
            }
            const uint64_t neg = ~win;                    // sign bit set where the weight is -1
            if (kt >= STAGES) mbar_wait(bar_empty(s), ph ^ 1, s_abort);
            unsigned char *arow = smem_gen + (size_t)s * STAGE_BYTES + (size_t)r * 128;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint32_t b = (uint32_t)(neg >> (8 * c)) & 0xFFu;
                uint4 q;
                q.x = one2 | ((b & 1u) << 15) | ((b & 2u) << 30);
                q.y = one2 | ((b & 4u) << 13) | ((b & 8u) << 28);
                q.z = one2 | ((b & 16u) << 11) | ((b & 32u) << 26);
                q.w = one2 | ((b & 64u) << 9) | ((b & 128u) << 24);
                *reinterpret_cast<uint4 *>(arow + ((c ^ (r & 7)) << 4)) = q;   // 128-byte swizzle
            }
            fence_proxy_async_smem();                     // make the generic-proxy writes visible to the MMA
            mbar_arrive(bar_full_w(s));
        }
        // ------------------------------------------------------------ epilogue
        mbar_wait(bar_accum, 0, s_abort);
        tc_fence_after();
        asm volatile("griddepcontrol.wait;" ::: "memory");    // the row sums
        const int nrow = n0 + r;
        const float al = __half2float(a.alpha[n]);
        const float mu = a.mu ? __half2float(a.mu[n]) : 0.f;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
#pragma unroll 1
        for (int c0 = 0; c0 < BM; c0 += 32) {
            uint32_t rr[32];
            tmem_ld32(tmem_d + lane_base + c0, rr);
            tmem_ld_wait();
            if (nrow < a.N) {
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const int m = m0 + c0 + i;
                    if (m < a.M) {
                        float y = al * __uint_as_float(rr[i]);
                        if (a.mu) y += mu * p.sumx[m];
                        store_from_float(a.y, a.y_dt, (size_t)m * a.N + nrow, y);
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*s_abort) {
        // give copies that may still be in flight time to land before shared memory is released
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 2) tmem_dealloc(tmem_d, BM);
}

// ------------------------------------------------------------------------------------ even v, weights in tensor memory
// With both operands in shared memory the kernel above is bound by shared-memory bandwidth: per 64-wide k step the
// tensor core reads the A and B tiles while the decode warps write 16 KB of A and TMA writes the x tile, more than
// the 128 bytes per clock an SM's shared memory delivers.  Here the decoded +-1 tile never touches shared memory: each
// decode thread owns one weight row = one tensor-memory lane, expands the row's 64 weights of a k step into 32
// registers and stores them with tcgen05.st into a ring of A tiles in tensor memory (32 columns per k step); the MMAs
// take A from tensor memory and only the x tile from shared memory.
//   warp 0 TMA producer (x tiles, table) | warp 1 MMA issuer | warp 2 tensor-memory allocation, index tiles
//   warps 4-19: four groups of four warps; group g expands the stages g, g + 4, ...; then all 16 run the epilogue.
// Tensor memory (512 columns): accumulator in columns [0, BM), A ring of STAGES x 32 KS columns from column 256.
//
// Index tiles (128 rows x 64 blocks = V k steps, 128-byte swizzle) arrive by TMA; the codeword table of the "fp16 layout" is
// bulk-copied into shared memory when it fits.  That layout keeps the bits of a weight pair (2j, 2j+1) of a block at
// P0 + j of both halves, so ((~w << (15 - P0 - j)) & 0x80008000) | {1.0, 1.0} is the pair as +-1 in bf16 / fp16: one
// shift and one LOP3 per pair.  v = 16: a k step is four whole blocks.  Other v: a step starts (64 step) mod v weights
// into a block; the V / gcd(V, 64) starting points are compiled in.
//
// An x tile has bn rows (a multiple of 16 up to BM; the UMMA N), chosen so that the tiles of M are even and the rows past M
// few.  Few tiles and a long K (SPLIT): the CTAs of a cluster along grid.z share K, leave their accumulators in shared
// memory, and each adds a share of the columns over the cluster in a fixed order (distributed shared memory).
//
// Launched with programmatic stream serialisation: barriers, tensor memory, table and first indices are ready before
// the predecessor has finished; x is read after it (or right away where the predecessor is the row-sum kernel, which
// itself waited for it; then the epilogue waits).  Its own successors may start early (a transform behind it: 13.0 -> 10.5 us for 24 rows,
// K = 1024).  With a mean term only when its k steps are done, and only where the next call is likely to begin with no
// more CTAs than there are SMs: a transform, or row sums of few rows.  Small CTAs that come while other tiles run go to the SMs
// that are idle or end first, eight to one, and the next contraction waits for those: 4096 x 4096 (v = 8) at 256 and 512 rows 16.1 and
// 19.9 us without, 17.5 and 22.7 when they came with any number of rows; below 33 rows there is nothing to gain (4096 x 11008, 16 rows 13.2 and
// 13.8).  With it 4096 x 11008 at 33 and 77 rows 14.8 -> 14.3 and 15.8 -> 15.3, a 40 x 64 transform and the layer behind it at 33 and 129
// rows 15.4 -> 13.2 and 18.3 -> 15.8.  (When the accumulator has been read, another 0.2 us with a mean term, but small calls
// without one took 0.1 us longer: 1000 x 1024, 77 rows 5.05 and 5.19.)
constexpr int G2_DWARPS = 16;                    // decode warps (four groups of four)
constexpr int G2_THREADS = 128 + G2_DWARPS * 32;
constexpr uint32_t G2_IDX_BYTES = 128 * 128;     // one index tile
constexpr int G4_A_COL0 = 256;

struct Gemm2Params {
    LinearArgs a;
    const float *sumx;       // [M] row sums of x, or nullptr
    const uint32_t *tab;     // fp16-layout codeword words [Kc4]
    int k_tiles;
    int tab_bytes;           // > 0: table staged in shared memory
    int bn;                  // rows of x per tile
    int early;               // with a mean term: the next kernel may start during the epilogue
};

struct SplitArgs {
    int split_tiles;         // k tiles (whole index tiles) per CTA along grid.z
};

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ float4 dsmem_ld128(uint32_t addr, uint32_t rank) {
    uint32_t peer;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(peer) : "memory");
    return v;
}

__device__ __forceinline__ void umma_f16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
        :: "r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
           "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
           "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
           "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__host__ __device__ constexpr int gcd64(int v) { return v % 16 == 0 ? 16 : v % 8 == 0 ? 8 : v % 4 == 0 ? 4 : 2; }   // (v even, below 32)
// Geometry of k step PH of an index tile of blocks of V: first pair of the step within its first block, blocks it touches.
__host__ __device__ constexpr int step_pair0(int V, int PH) { return (64 * PH % V) / 2; }
__host__ __device__ constexpr int step_blocks(int V) { return (64 + V - gcd64(V) + V - 1) / V; }

// The 64 weights of a k step from the (inverted) codewords of its blocks, for the starting point numbered ph.
template <int V, int PH>
__device__ __forceinline__ void expand_step(int ph, const uint32_t (&w)[step_blocks(V)], uint32_t one2, uint32_t (&regs)[32])
{
    constexpr int H = V / 2, P0 = 12 - 2 * ((V + 3) / 4);
    if (PH + 1 >= V / gcd64(V) || ph == PH) {
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int q = step_pair0(V, PH) + i, c = q / H, j = q - H * c;
            regs[i] = ((w[c] << (15 - P0 - j)) & 0x80008000u) | one2;
        }
    } else if constexpr (PH + 1 < V / gcd64(V)) {
        expand_step<V, PH + 1>(ph, w, one2, regs);
    }
}

__device__ __forceinline__ void put(float *p, float f) { *p = f; }
__device__ __forceinline__ void put(__half *p, float f) { *p = __float2half_rn(f); }
__device__ __forceinline__ void put(__nv_bfloat16 *p, float f) { *p = __float2bfloat16_rn(f); }

// One feature's results for up to 32 consecutive rows of y, from registers.  The type of y, the mean term and the end of the rows
// are looked at once per 32 rows: with a look at each of them for every element the epilogue, then a quarter of a CTA's time when x
// tiles are 256 rows high (a tenth now), was bound by the issue of its instructions (11008 x 4096, 2048 rows, fp32 result 164 -> 151 us; 4096 x 4096
// behind a transform, 512 rows, bf16 27.7 -> 25.1 us).  One pointer that advances, not 32 addresses side by side: those made the form
// with x tiles above 128 rows spill.
template <typename T>
__device__ __forceinline__ void store_column(T *y, int N, int rows, const uint32_t (&r)[32])
{
    if (rows >= 32) {
#pragma unroll
        for (int i = 0; i < 32; ++i, y += N) put(y, __uint_as_float(r[i]));
    } else {
#pragma unroll
        for (int i = 0; i < 32; ++i, y += N)
            if (i < rows) put(y, __uint_as_float(r[i]));
    }
}

template <int BM, int STAGES, int KS, bool SPLIT, int V>
__global__ void __launch_bounds__(G2_THREADS, 1)
gemm_ts_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_i, const Gemm2Params p, const SplitArgs sp)
{
    const uint32_t B_BYTES = (uint32_t)p.bn * G_BK * 2;            // one x tile (64 k); a stage holds KS of them
    const uint32_t STAGE_BYTES = KS * B_BYTES;
    constexpr int ACOLS = 32 * KS;                                 // tensor-memory columns of a stage's A tile
    constexpr int KPT = V;                                         // k steps per index tile
    constexpr int NBLK = step_blocks(V);                           // blocks a k step may touch
    static_assert(V % 2 == 0 && V >= 8 && V <= 24, "pairs of weights within 16-bit halves");
    // With x tiles of up to 128 rows an MMA runs for 64 clk or less, less than it takes one thread to issue it next to
    // sixteen busy decode warps; then two threads issue (warp 1: even stages into accumulator 0; warp 3: odd stages into
    // accumulator 1 in columns [128, 256)) and the epilogue adds the two accumulators.
    constexpr int NACC = (BM == 128) ? 2 : 1;
    static_assert(BM * ((BM == 128) ? 2 : 1) <= G4_A_COL0, "accumulators and A ring must not overlap");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char *smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    unsigned char *s_idx = smem_gen + (size_t)STAGES * STAGE_BYTES;                 // 2 index tiles
    uint32_t *s_tab = reinterpret_cast<uint32_t *>(s_idx + 2 * G2_IDX_BYTES);
    uint64_t *bars = reinterpret_cast<uint64_t *>(reinterpret_cast<unsigned char *>(s_tab) + ((p.tab_bytes + 15) & ~15));
    // One ring of STAGES stages holds both operands of a k step: the x tile in shared memory and the A tile in tensor
    // memory.  full[s]: the TMA arrival (with its bytes) plus the four decode warps; empty[s]: the MMAs' commit.
    // bars: [0,S) full, [S,2S) empty, accum, full_i[2], empty_i[2], tab_full
    static_assert(STAGES % 4 == 0 && STAGES * ACOLS <= 512 - G4_A_COL0 && KPT % KS == 0, "a decode group must meet a stage in consecutive phases");
    constexpr int NB = 2 * STAGES + 6;
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(bars + NB);
    volatile int *s_abort = reinterpret_cast<volatile int *>(s_tmem + 1);

    const LinearArgs &a = p.a;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int bn = p.bn;
    const int n0 = blockIdx.x * G_BN, m0 = blockIdx.y * bn;
    // a CTA covers the k tiles [kt_first, kt_first + KT): all of them, or its share along grid.z (whole index tiles)
    const int kt_first = SPLIT ? blockIdx.z * sp.split_tiles : 0;
    const int KT = SPLIT ? min(sp.split_tiles, p.k_tiles - kt_first) : p.k_tiles;
    const int NS = (KT + KS - 1) / KS;                              // stages' worth of k steps
    const bool is_bf16 = (a.x_dt == BTC_BF16);
    auto bar_full = [&](int s) { return smem_u32(bars + s); };
    auto bar_empty = [&](int s) { return smem_u32(bars + STAGES + s); };
    const uint32_t bar_accum = smem_u32(bars + 2 * STAGES);
    auto bar_full_i = [&](int b) { return smem_u32(bars + 2 * STAGES + 1 + b); };
    auto bar_empty_i = [&](int b) { return smem_u32(bars + 2 * STAGES + 3 + b); };
    const uint32_t bar_tab = smem_u32(bars + 2 * STAGES + 5);

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(bar_full(s), 1 + 4); mbar_init(bar_empty(s), 1); }
        mbar_init(bar_accum, NACC);
        for (int b = 0; b < 2; ++b) { mbar_init(bar_full_i(b), 1); mbar_init(bar_empty_i(b), G2_DWARPS); }
        mbar_init(bar_tab, 1);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) tmem_alloc(smem_u32(s_tmem), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_d = *s_tmem;
    if (!p.sumx) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 0) {
        if (lane == 0) {
            if (p.tab_bytes > 0) {
                mbar_expect_tx(bar_tab, (uint32_t)p.tab_bytes);
                bulk_g2s(smem_u32(s_tab), p.tab, (uint32_t)p.tab_bytes, bar_tab);
            }
            for (int ks = 0; ks < NS; ++ks) {
                const int kt0 = ks * KS;
                if (ks == 0 && !p.sumx) asm volatile("griddepcontrol.wait;" ::: "memory");     // x
                const int s = ks % STAGES;
                if (ks >= STAGES && !mbar_wait(bar_empty(s), ((ks / STAGES) & 1) ^ 1, s_abort)) break;
                mbar_expect_tx(bar_full(s), STAGE_BYTES);
#pragma unroll
                for (int j = 0; j < KS; ++j)             // (a box past K arrives as zeros)
                    tma_load_2d(smem_base + s * STAGE_BYTES + j * B_BYTES, &tmap_x, (kt_first + kt0 + j) * G_BK, m0, bar_full(s));
            }
        }
    } else if (warp == 2) {
        // Index tiles, as soon as there is room.  In turn with the x tiles, which wait for MMAs, a tile was sent for four stages before
        // its first use, less than it takes to arrive, and the decode warps stood there at every tile (1.6 k clk a stage of two k
        // steps, most of a round of the ring).  With this, and a stage's first step expanded before the stage is free: 4096 x
        // 11008, 77 rows 17.4 -> 15.8 us, 4096 x 4096 behind a transform, 512 rows 25.2 -> 23.1 (16.9 and 25.0 with the latter alone).
        // A ring of up to eight x tiles with its own barriers beside the four A tiles took it all back (17.3, 24.7).
        if (lane == 0) {
            for (int it = 0; it * KPT < KT; ++it) {
                const int ib = it & 1;
                if (it >= 2 && !mbar_wait(bar_empty_i(ib), ((it >> 1) & 1) ^ 1, s_abort)) break;
                mbar_expect_tx(bar_full_i(ib), G2_IDX_BYTES);
                tma_load_2d(smem_u32(s_idx + (size_t)ib * G2_IDX_BYTES), &tmap_i, (kt_first / KPT) * 64 + it * 64, n0, bar_full_i(ib));
            }
        }
        __syncwarp();
    } else if (warp == 1 || (NACC == 2 && warp == 3)) {
        if (lane == 0) {
            const int me = (warp == 1) ? 0 : 1;                    // which accumulator / which stages
            uint32_t idesc = (1u << 4) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(G_BN >> 4) << 24);
            if (is_bf16) idesc |= (1u << 7) | (1u << 10);
            const uint32_t d_tm = tmem_d + me * BM;
            for (int ks = me; ks < NS; ks += NACC) {
                const int s = ks % STAGES;
                if (!mbar_wait<false>(bar_full(s), (ks / STAGES) & 1, s_abort)) break;
                tc_fence_after();
                const uint32_t a_tm = tmem_d + G4_A_COL0 + s * ACOLS;
#pragma unroll
                for (int j = 0; j < KS; ++j) {
                    const uint64_t bdesc = make_smem_desc(smem_base + s * STAGE_BYTES + j * B_BYTES);
#pragma unroll
                    for (int k = 0; k < G_BK / 16; ++k)
                        umma_f16_ts(d_tm, a_tm + 32 * j + 8 * k, bdesc + 2 * k, idesc, (ks >= NACC || j || k) ? 1u : 0u);
                }
                umma_commit(bar_empty(s));
            }
            umma_commit(bar_accum);
        }
    } else if (warp >= 4) {
        const int r = (tid - 128) & 127;               // weight row of the tile = tensor-memory lane
        const int grp = (tid - 128) >> 7;              // k steps grp, grp + 4, ...: STAGES is a multiple of 4, so a stage is always
                                                       // met by the same group, phase after phase: its parity waits are unambiguous
        const uint32_t one2 = is_bf16 ? 0x3F803F80u : 0x3C003C00u;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const bool tab_smem = p.tab_bytes > 0;
        if (tab_smem && !mbar_wait(bar_tab, 0, s_abort)) { /* fall through: waits below bail out */ }
        bool ok = true;
        int cur_it = -1;
        for (int ks = grp; ks < NS && ok; ks += 4) {
            const int kt0 = ks * KS;
            const int it = kt0 / KPT, ib = it & 1;
            if (it != cur_it) {
                if (!mbar_wait(bar_full_i(ib), (it >> 1) & 1, s_abort)) { ok = false; break; }
                cur_it = it;
            }
            // the codewords of this row's blocks
            uint32_t w[KS][NBLK];
#pragma unroll
            for (int j = 0; j < KS; ++j) {
                const int ktl = kt0 + j - it * KPT;
                const unsigned char *irow_s = s_idx + (size_t)ib * G2_IDX_BYTES + (size_t)r * 128;
                uint32_t idx[NBLK];
                if constexpr (V == 16) {                         // (8 bytes)
                    const int boff = ktl * 8;
                    const uint2 quad = *reinterpret_cast<const uint2 *>(irow_s + ((((boff >> 4) & 7) ^ (r & 7)) << 4) + (boff & 15));
                    idx[0] = quad.x & 0xffffu; idx[1] = quad.x >> 16; idx[2] = quad.y & 0xffffu; idx[3] = quad.y >> 16;
                } else {
                    const int f = 64 * ktl / V;
#pragma unroll
                    for (int b = 0; b < NBLK; ++b) {             // (the last step of a tile ends with its last block)
                        const int boff = min(f + b, 63) * 2;
                        idx[b] = *reinterpret_cast<const uint16_t *>(irow_s + (((boff >> 4) ^ (r & 7)) << 4) + (boff & 15));
                    }
                }
#pragma unroll
                for (int b = 0; b < NBLK; ++b) w[j][b] = ~(tab_smem ? s_tab[idx[b]] : __ldg(p.tab + idx[b]));
            }
            if (((ks + 4) * KS) / KPT != it || ks + 4 >= NS) {   // this group's last stage in the index tile
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_empty_i(ib));
            }
            const int sa = ks % STAGES;
            // register i holds the weights 2i, 2i+1 of the k step (K elements 2i, 2i+1 of this row of A); those of a stage's first
            // step are ready before the stage is where it has two (with one the
            // MMAs set the pace)
            uint32_t regs[32];
            if (KS > 1) {
                expand_step<V, 0>(kt0 % (V / gcd64(V)), w[0], one2, regs);
#pragma unroll
                for (int i = 0; i < 32; ++i) asm volatile("" : "+r"(regs[i]));
            }
            if (ks >= STAGES && !mbar_wait(bar_empty(sa), ((ks / STAGES) & 1) ^ 1, s_abort)) { ok = false; break; }
            tc_fence_after();
#pragma unroll
            for (int j = 0; j < KS; ++j) {
                if (KS == 1 || j) expand_step<V, 0>((kt0 + j) % (V / gcd64(V)), w[j], one2, regs);
                tmem_st32(tmem_d + lane_base + G4_A_COL0 + sa * ACOLS + 32 * j, regs);
            }
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_full(sa));
        }
        // ------------------------------------------------------------ epilogue: four warps per lane quadrant
        if (p.early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        asm volatile("griddepcontrol.wait;" ::: "memory");     // (y, and the row sums)
        const int wl = warp - 4;
        const int q4 = wl & 3, quarter = wl >> 2;
        const int nl = q4 * 32 + lane, nrow = n0 + nl;
        const int nc = min(nrow, a.N - 1);
        const float al = SPLIT ? 0.f : __half2float(a.alpha[nc]);           // (before the wait: the last MMAs cover the loads)
        const float mu = !SPLIT && a.mu ? __half2float(a.mu[nc]) : 0.f;
        if (ok && mbar_wait(bar_accum, 0, s_abort)) {
            tc_fence_after();
            float *tile = reinterpret_cast<float *>(smem_gen);             // SPLIT: [bn][128], where the x tiles were
#pragma unroll 1
            for (int c0 = quarter * 32; c0 < bn; c0 += 128) {
                uint32_t rr[32];
                __syncwarp();                                      // (lanes past N did not store in the turn before)
                tmem_ld32(tmem_d + lane_base + c0, rr);
                if (NACC == 2 && NS > 1) {                         // (with a single stage accumulator 1 was never written)
                    uint32_t r2[32];
                    tmem_ld32(tmem_d + lane_base + BM + c0, r2);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; ++i) rr[i] = __float_as_uint(__uint_as_float(rr[i]) + __uint_as_float(r2[i]));
                } else {
                    tmem_ld_wait();
                }
                if (SPLIT) {
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (c0 + i < bn) tile[(c0 + i) * 128 + nl] = __uint_as_float(rr[i]);
                } else {
                    const int rows = min(bn - c0, a.M - m0 - c0);
                    if (a.mu) {
                        // (a row's sum per lane, handed to the warp: 32 of them in every thread left no registers for a CTA of the
                        // row sums beside this one; 11008 x 4096, 2048 rows, bf16 result 129 -> 123 us)
                        const float sums = lane < rows ? p.sumx[m0 + c0 + lane] : 0.f;
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            const float sx = __shfl_sync(0xffffffffu, sums, i);
                            rr[i] = __float_as_uint(__fmaf_rn(mu, sx, __fmul_rn(al, __uint_as_float(rr[i]))));
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i) rr[i] = __float_as_uint(al * __uint_as_float(rr[i]));
                    }
                    if (nrow < a.N && rows > 0) {
                        const size_t o = (size_t)(m0 + c0) * a.N + nrow;
                        if (a.y_dt == BTC_F32) store_column(reinterpret_cast<float *>(a.y) + o, a.N, rows, rr);
                        else if (a.y_dt == BTC_F16) store_column(reinterpret_cast<__half *>(a.y) + o, a.N, rows, rr);
                        else store_column(reinterpret_cast<__nv_bfloat16 *>(a.y) + o, a.N, rows, rr);
                    }
                }
            }
        }
    }
    if constexpr (SPLIT) {
        // (columns advance by whole multiples of 32 threads: a thread's four features stay the same, and what belongs to them is
        // fetched while the cluster meets)
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const int nq = (tid & 31) * 4, n = n0 + nq;
        __syncwarp();
        cluster_arrive();
        float al[4], mu[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            al[k] = __half2float(a.alpha[min(n + k, a.N - 1)]);
            mu[k] = a.mu ? __half2float(a.mu[min(n + k, a.N - 1)]) : 0.f;
        }
        cluster_wait();
        const int splits = gridDim.z, z = blockIdx.z;
        const int per = (bn + splits - 1) / splits, c1 = min(min(bn, a.M - m0), (z + 1) * per);
        if (!*s_abort)
            for (int c = z * per + (tid >> 5); c < c1; c += G2_THREADS / 32) {
                const int m = m0 + c;
                const float sx = a.mu ? p.sumx[m] : 0.f;
                float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int q = 0; q < splits; ++q) {
                    const float4 f = dsmem_ld128(smem_base + (uint32_t)(c * 128 + nq) * 4u, (uint32_t)q);
                    t.x += f.x; t.y += f.y; t.z += f.z; t.w += f.w;
                }
                const float v[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (n + k < a.N) {
                        float y = al[k] * v[k];
                        if (a.mu) y += mu[k] * sx;
                        store_from_float(a.y, a.y_dt, (size_t)m * a.N + n + k, y);
                    }
            }
        cluster_arrive();                                          // (nobody leaves while its shared memory is being read)
        cluster_wait();
    }
    tc_fence_before();
    __syncthreads();
    if (*s_abort) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 2) tmem_dealloc(tmem_d, 512);
}

// ------------------------------------------------------------------------------------ host side
typedef CUresult (*encode_tiled_fn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                    const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                    CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                    CUtensorMapFloatOOBfill);

static encode_tiled_fn get_encode()
{
    static encode_tiled_fn fn = nullptr;
    if (!fn) {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult qr;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qr) == cudaSuccess &&
            qr == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<encode_tiled_fn>(ptr);
    }
    return fn;
}

template <int BM, int STAGES>
static int launch_cfg(const CUtensorMap &tm, const GemmParams &p, cudaStream_t s)
{
    constexpr size_t smem = (size_t)STAGES * (G_A_BYTES + BM * G_BK * 2) + 1024 + (3 * STAGES + 1) * 8 + 16;
    auto kern = gemm_tcgen05_kernel<BM, STAGES>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e);
    dim3 grid((p.a.N + G_BN - 1) / G_BN, (p.a.M + BM - 1) / BM);
    kern<<<grid, G_THREADS, smem, s>>>(tm, p);
    return cuda_check_launch();
}

// Tiling of a (M, N, K) problem: rows of x per tile (bn), tiles of x, K splits (whole index tiles, clusters of up to eight).
// Time in clocks, fitted to measurements of every width at K = 2000 and 4096, made when the epilogue took longer: a CTA per SM in
// rounds, the last one as long as the others, each a fixed part (launch, tensor memory, first tiles, epilogue) and its k steps.  A step of tiles up to 128 wide
// costs what their MMAs and x tiles cost or the decode of its weights; wider ones have one issuing thread and cost
// about the same whatever their width: 11008 x 4096 at 300 rows took 53 us as two tiles of 160 and 36 as three of 112.  Clock
// stamps of the kernel as it is, v = 16, and as it was when this was fitted: a step 553 at 256 wide (its MMAs alone: 512), 232 at 128 and 219
// at 80 (351 and 325, index tiles in turn with x); set-up to first MMA 2.7 k, 3.2 k and 3.2 k (2.7 k, 3.5 k, 3.5 k), last MMA to end, the epilogue,
// 4.6 k, 2.2 k (12.1 k, 7.0 k) and, sum over the cluster included, 5.7 k.  So narrow steps are priced above what they now cost, and a wide
// tile may be taken where three rounds of narrow ones would be faster: the steps have not been fitted again.  The fixed parts alone
// have, and are kept on measurement (of the slower steps): with 12 000 and 7 000 for launches without a split the choice changes for
// one shape in nine and mostly for the worse (us, as is / 4 k less; v = 16, 8192 codewords): 512 x 11008 x 4096 (M x N x K) 47.2 / 46.6,
// 645 x 7822 x 1024 18.8 / 18.8, 714 x 7739 x 1024 18.1 / 19.0, 1776 x 3270 x 7424 76.6 / 77.1, 539 x 10900 x 5376 56.4 / 58.7, 12 x 6580 x 4352
// 12.8 / 15.0, 150 x 2050 x 2432 8.3 / 10.3, 230 x 3970 x 4992 16.0 / 18.3, 700 x 8000 x 1200 (v = 10) 25.5 / 32.9.  Codewords
// gathered from L1 / L2 (table too large for shared memory) share that path with the x tiles.  A split adds the sum over the
// cluster.
struct GemmPlan { int bn, mt, splits, split_tiles; };

static bool gemm_table_fits(int bn, int Kc)
{
    const size_t fixed = (size_t)4 * (bn > 128 ? 1 : 2) * bn * G_BK * 2 + 1024 + 2 * G2_IDX_BYTES + 512;
    return fixed + (size_t)((Kc + 3) / 4 * 4) * 4 <= 227u * 1024u;
}

static GemmPlan gemm_plan(int M, int N, int K, int v, int Kc)
{
    const int k_tiles = (K + G_BK - 1) / G_BK, rows = (N + G_BN - 1) / G_BN;
    const int idx_tiles = (k_tiles + v - 1) / v;
    const double decode = v == 16 ? 330.0 : v == 8 ? 430.0 : 350.0 + 20.0 * step_blocks(v);
    GemmPlan best = {0, 0, 1, k_tiles};
    double best_t = 0;
    const int sms = device_sms(), in_clusters = sms * 136 / 148;       // (clusters do not fill every GPC)
    for (int mt = (M + 255) / 256; mt <= (M + 255) / 256 + (M + 127) / 128; ++mt) {
        int bn = ((M + mt - 1) / mt + 15) / 16 * 16;
        if (bn < 16) bn = 16;
        const int mtn = (M + bn - 1) / bn;
        const bool wide = bn > 128;
        const double mma = 200.0 + 1.6 * bn, fit = wide ? decode + 230.0 : mma > decode ? mma : decode;
        const double far = wide ? 400.0 + 2.3 * bn : 480.0 + 2.2 * bn, step = gemm_table_fits(bn, Kc) || far < fit ? fit : far;
        for (int sp = 1; sp <= 8 && sp <= idx_tiles; ++sp) {
            const int per = (idx_tiles + sp - 1) / sp;                 // index tiles per split
            const int n = (idx_tiles + per - 1) / per;
            if (n != sp) continue;
            const long long ctas = (long long)rows * mtn * sp;
            const int at_once = sp == 1 ? sms : in_clusters > sp ? in_clusters / sp * sp : sp;
            const int steps = per * v < k_tiles ? per * v : k_tiles;
            const double t = (double)((ctas + at_once - 1) / at_once) * ((wide ? 16000.0 : 11000.0) + steps * step + (sp > 1 ? 3500.0 + 20.0 * bn : 0.0));
            if (best.bn == 0 || t < best_t) { best = {bn, mtn, sp, per * v}; best_t = t; }
        }
        if (M <= 256 && bn <= 32) break;
    }
    return best;
}

template <int BM, int STAGES, int KS, bool SPLIT, int V>
static int launch_ts(const CUtensorMap &tm, const CUtensorMap &ti, const Gemm2Params &p, const GemmPlan &g, cudaStream_t s)
{
    const size_t smem = (size_t)STAGES * KS * (p.bn * G_BK * 2) + 1024 + 2 * G2_IDX_BYTES + ((p.tab_bytes + 15) & ~15) +
                        (2 * STAGES + 6) * 8 + 16;
    auto kern = gemm_ts_kernel<BM, STAGES, KS, SPLIT, V>;
    static std::atomic<uint64_t> done{0};                          // (the attribute, once per device)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e);
    if (dev >= 64 || !((done.load(std::memory_order_relaxed) >> dev) & 1u)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return cuda_fail(e);
        if (dev < 64) done.fetch_or(uint64_t(1) << dev, std::memory_order_relaxed);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((p.a.N + G_BN - 1) / G_BN, g.mt, g.splits);
    cfg.blockDim = dim3(G2_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[3];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    // no more shared memory than asked for: what is left caches the codewords that come from global memory
    at[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    at[1].val.sharedMemCarveout = (unsigned)((smem + 1024) * 100 / (228 * 1024));
    at[2].id = cudaLaunchAttributeClusterDimension;
    at[2].val.clusterDim.x = 1; at[2].val.clusterDim.y = 1; at[2].val.clusterDim.z = (unsigned)g.splits;
    cfg.attrs = at;
    cfg.numAttrs = SPLIT ? 3 : 2;
    const SplitArgs sp = {g.split_tiles};
    e = cudaLaunchKernelEx(&cfg, kern, tm, ti, p, sp);
    return e == cudaSuccess ? BTC_OK : cuda_fail(e);
}

template <int V>
static int launch_ts_v(const CUtensorMap &tm, const CUtensorMap &ti, const Gemm2Params &p, const GemmPlan &g, cudaStream_t s)
{
    if (g.bn > 128) return g.splits > 1 ? launch_ts<256, 4, 1, true, V>(tm, ti, p, g, s) : launch_ts<256, 4, 1, false, V>(tm, ti, p, g, s);
    return g.splits > 1 ? launch_ts<128, 4, 2, true, V>(tm, ti, p, g, s) : launch_ts<128, 4, 2, false, V>(tm, ti, p, g, s);
}

size_t gemm_tcgen05_workspace_bytes(int M)
{
    return M > 8 ? (size_t)M * sizeof(float) : 0;   // row sums of x for the mean term
}

int launch_gemm_tcgen05(const LinearArgs &a, bool transformed, cudaStream_t s)
{
    if (a.K % 8) return BTC_ERR_UNSUPPORTED;                   // TMA row pitch must be a multiple of 16 bytes
    encode_tiled_fn enc = get_encode();
    if (!enc) return BTC_ERR_UNSUPPORTED;
    const bool ts = a.v >= 8 && a.v <= 24 && a.v % 2 == 0 && a.Kb % 8 == 0;
    const GemmPlan g = gemm_plan(a.M, a.N, a.K, ts ? a.v : 16, a.Kc);
    const int BM = ts ? g.bn : (a.M > 128 ? 256 : 128);

    CUtensorMap tm;
    const cuuint64_t dims[2] = {(cuuint64_t)a.K, (cuuint64_t)a.M};
    const cuuint64_t strides[1] = {(cuuint64_t)a.K * 2};
    const cuuint32_t box[2] = {(cuuint32_t)G_BK, (cuuint32_t)BM};
    const cuuint32_t estr[2] = {1, 1};
    const CUtensorMapDataType dt = a.x_dt == BTC_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    CUresult r = enc(&tm, dt, 2, const_cast<void *>(a.x), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cuda_fail(cudaErrorInvalidValue);

    GemmParams p;
    p.a = a;
    p.k_tiles = (a.K + G_BK - 1) / G_BK;
    p.sumx = nullptr;
    if (a.mu) {
        if (!a.workspace || a.workspace_bytes < (size_t)a.M * sizeof(float)) return BTC_ERR_WORKSPACE;
        float *sx = reinterpret_cast<float *>(a.workspace);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)a.M);
        cfg.blockDim = dim3(256);
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, rowsum_kernel, a.x, a.x_dt, a.K, sx);
        if (e != cudaSuccess) return cuda_fail(e);
        p.sumx = sx;
    }
    if (ts) {
        CUtensorMap ti;
        const cuuint64_t idims[2] = {(cuuint64_t)a.Kb, (cuuint64_t)a.N};
        const cuuint64_t istr[1] = {(cuuint64_t)a.Kb * 2};
        const cuuint32_t ibox[2] = {64, 128};
        if (enc(&ti, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, const_cast<uint16_t *>(a.idx), idims, istr, ibox, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS) {
            Gemm2Params q;
            q.a = a; q.sumx = p.sumx; q.k_tiles = p.k_tiles; q.bn = g.bn;
            q.early = a.mu && (transformed || (a.M > 32 && a.M <= device_sms()));
            const int Kc4 = (a.Kc + 3) / 4 * 4;
            q.tab = a.Cp + Kc4;
            // shared memory holds only x tiles (four stages), index tiles and the table
            q.tab_bytes = gemm_table_fits(g.bn, a.Kc) ? Kc4 * 4 : 0;
            switch (a.v) {
            case 8: return launch_ts_v<8>(tm, ti, q, g, s);
            case 10: return launch_ts_v<10>(tm, ti, q, g, s);
            case 12: return launch_ts_v<12>(tm, ti, q, g, s);
            case 14: return launch_ts_v<14>(tm, ti, q, g, s);
            case 16: return launch_ts_v<16>(tm, ti, q, g, s);
            case 18: return launch_ts_v<18>(tm, ti, q, g, s);
            case 20: return launch_ts_v<20>(tm, ti, q, g, s);
            case 22: return launch_ts_v<22>(tm, ti, q, g, s);
            default: return launch_ts_v<24>(tm, ti, q, g, s);
            }
        }
        return BTC_ERR_UNSUPPORTED;                            // (a shape the tensor map cannot describe)
    }
    if (BM == 256) return launch_cfg<256, 4>(tm, p, s);
    return launch_cfg<128, 6>(tm, p, s);
}

}  // namespace btc

extern "C" BTC_API int btc_device_status_reset(void)
{
    const int zero = 0;
    cudaError_t e = cudaMemcpyToSymbol(btc::g_gemm_status, &zero, sizeof(int));
    if (e != cudaSuccess) return btc::cuda_fail(e);
    int rc = btc::index_status_reset();
    if (rc != BTC_OK) return rc;
    rc = btc::km_status_reset();
    if (rc != BTC_OK) return rc;
    return btc::gemv_status_reset();
}

extern "C" BTC_API int btc_selftest_bounded_wait(void *stream)
{
    return btc::gemv_selftest_wait((cudaStream_t)stream);
}

extern "C" BTC_API int btc_device_status(int *status_host)
{
    if (!status_host) return BTC_ERR_NULL;
    int v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, btc::g_gemm_status, sizeof(int));
    if (e != cudaSuccess) return btc::cuda_fail(e);
    int v2 = 0;
    const int rc = btc::gemv_status_read(&v2);
    if (rc != BTC_OK) return rc;
    int v3 = 0;
    const int rc3 = btc::index_status_read(&v3);
    if (rc3 != BTC_OK) return rc3;
    int v4 = 0;
    const int rc4 = btc::km_status_read(&v4);
    if (rc4 != BTC_OK) return rc4;
    *status_host = v ? v : (v2 ? v2 : (v4 ? v4 : v3));
    return BTC_OK;
}

// ---------------------------------------------------------------------------------------------
// btc_linear_gemm for callers that cannot allocate: the row-sum scratch of the mean term lives in
// a fixed array of the device image instead of a caller-supplied workspace.
//
// In host code `g_static_scratch` is only a handle for the runtime, not a device address, so it
// must never be passed to a kernel as is; its address on the current device comes from
// cudaGetSymbolAddress, looked up once per device and cached.
#include <mutex>

namespace btc {

static __device__ __align__(256) unsigned char g_static_scratch[BTC_STATIC_SCRATCH_BYTES];

constexpr int MAX_DEVICES = 64;
static void *g_static_scratch_addr[MAX_DEVICES] = {};
static std::mutex g_static_scratch_mutex;

// Device address of g_static_scratch on the current device (cached per device); no allocation.
static int static_scratch_address(void **out)
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e);
    if (dev < 0 || dev >= MAX_DEVICES) return BTC_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_static_scratch_mutex);
    if (!g_static_scratch_addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess) return cuda_fail(e);
        if (!p) return cuda_fail(cudaErrorInvalidSymbol);
        g_static_scratch_addr[dev] = p;
    }
    *out = g_static_scratch_addr[dev];
    return BTC_OK;
}

}  // namespace btc

extern "C" BTC_API int btc_linear_gemm_static_scratch(const void *x, int x_dtype, const uint16_t *idx,
                                                      const uint32_t *C_packed, const void *alpha,
                                                      const void *mu, const btc_transform *T, void *y,
                                                      int y_dtype, int M, int N, int K, int v, int Kc,
                                                      void *stream)
{
    if (T) return BTC_ERR_UNSUPPORTED;
    if (v < 1 || v > 32 || Kc < 1 || Kc > 65536 || M < 1 || N < 1 || K < 1 || K % v) return BTC_ERR_SHAPE;
    if (btc::gemm_tcgen05_workspace_bytes(M) > (size_t)BTC_STATIC_SCRATCH_BYTES) return BTC_ERR_WORKSPACE;
    void *scratch = nullptr;
    const int rc = btc::static_scratch_address(&scratch);
    if (rc != BTC_OK) return rc;
    const size_t usable = (btc::gemm_tcgen05_workspace_bytes(M) + 255) / 256 * 256;
    return btc_linear_gemm(x, x_dtype, idx, C_packed, alpha, mu, nullptr, y, y_dtype, M, N, K, v, Kc, scratch,
                           usable, stream);
}
