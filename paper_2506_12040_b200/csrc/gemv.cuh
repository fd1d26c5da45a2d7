// Decode path (M <= 8): device code, shared by gemv_int.cu and gemv_half.cu; gemv.cu plans the launches.
//
// One launch streams the index matrices of up to IM_MAXP independent layers once and evaluates every block dot
//     <x_j, C[idx]> = 2 * sum_{bit=1} x  -  sum x            (identity for +-1 codewords)
// (block-dot sum of the paper's appendix "Binary codebook LUT-GEMM") on the warp-level MMA.  Class c of a block are its
// weights 4c .. 4c+3.
//
// Integer form (M <= 2, v a multiple of 4).  The "byte-lane" codeword keeps weight t at bit (t >> 2) of byte (t & 3), so
// `word & (0x01010101 << c)` IS the four bytes {0 or 2^c} of class c: one LOP3 expands four weights into an A register of
// mma.sync.m16n8k32 (u8 x s8 -> s32).  B holds the activations as three balanced base-256 digits of a block-fixed-point
// integer X = rint(x * 2^s), |X| <= 2^(22 - cmax), pre-shifted by cmax - c; s comes from the largest magnitude among the
// slice's 32 blocks.  Digit d of row m is column 4m + d, so both rows of x see the same lanes and the same order of
// operations.  Digit sums are exact, and so is the sum of the X.
//
// fp16 form (M <= 8, v even).  A half with one bit p <= 11 set is the fp16 number 2^(p-24).  The "fp16 layout" codeword keeps
// weight t at bit (t & 1) * 16 + P0 + (t >> 1), P0 = 12 - 2 classes, so `word & (0x00010001 << (P0 + i))` is the pair of
// multiplicands {0 or 2^(P0+i-24)} of the weights 2i, 2i+1: one LOP3 per two weights for mma.sync.m16n8k16 against the
// activations themselves (row m of x is column m of B), as fp16 times 2^(E-i), E per (slice, row) from the largest magnitude
// so that nothing overflows and small activations keep their bits.  Exact products, fp32 sums.  The cost does not depend
// on M.
//
// Work split.  A tile is 16 output rows; a K-pass is P.slices (8, or 4 where those cover K: a function of K/v alone, so that
// in the integer form a layer's result does not depend on what shares its launch) slices of 4 BLK blocks, one warp each; the CTA's other warps take
// further tiles.  Lane (g = lane / 4, t = lane % 4) of a slice's warp owns rows g and g + 8 and the blocks BLK t .. BLK t +
// BLK - 1 of the slice; its activations stay in registers as B fragments for the pass.  NW = 8 warps (integer form): two CTAs
// per SM (<= 113 KB, 128 registers), which also lets the next launch's CTAs load their table and first indices while this
// launch computes.  NW = 16: one CTA per SM, for codeword tables too large for that, and for the fp16 form, whose
// fragments cost several times as much to build: there the warps of a slice share the work.
// Long K in the fp16 form (SPLIT): the kw CTAs of a cluster take the same rows and every kw-th pass, and add their sums through
// distributed shared memory in a fixed order; a CTA then builds fragments once or twice instead of once per pass.  A template
// parameter: the cluster's code in every launch cost the small ones 0.2 .. 0.5 us.
// Every tile leaves one partial result per (slice, row, m) in shared memory; after the last pass of a chunk of tiles the
// warps meet once, add the slices in a fixed order, apply alpha and mu and store.  Indices arrive through a ring of (tiles,
// pass) stages by TMA (boxes of 64 blocks with the 128-byte swizzle; rows past N and blocks past K/v arrive as zeros).
// There is no producer warp -- a ninth warp would cost every thread a quarter of its registers, which are handed out per SM
// quadrant -- the warps take turns to refill the stage that was just read.
// Bound: latency.  No pipe is above half (issue 0.51 per clock and quadrant, ALU 42 %, shared-memory wavefronts 37 %).  Clocks of
// a CTA, seven layers of 26 MB of indices, M = 1 (25 k from launch to launch): set-up, table and first indices 3.6 k, fragments
// 2 k (7.8 k for the layer of three passes), tiles 15.4 k at 1.3 k per stage (four warps per scheduler wait for gathers and
// MMAs in turn), meeting and sum 2 k.  13.2 us at M = 1 (the two kernels before it: 14.0; but 18.4, where they took 16.4, for a
// launch that overlaps no other), 23.1 at M = 8 (38.1).  One 4096 x 4096 layer, M = 1: 3.1 us in a graph, 4.3 a call, of which
// the host takes 3.6; 13824 x 5120, v = 20, M = 4: 13.0 (21.3).
// Every mbarrier wait is bounded; when one runs out the CTA raises the status word and drains.
#pragma once
#include <cuda.h>
#include <atomic>
#include <type_traits>
#include "btc_internal.cuh"

namespace btc {
namespace gv {

constexpr int MAX_STAGES = 8;
constexpr int MAX_SLICES = 8;

// blocks per lane: 8, or 4 where the fp16 form's fragments would take 80 registers
__host__ __device__ constexpr int lane_blocks(bool half, int ncls) { return half && ncls > 4 ? 4 : 8; }

struct Problem {
    const void *x;
    const void *tab;            // codewords: 32-bit words in the form's layout or, TAB_HALVES, byte-lane halves
    const __half *alpha;
    const __half *mu;           // may be nullptr
    void *y;
    int M, N, v, Kb;
    int xs;                     // elements from one row of x to the next
    int acc;                    // 1: add to what y (fp32) holds
    int x_dt, y_dt;
    int slices_log2, parts;     // slices per K-pass (2 or 3), K-passes
    int kw;                     // CTAs that share the passes: 1, or the cluster's size
    int tab_bytes;              // bytes of the table to stage in shared memory
    int cost, fixed;            // of one stage, and of a CTA's set-up (planning only)
    int groups, per, rem;       // stages' worth of rows (NW / slices tiles each); groups / workers and groups % workers (CTAs / kw)
    int cta_begin, cta_count;
};

struct Layout { int misc, stage_x, stage_x_pitch, park, chunk, tab, stage_bytes, stages, total; };   // (the ring comes first: 1024-byte alignment)

struct Batch {
    CUtensorMap map[IM_MAXP];   // indices: uint16 {K/v, N}, box {64, rows}, 128-byte swizzle; dense fields as 32-bit words, unswizzled
    Problem p[IM_MAXP];
    Layout L;
    int count;
    int tab_head;               // TAB_HEAD: entries staged in shared memory, the rest is gathered from global memory
    int *status;
};

enum { TAB_WORDS = 1, TAB_HEAD = 2, TAB_HALVES = 3 };

// Partial results parked between two meetings of the warps: (tile, slice) entries of 128 or 64 floats, NW per stage.
constexpr int max_park_entries(bool half) { return half ? 128 : 96; }
constexpr int entry_floats(bool half) { return half ? 128 : 64; }
// misc: mbarriers (2 MAX_STAGES + 1), abort flag, sum x per (slice, column)
constexpr int MISC_ABORT = (2 * MAX_STAGES + 1) * 8, MISC_SX = MISC_ABORT + 8;
constexpr int MISC_SXT = MISC_SX + MAX_SLICES * 8 * 4;       // (their sum, for the other CTAs of a cluster)
constexpr int MISC_BYTES = MISC_SXT + 8 * 4;
// Where x becomes B fragments.  Integer form, per warp: digit planes, 3 digits x (32 blocks, one spare per 8) x NCLS words.
// fp16 form, per slice: the rows of x (an even number) as 4 BLK blocks of NCLS quads of 16-bit numbers, in four quarters (what
// one t owns) 16 bytes apart, so that the 16-byte reads of two rows and four quarters fall on different banks; then E per row.
__host__ __device__ constexpr int plane_words(int ncls) { return 36 * ncls; }
__host__ __device__ constexpr int quarter_bytes(int ncls) { return lane_blocks(true, ncls) * ncls * 8 + 16; }
__host__ __device__ constexpr int stage_x_bytes(bool half, int ncls, int rows) { return half ? rows * 4 * quarter_bytes(ncls) + 32 : 12 * plane_words(ncls); }

// ------------------------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait, called by all 32 lanes of a warp together; the answer is the same in every lane (a vote), so the
// full-mask shuffles and MMAs that follow never see a split warp.  False once the limit (about 1 s) has passed or the
// CTA-wide abort flag is up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status,
                                          long long limit_clk = 2000000000LL) {
    bool ok = mbar_try(bar, parity);
    if (!__all_sync(0xffffffffu, ok)) {
        const long long t0 = clock64();
        int spins = 0;
        for (;;) {
            ok = mbar_try(bar, parity);
            if (__all_sync(0xffffffffu, ok)) break;
            __nanosleep(spins < 4 ? 20 : 100);
            if ((++spins & 255) == 0) {
                bool give_up = (*abort_flag != 0);
                if (!give_up && clock64() - t0 > limit_clk) {
                    *abort_flag = 1;
                    atomicExch(status, (int)BTC_ERR_TIMEOUT);
                    give_up = true;
                }
                if (__any_sync(0xffffffffu, give_up)) return false;
            }
        }
    }
    return true;
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar) : "memory");
}
// (B operands are 64-bit values, so that the two registers always sit in an aligned pair; ZERO: the accumulator starts at 0)
template <bool ZERO>
__device__ __forceinline__ void mma(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint64_t b) {
    if (ZERO)
        asm("{\n\t.reg .b32 b0, b1;\n\tmov.b64 {b0, b1}, %8;\n\t"
                     "mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {b0,b1}, {%9,%9,%9,%9};\n\t}"
                     : "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "l"(b), "r"(0));
    else
        asm("{\n\t.reg .b32 b0, b1;\n\tmov.b64 {b0, b1}, %8;\n\t"
                     "mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {b0,b1}, {%0,%1,%2,%3};\n\t}"
                     : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "l"(b));
}
template <bool ZERO>
__device__ __forceinline__ void mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint64_t b) {
    if (ZERO)
        asm("{\n\t.reg .b32 b0, b1;\n\tmov.b64 {b0, b1}, %8;\n\t"
                     "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {b0,b1}, {%9,%9,%9,%9};\n\t}"
                     : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "l"(b), "f"(0.f));
    else
        asm("{\n\t.reg .b32 b0, b1;\n\tmov.b64 {b0, b1}, %8;\n\t"
                     "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {b0,b1}, {%0,%1,%2,%3};\n\t}"
                     : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "l"(b));
}
__device__ __forceinline__ uint64_t pack2(uint32_t lo, uint32_t hi) { return (uint64_t)lo | ((uint64_t)hi << 32); }
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t a, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ float peer_ld(uint32_t a) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float4 peer_ld4(uint32_t a) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}
// Index stages are rewritten: these loads stay where they are (volatile); the codeword table is not: the compiler may move
// its loads (their addresses depend on an index that was read after the waits).
__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t a) {
    uint16_t v;
    asm("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
    return v;
}
// Two 16-bit indices packed in one word -> base + S * index of both.  A 16-bit dot product with (S, 0) or (0, S) takes the half
// out, scales it and adds the base in one instruction, and on the multiply-add pipe: the integer ALU, half as wide as the
// issue port, has all the masking to do (a widening 16-bit multiply-add compiles to two ALU instructions per index).
template <int S>
__device__ __forceinline__ void pair_addr(uint32_t pair, uint32_t base, uint32_t &lo, uint32_t &hi) {
    asm("dp2a.lo.u32.u32 %0, %1, %2, %3;" : "=r"(lo) : "r"(pair), "r"(S), "r"(base));
    asm("dp2a.lo.u32.u32 %0, %1, %2, %3;" : "=r"(hi) : "r"(pair), "r"(S << 8), "r"(base));
}
__device__ __forceinline__ __half2 half2_pow2(int e) {     // {2^e, 2^e}, -14 <= e <= 15
    const uint32_t h = (uint32_t)(15 + e) << 10, w = h | (h << 16);
    return *reinterpret_cast<const __half2 *>(&w);
}
__device__ __forceinline__ float pow2(int e) { return __uint_as_float((uint32_t)(127 + e) << 23); }

__device__ __forceinline__ float lo_half(uint32_t w) { return __half2float(__ushort_as_half((unsigned short)w)); }

// Codewords of the indices packed in `pair`.
template <int TAB>
__device__ __forceinline__ void lookup2(uint32_t pair, uint32_t s_tab, const uint32_t *gtab, uint32_t head, uint32_t &lo, uint32_t &hi)
{
    if (TAB == TAB_HEAD) {
        const uint32_t i0 = pair & 0xffffu, i1 = pair >> 16;
        lo = i0 < head ? lds32(s_tab + 4 * i0) : __ldg(gtab + i0);
        hi = i1 < head ? lds32(s_tab + 4 * i1) : __ldg(gtab + i1);
        return;
    }
    uint32_t a0, a1;
    pair_addr<TAB == TAB_HALVES ? 2 : 4>(pair, s_tab, a0, a1);
    if (TAB == TAB_HALVES) {
        lo = lds16(a0); hi = lds16(a1);
    } else {
        lo = lds32(a0); hi = lds32(a1);
    }
}

// NP pairs of consecutive IB-bit fields starting at bit `bit0` of a packed row at shared address `row` (4-byte aligned);
// up to one word past the last needed bit may be read.
template <int IB, int NP>
__device__ __forceinline__ void unpack_pairs(uint32_t row, uint32_t bit0, uint32_t *pair)
{
    constexpr int NW = (2 * NP * IB + 31) / 32;
    constexpr uint32_t mask = (1u << IB) - 1u;
    const uint32_t wp = row + ((bit0 >> 5) << 2), sh = bit0 & 31u;
    uint32_t w[NW + 1], a[NW + 1];
#pragma unroll
    for (int k = 0; k <= NW; ++k) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w[k]) : "r"(wp + 4 * k));
#pragma unroll
    for (int k = 0; k < NW; ++k) a[k] = __funnelshift_r(w[k], w[k + 1], sh);
    a[NW] = 0u;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        const int b0 = 2 * i * IB, b1 = b0 + IB;
        const uint32_t f0 = __funnelshift_r(a[b0 >> 5], a[(b0 >> 5) + 1], b0 & 31) & mask;
        const uint32_t f1 = __funnelshift_r(a[b1 >> 5], a[(b1 >> 5) + 1], b1 & 31) & mask;
        pair[i] = f0 | (f1 << 16);
    }
}

// Eight consecutive activations starting at element k as floats.
__device__ __forceinline__ void cvt8(const uint4 &q, int dt, float (&f)[8])
{
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (dt == BTC_F16) {
            const float2 p = __half22float2(*reinterpret_cast<const __half2 *>(&w[i]));
            f[2 * i] = p.x; f[2 * i + 1] = p.y;
        } else {
            f[2 * i] = __uint_as_float(w[i] << 16);
            f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
}
__device__ __forceinline__ void load8(const unsigned char *xrow, int dt, int k, bool in, float (&f)[8])
{
    if (dt == BTC_F32) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (in) {
            const float *src = reinterpret_cast<const float *>(xrow) + k;
            const uint4 qa = ld_x128(src), qb = ld_x128(src + 4);
            a = make_float4(__uint_as_float(qa.x), __uint_as_float(qa.y), __uint_as_float(qa.z), __uint_as_float(qa.w));
            b = make_float4(__uint_as_float(qb.x), __uint_as_float(qb.y), __uint_as_float(qb.z), __uint_as_float(qb.w));
        }
        f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
    } else {
        uint4 q = make_uint4(0u, 0u, 0u, 0u);
        if (in) q = ld_x128(reinterpret_cast<const uint16_t *>(xrow) + k);
        cvt8(q, dt, f);
    }
}

// Largest of `am` and the magnitudes (as bits) of eight fp16 or bf16 numbers, per half of the word.
__device__ __forceinline__ uint32_t abs_max16(const uint4 &q, uint32_t am)
{
    return __vmaxu2(__vmaxu2(__vmaxu2(am, q.x & 0x7fff7fffu), __vmaxu2(q.y & 0x7fff7fffu, q.z & 0x7fff7fffu)), q.w & 0x7fff7fffu);
}

// Scale of a set of activations from the bits of their largest magnitude: X = rint(x * sc) has |X| <= 2^pbits, inv = 1 / sc,
// both powers of two.  All zero: sc = inv = 0.  An inf or a nan: inv = nan, so every output of that row of x becomes nan.
__device__ __forceinline__ void fix_scale(uint32_t amax_bits, int pbits, float &sc, float &inv)
{
    const int ex = max((int)(amax_bits >> 23) - 126, -100);
    const bool nz = amax_bits != 0u && amax_bits < 0x7f800000u;
    sc = nz ? pow2(pbits - ex) : 0.0f;
    inv = nz ? pow2(ex - pbits) : (amax_bits == 0u ? 0.0f : __uint_as_float(0x7fc00000u));
}

// ------------------------------------------------------------------------------------ B fragments
// Integer form: two registers per pair of classes; the odd last class of two neighbouring blocks shares an MMA.
template <int NCLS, bool HALF, int BLK> struct Frags {
    static constexpr int NP = HALF ? NCLS : NCLS / 2;                       // MMAs per block
    static constexpr int NO = (!HALF && (NCLS & 1)) ? BLK / 2 : 0;         // shared ones
    uint64_t b[BLK][NP];
    uint64_t o[NO > 0 ? NO : 1];
};

// One tile against the fragments.  Integer form: two chains (an MMA need not wait for the one before it).  A 16-bit half h
// of the table stands for the byte-lane word whose low nibbles are those of h | (h << 12): the shift is a multiplication (the
// multiply-add pipe has room), the OR rides in the masking.
template <int NCLS, bool HALVES, int BLK>
__device__ __forceinline__ void mma_tile(const Frags<NCLS, false, BLK> &F, const uint32_t (&w0)[BLK], const uint32_t (&w1)[BLK], int (&acc)[2][4])
{
    auto pick = [](uint32_t w, uint32_t sw, uint32_t m) {
        uint32_t r;
        if (HALVES) asm("lop3.b32 %0, %1, %2, %3, 0xA8;" : "=r"(r) : "r"(w), "r"(sw), "r"(m));      // (w | sw) & m
        else r = w & m;
        return r;
    };
    uint32_t s0[BLK], s1[BLK];
#pragma unroll
    for (int e = 0; e < BLK; ++e) {
        s0[e] = HALVES ? w0[e] * 4096u : 0u;
        s1[e] = HALVES ? w1[e] * 4096u : 0u;
#pragma unroll
        for (int cp = 0; cp < NCLS / 2; ++cp) {
            constexpr int NP = NCLS / 2;
            const uint32_t ma = 0x01010101u << (2 * cp), mb = 0x01010101u << (2 * cp + 1);
            const uint32_t a0 = pick(w0[e], s0[e], ma), a1 = pick(w1[e], s1[e], ma), a2 = pick(w0[e], s0[e], mb), a3 = pick(w1[e], s1[e], mb);
            if (e * NP + cp < 2) mma<true>(acc[(e * NP + cp) & 1], a0, a1, a2, a3, F.b[e][cp]);
            else mma<false>(acc[(e * NP + cp) & 1], a0, a1, a2, a3, F.b[e][cp]);
        }
    }
    if (NCLS & 1) {
        const uint32_t ml = 0x01010101u << (NCLS - 1);
#pragma unroll
        for (int e = 0; e < BLK; e += 2)
            mma<false>(acc[(e >> 1) & 1], pick(w0[e], s0[e], ml), pick(w1[e], s1[e], ml), pick(w0[e + 1], s0[e + 1], ml), pick(w1[e + 1], s1[e + 1], ml), F.o[e / 2]);
    }
}
// fp16 form, blocks B0 .. B0 + NB - 1 of the lane (FIRST: the accumulators start at 0).
template <int NCLS, int B0, int NB, bool FIRST, int BLK>
__device__ __forceinline__ void mma_part(const Frags<NCLS, true, BLK> &F, const uint32_t (&w0)[NB], const uint32_t (&w1)[NB], float (&acc)[2][4])
{
    constexpr int P0 = 12 - 2 * NCLS;
#pragma unroll
    for (int e = 0; e < NB; ++e)
#pragma unroll
        for (int c = 0; c < NCLS; ++c) {
            const uint32_t ma = 0x00010001u << (P0 + 2 * c), mb = 0x00010001u << (P0 + 2 * c + 1);
            if (FIRST && e * NCLS + c < 2) mma<true>(acc[(e * NCLS + c) & 1], w0[e] & ma, w1[e] & ma, w0[e] & mb, w1[e] & mb, F.b[B0 + e][c]);
            else mma<false>(acc[(e * NCLS + c) & 1], w0[e] & ma, w1[e] & ma, w0[e] & mb, w1[e] & mb, F.b[B0 + e][c]);
        }
}

// X32 (fp16 form): fp32 activations; the integer form tells by P.x_dt.
template <int NCLS, bool HALF, int TAB, int IB, int NW, bool X32, bool SPLIT>
__global__ void __launch_bounds__(NW * 32, NW == 8 ? 2 : 1)
gemv_kernel(const __grid_constant__ Batch batch)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int CT = NW * 32;
    constexpr int BLK = lane_blocks(HALF, NCLS), SLB = 4 * BLK;      // blocks per lane, per slice
    constexpr int EF = entry_floats(HALF);
    using F = Frags<NCLS, HALF, BLK>;
    using A = typename std::conditional<HALF, float, int>::type;
    constexpr bool HALVES = TAB == TAB_HALVES;
    const Layout &L = batch.L;
    const uint32_t sbase = smem_addr(smem);
    volatile int *s_abort = reinterpret_cast<volatile int *>(smem + L.misc + MISC_ABORT);
    float *s_sx = reinterpret_cast<float *>(smem + L.misc + MISC_SX);            // [slice][8]
    float *s_park = reinterpret_cast<float *>(smem + L.park);
    const uint32_t s_tab = sbase + L.tab;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int NST = L.stages, RC = HALF ? L.chunk : max_park_entries(false) / NW;      // stages of the ring, stages per chunk
    auto bar_full = [&](int s) { return sbase + L.misc + 8 * s; };
    auto bar_empty = [&](int s) { return sbase + L.misc + 8 * (MAX_STAGES + s); };
    const uint32_t bar_tab = sbase + L.misc + 8 * (2 * MAX_STAGES);

    // the one layer this CTA works on, and its stages' worth of rows
    int pi = 0;
    while (pi + 1 < batch.count && (int)blockIdx.x >= batch.p[pi + 1].cta_begin) ++pi;
    const Problem &P = batch.p[pi];
    const int kw = SPLIT ? P.kw : 1, cta = (int)blockIdx.x - P.cta_begin;
    const int rank = SPLIT ? cta / kw : cta, kq = cta - rank * kw;  // worker, and which passes: kq, kq + kw, ...
    const int nown = SPLIT ? (P.parts - kq + kw - 1) / kw : P.parts;
    const int glo = rank * P.per + min(rank, P.rem), ghi = glo + P.per + (rank < P.rem ? 1 : 0);
    const int sl2 = P.slices_log2, SL = 1 << sl2, RG = NW >> sl2;    // slices, tiles per stage
    const int PW = SLB << sl2, SROWS = 16 * RG;                      // blocks per pass, rows per stage
    const uint32_t box = (uint32_t)SROWS * 128;                      // bytes of one box of indices

    // ---- index ring: number n of this CTA's walk (chunks of RC stages, passes, stages) sits in stage n % NST; warp n % NW
    //      sends for it
    const int total = (ghi - glo) * nown;
    auto issue = [&](int n, int st) {                    // (one lane)
        int c = glo, len = min(RC, ghi - c), j = 0;
        while (n >= len * nown) { n -= len * nown; c += len; len = min(RC, ghi - c); }
        while (n >= len) { n -= len; ++j; }
        j = kq + j * kw;
        const uint32_t dst = sbase + st * L.stage_bytes, bar = bar_full(st);
        mbar_expect_tx(bar, (uint32_t)L.stage_bytes);
        if constexpr (IB > 0) {
            tma_2d(dst, &batch.map[pi], j * (PW / 32 * IB), (c + n) * SROWS, bar);
        } else {
            for (int b = 0; b < PW / 64; ++b) tma_2d(dst + b * box, &batch.map[pi], j * PW + b * 64, (c + n) * SROWS, bar);
        }
    };
    if (tid == 0) {
        mbar_init(bar_tab, 1);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (total > 0) {
            mbar_expect_tx(bar_tab, (uint32_t)P.tab_bytes);
            bulk_g2s(s_tab, P.tab, (uint32_t)P.tab_bytes, bar_tab);
        }
    }
    if (warp < NST && lane == 0) {                       // (NST <= 8 <= NW)
        mbar_init(bar_full(warp), 1);
        mbar_init(bar_empty(warp), NW);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if ((HALF || warp == 0) && warp < total) issue(warp, warp);
    }
    if (HALF && P.v != 4 * NCLS)                         // the last class of a block has two weights: its other half stays zero
        for (int i = tid; i < MAX_SLICES * L.stage_x_pitch / 4; i += CT) reinterpret_cast<uint32_t *>(smem + L.stage_x)[i] = 0u;
    __syncthreads();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // Integer form: the other stages behind the table and the first one, which are waited for first, as copies are served in order (a
    // chain of 128 dependent launches 784.8 -> 779.0 us, q, k and v behind a transform 9.5 -> 9.4).  The fp16 form, which waits for
    // its activations longer, sends all before (6001 x 4096, v = 8, five rows 8.1 us, 8.3 that way).
    if (!HALF && warp > 0 && warp < NST && warp < total && lane == 0) issue(warp, warp);
    __syncwarp();

    const int g = lane >> 2, t = lane & 3;
    // MMA row g (and g + 8) carries tile row sg (and sg + 8): neighbouring g differ in bit 2 of the row, so the lanes of a
    // shared-memory phase read distinct swizzled chunks
    const int sg = ((g & 1) << 2) | (g >> 1);
    const int slice = warp & (SL - 1), rg = warp >> sl2;
    auto slice_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + slice), "r"(RG * 32) : "memory"); };      // the warps of a slice
    const int M = P.M, v = P.v, Kb = P.Kb;
    const bool x32 = HALF ? X32 : P.x_dt == BTC_F32, f16 = P.x_dt == BTC_F16;
    const unsigned char *x = static_cast<const unsigned char *>(P.x);
    const uint32_t *gtab = static_cast<const uint32_t *>(P.tab);
    const uint32_t head = (uint32_t)batch.tab_head;
    bool ok = true, tab_ready = false;
    int li = 0, s = 0;                                   // number in the walk; ring stage of the next tile to be read
    uint32_t rph = 0;
    // this lane's indices inside a stage (128-byte swizzle: 16-byte chunk c of row q sits at chunk c ^ (q & 7))
    const int boff = (slice * SLB + BLK * t) * 2;
    const uint32_t idx_off = sbase + (IB ? (uint32_t)((rg * 16 + sg) * (PW / 8 * IB))
                                         : (uint32_t)(boff >> 7) * box + (uint32_t)(rg * 16 + sg) * 128 + ((((boff >> 4) & 7) ^ sg) << 4) + (boff & 15));
    F B;
    // per lane: scale of the columns it holds (2t, 2t+1), and its share of sum x in them
    float ka = 0.f, kb = 0.f, kc = 0.f, kd = 0.f;
    float sx0 = 0.f, sx1 = 0.f;

    for (int c0 = glo; c0 < ghi; c0 += RC) {
        const int c1 = min(c0 + RC, ghi), nrows = (c1 - c0) * SROWS;
        // alpha / mu of the outputs this thread will finish (static data: loaded ahead of the dependency wait).  fp16 form: thread =
        // (tile, lane slot), rows sg and sg + 8; integer form: thread = (m, row)
        constexpr int OPT = (max_park_entries(HALF) / 4 * 32 + CT - 1) / CT * (HALF ? 2 : 1);
        uint32_t am_reg[OPT];                            // alpha below, mu above
        auto out_row = [&](int q) {
            if (HALF) return ((tid + (q >> 1) * CT) >> 5) * 16 + sg + 8 * (q & 1);
            const int o = tid + q * CT;
            return o >= nrows ? o - nrows : o;
        };
#pragma unroll
        for (int q = 0; q < OPT; ++q) {
            const int rl = out_row(q), n = c0 * SROWS + rl;
            am_reg[q] = 0;
            if (rl < nrows && n < P.N) {
                am_reg[q] = __ldg(reinterpret_cast<const unsigned short *>(P.alpha) + n);
                if (P.mu) am_reg[q] |= (uint32_t)__ldg(reinterpret_cast<const unsigned short *>(P.mu) + n) << 16;
            }
        }
        if (nown > 1 || c0 == glo) sx0 = sx1 = 0.f;

        for (int jj = 0; jj < nown && ok; ++jj) {
            const int j = kq + jj * kw;
            const int jb0 = j * PW + slice * SLB;                    // first block of the slice
            const int kleft = (Kb - jb0) * v;                        // activations from there to the end of the row (<= 0: an empty slice)
            // Integer form: a tile's codewords are looked up while the previous tile's MMAs are in flight, those of a pass's first
            // tile before the activations are waited for.  The fp16 form, whose fragments take twice the registers, carries the
            // indices over and looks four blocks up at a time.
            uint32_t pa[BLK / 2], pb[BLK / 2], w0[HALF ? 4 : BLK], w1[HALF ? 4 : BLK];
            auto lookup = [&](int p0, int np) {
#pragma unroll
                for (int i = 0; i < np; ++i) {
                    lookup2<TAB>(pa[p0 + i], s_tab, gtab, head, w0[2 * i], w0[2 * i + 1]);
                    lookup2<TAB>(pb[p0 + i], s_tab, gtab, head, w1[2 * i], w1[2 * i + 1]);
                }
            };
            auto fetch = [&]() {
                ok = mbar_wait(bar_full(s), rph, s_abort, batch.status);
                if (!ok) return;                                     // (a wait gave up: nothing is looked up any more)
                const uint32_t row = idx_off + s * L.stage_bytes;
                if constexpr (IB > 0) {
                    const uint32_t f = (uint32_t)((slice * SLB + BLK * t) * IB);
                    unpack_pairs<IB, BLK / 2>(row, f, pa);
                    unpack_pairs<IB, BLK / 2>(row + 8 * (PW / 8 * IB), f, pb);
                } else if constexpr (BLK == 8) {
                    const uint4 q = lds128(row), r = lds128(row + 1024);     // row + 8: same row & 7
                    pa[0] = q.x; pa[1] = q.y; pa[2] = q.z; pa[3] = q.w;
                    pb[0] = r.x; pb[1] = r.y; pb[2] = r.z; pb[3] = r.w;
                } else {
                    const uint2 q = lds64(row), r = lds64(row + 1024);
                    pa[0] = q.x; pa[1] = q.y; pb[0] = r.x; pb[1] = r.y;
                }
                // the index loads must have RETURNED before the stage is handed back: the arrive does not wait for loads in
                // flight, and the next copy into this stage may land within a few hundred clocks
#pragma unroll
                for (int i = 0; i < BLK / 2; ++i) asm volatile("" :: "r"(pa[i]), "r"(pb[i]) : "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_empty(s));
                if (++s == NST) { s = 0; rph ^= 1u; }
                if (!HALF) lookup(0, BLK / 2);
            };
            if (!tab_ready) {
                ok = mbar_wait(bar_tab, 0, s_abort, batch.status);
                tab_ready = true;
            }
            constexpr bool EARLY = HALF || NCLS <= 4;                // (v = 20: registers)
            if (EARLY && ok) fetch();
            if (jj == 0 && c0 == glo) asm volatile("griddepcontrol.wait;" ::: "memory");

            if (nown > 1 || c0 == glo) {
                if constexpr (HALF) {
                    // ---- the warps of a slice take its rows of x in turn: 8 activations per lane and step, left in shared memory block
                    //      by block; then lane (g = m, t) of each picks up its own blocks.  (Every lane reading its blocks from global
                    //      memory itself, each load on another line, took several times as long.)
                    constexpr int NPR = (SLB * 4 * NCLS / 8 + 31) / 32;  // steps per row
                    constexpr int QB = quarter_bytes(NCLS), RB = 4 * QB, MR = 8 / (NW / MAX_SLICES);     // most rows per warp
                    const int np = SLB * v / 8;                          // pieces of 8 activations
                    const int kin = min(kleft, SLB * v);
                    const uint32_t rcp = (65536u + v - 1) / v;
                    unsigned char *stage = smem + L.stage_x + slice * L.stage_x_pitch;
                    int *s_e = reinterpret_cast<int *>(stage + L.stage_x_pitch - 32);
                    uint4 raw[MR][NPR];
                    if (!x32) {
#pragma unroll
                        for (int i = 0; i < MR; ++i) {
                            const int m = rg + i * RG;
                            const unsigned char *src = x + ((size_t)m * P.xs + (size_t)jb0 * v + 8 * lane) * 2;
#pragma unroll
                            for (int u = 0; u < NPR; ++u) {
                                raw[i][u] = make_uint4(0u, 0u, 0u, 0u);
                                if (m < M && 8 * (lane + 32 * u) < kin) raw[i][u] = ld_x128(src + u * 512);
                            }
                        }
                    }
                    if (jj > 0 || c0 > glo) slice_sync();                 // (the fragments of the pass before have been picked up)
#pragma unroll
                    for (int i = 0; i < MR; ++i) {
                        const int m = rg + i * RG;
                        if (m < M) {
                            uint32_t am = 0u;
#pragma unroll
                            for (int u = 0; u < NPR; ++u) {
                                if (x32) {                               // (read twice; the second time from L1)
                                    float f[8];
                                    load8(x + (size_t)m * P.xs * 4, BTC_F32, jb0 * v + 8 * (lane + 32 * u), 8 * (lane + 32 * u) < kin, f);
#pragma unroll
                                    for (int k = 0; k < 8; ++k) am = max(am, __float_as_uint(f[k]) & 0x7fffffffu);
                                } else {
                                    am = abs_max16(raw[i][u], am);
                                }
                            }
                            if (!x32) am = max(am & 0xffffu, am >> 16);
                            am = __reduce_max_sync(0xffffffffu, am);
                            // largest magnitude f * 2^e, f in [1, 2): x * 2^(14 - e) stays below 2^15.  (fp16: E <= 15 keeps the factors
                            // representable, and what is smaller stays exact all the same)
                            const int e2 = f16 ? (int)(am >> 10) - 15 : (x32 ? (int)(am >> 23) : (int)(am >> 7)) - 127;
                            const int E = f16 ? min(14 - e2, 15) : min(max(14 - e2, -90), 100);
                            if (lane == 0) s_e[m] = E;
                            const float sc = pow2(x32 ? E : 0);
#pragma unroll
                            for (int u = 0; u < NPR; ++u) {
                                const int p = lane + 32 * u;
                                uint4 q = raw[i][u];
                                if (x32) {
                                    float f[8];
                                    load8(x + (size_t)m * P.xs * 4, BTC_F32, jb0 * v + 8 * p, 8 * p < kin, f);
                                    __half2 h[4];
#pragma unroll
                                    for (int k = 0; k < 4; ++k) h[k] = __floats2half2_rn(f[2 * k] * sc, f[2 * k + 1] * sc);
                                    q = *reinterpret_cast<const uint4 *>(h);
                                }
                                if (p < np) {
                                    if (v == 4 * NCLS) {                 // a quarter is BLK blocks = BLK NCLS / 2 pieces
                                        *reinterpret_cast<uint4 *>(stage + m * RB + p * 16 + (p / (BLK * NCLS / 2)) * 16) = q;
                                    } else {                             // v = 4 NCLS - 2: pair by pair into blocks of 4 NCLS
                                        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
                                        int blk = (int)((uint32_t)(8 * p) * rcp >> 16), pos = 8 * p - blk * v;
#pragma unroll
                                        for (int k = 0; k < 4; ++k) {
                                            *reinterpret_cast<uint32_t *>(stage + m * RB + blk * (8 * NCLS) + (blk / BLK) * 16 + pos * 2) = w[k];
                                            pos += 2;
                                            if (pos == v) { pos = 0; ++blk; }
                                        }
                                    }
                                }
                            }
                        }
                    }
                    slice_sync();
                    const int mg = min(g, M - 1);                        // (columns past M repeat the last row; nobody reads them)
                    const int Eg = s_e[mg], Elo = s_e[min(2 * t, M - 1)], Ehi = s_e[min(2 * t + 1, M - 1)];
                    // times 2^(E-i) for pair i (fp32 activations already carry 2^E).  The loads are volatile so that each is converted
                    // before many more have come in: raw and converted fragments together would not fit the registers.
                    const uint32_t src = smem_addr(stage) + mg * RB + t * QB;
                    auto scaled = [&](uint32_t w, int i) {
                        __half2 h;
                        if (!f16 && !x32) {
                            const float sc = pow2(Eg - i);
                            h = __floats2half2_rn(__uint_as_float(w << 16) * sc, __uint_as_float(w & 0xffff0000u) * sc);
                        } else {
                            h = __hmul2(*reinterpret_cast<const __half2 *>(&w), half2_pow2((f16 ? Eg : 0) - i));
                        }
                        return *reinterpret_cast<const uint32_t *>(&h);
                    };
#pragma unroll
                    for (int e = 0; e < BLK; ++e)
#pragma unroll
                        for (int c = 0; c < NCLS; ++c) {
                            if (NCLS % 2 == 0) {
                                if (c % 2 == 0) {
                                    const uint4 q = lds128(src + (e * NCLS + c) * 8);
                                    B.b[e][c] = pack2(scaled(q.x, 2 * c), scaled(q.y, 2 * c + 1));
                                    B.b[e][c + (NCLS > 1)] = pack2(scaled(q.z, 2 * c + 2), scaled(q.w, 2 * c + 3));
                                }
                            } else {
                                const uint2 q = lds64(src + (e * NCLS + c) * 8);
                                B.b[e][c] = pack2(scaled(q.x, 2 * c), scaled(q.y, 2 * c + 1));
                            }
                        }
                    // columns this lane holds: m = 2t, 2t+1; sum x from the same MMAs with all mask bits as A
                    ka = pow2(25 - (12 - 2 * NCLS) - Elo);
                    kb = pow2(25 - (12 - 2 * NCLS) - Ehi);
                    float all[2][4];
                    const uint32_t ones[4] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu};
                    mma_part<NCLS, 0, 4, true>(B, ones, ones, all);
                    if constexpr (BLK == 8) mma_part<NCLS, 4, 4, false>(B, ones, ones, all);
                    kc = (all[0][0] + all[1][0]) * (0.5f * ka);
                    kd = (all[0][1] + all[1][1]) * (0.5f * kb);
                    sx0 += kc; sx1 += kd;
                } else {
                    // ---- the warp quantises its slice (8 activations per lane and step), digit planes go through shared memory
                    constexpr float MAGIC = 12582912.0f;                 // 1.5 * 2^23: float -> int by addition
                    constexpr uint32_t MAGIC_BITS = 0x4B400000u;
                    constexpr int cmax = NCLS - 1, PBITS = 22 - cmax;
                    constexpr int NGR = SLB * 4 * NCLS / 8, NG = (NGR + 31) / 32;    // groups of 8 in a slice (v = 4 NCLS), per lane
                    constexpr int PSW = plane_words(NCLS);
                    uint32_t *planes = reinterpret_cast<uint32_t *>(smem + L.stage_x + warp * L.stage_x_pitch);
                    float inv_own = 0.f, sx_own = 0.f;                   // of the row of x whose digits this lane's columns hold
                    uint4 cur[NG];
                    auto load_row = [&](int m) {
#pragma unroll
                        for (int u = 0; u < NG; ++u) {
                            const int k = 8 * (lane + 32 * u);
                            cur[u] = make_uint4(0u, 0u, 0u, 0u);
                            if (!x32 && k < min(kleft, 8 * NGR))
                                cur[u] = ld_x128(x + ((size_t)m * P.xs + (size_t)jb0 * (4 * NCLS) + k) * 2);
                        }
                    };
                    load_row(0);
#pragma unroll
                    for (int e = 0; e < BLK; ++e)
#pragma unroll
                        for (int c = 0; c < F::NP; ++c) B.b[e][c] = 0ull;
#pragma unroll
                    for (int e = 0; e < F::NO; ++e) B.o[e] = 0ull;
#pragma unroll 1
                    for (int m = 0; m < M; ++m) {
                        uint32_t am = 0u;
#pragma unroll
                        for (int u = 0; u < NG; ++u) {
                            if (x32) {                                   // (read twice; the second time from L1)
                                float f[8];
                                load8(x + (size_t)m * P.xs * 4, BTC_F32, jb0 * (4 * NCLS) + 8 * (lane + 32 * u), 8 * (lane + 32 * u) < min(kleft, 8 * NGR), f);
#pragma unroll
                                for (int i = 0; i < 8; ++i) am = max(am, __float_as_uint(f[i]) & 0x7fffffffu);
                            } else {
                                am = abs_max16(cur[u], am);
                            }
                        }
                        if (!x32) {                                      // to the bits of an fp32 number
                            am = max(am & 0xffffu, am >> 16);
                            am = f16 ? __float_as_uint(__half2float(__ushort_as_half((unsigned short)am))) : am << 16;
                        }
                        int xs = 0;
                        float sc, inv;
                        fix_scale(__reduce_max_sync(0xffffffffu, am), PBITS, sc, inv);
#pragma unroll
                        for (int u = 0; u < NG; ++u) {
                            const int gi = lane + 32 * u;
                            if (gi < NGR) {
                                float f[8];
                                if (x32) load8(x + (size_t)m * P.xs * 4, BTC_F32, jb0 * (4 * NCLS) + 8 * gi, 8 * gi < kleft, f);
                                else cvt8(cur[u], P.x_dt, f);
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    const int blk = (2 * gi + h) / NCLS, c = 2 * gi + h - blk * NCLS;
                                    uint32_t *dst = planes + (blk + (blk >> 3)) * NCLS + c;
                                    const uint32_t sh = 1u << (cmax - c), off = 0x8080u - MAGIC_BITS * sh;     // modulo 2^32
                                    // Y = X * 2^(cmax - c) + 0x8080: byte d of Y is balanced digit d, + 0x80 for d < 2
                                    uint32_t y[4];
#pragma unroll
                                    for (int i = 0; i < 4; ++i) {
                                        const uint32_t b = (uint32_t)__float_as_int(fmaf(f[4 * h + i], sc, MAGIC));
                                        xs += (int)(b - MAGIC_BITS);
                                        y[i] = b * sh + off;
                                    }
                                    const uint32_t t0 = __byte_perm(y[0], y[1], 0x5140), t1 = __byte_perm(y[2], y[3], 0x5140);
                                    const uint32_t t2 = __byte_perm(y[0], y[1], 0x0062), t3 = __byte_perm(y[2], y[3], 0x0062);
                                    dst[0] = __byte_perm(t0, t1, 0x5410) ^ 0x80808080u;
                                    dst[PSW] = __byte_perm(t0, t1, 0x7632) ^ 0x80808080u;
                                    dst[2 * PSW] = __byte_perm(t2, t3, 0x5410);
                                }
                            }
                        }
                        if (m + 1 < M) load_row(m + 1);
                        xs = __reduce_add_sync(0xffffffffu, xs);
                        if (m == (t >> 1)) { inv_own = inv; sx_own = (float)xs * inv; }
                        __syncwarp();
                        if ((g >> 2) == m && (g & 3) < 3) {              // column 4 m + d
                            const uint32_t *src = planes + (g & 3) * PSW + 9 * t * NCLS;
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                const uint32_t *q = src + e * NCLS;
                                if (NCLS == 4) {
                                    const uint4 w = *reinterpret_cast<const uint4 *>(q);
                                    B.b[e][0] = pack2(w.x, w.y);
                                    B.b[e][F::NP - 1] = pack2(w.z, w.w);
                                } else {
#pragma unroll
                                    for (int c = 0; c < NCLS / 2; ++c) B.b[e][c] = pack2(q[2 * c], q[2 * c + 1]);
                                    if (NCLS & 1)
                                        B.o[e >> 1] = (e & 1) ? pack2((uint32_t)B.o[e >> 1], q[NCLS - 1]) : (uint64_t)q[NCLS - 1];
                                }
                            }
                        }
                        __syncwarp();
                    }
                    // lane t = 2 m holds digits 0 and 1 of row m, lane 2 m + 1 digit 2: weights of its two columns, times two for the
                    // identity, whose - sum x goes with the former
                    ka = ((t & 1) ? 131072.0f : 2.0f) / (float)(1 << cmax) * inv_own;
                    kb = ((t & 1) ? 0.0f : 512.0f) / (float)(1 << cmax) * inv_own;
                    kc = (t & 1) ? 0.f : sx_own;
                    sx0 += kc;
                }
            }
            if (!EARLY && ok) fetch();

            // ---- the tiles of the chunk, for this pass
            for (int r = c0; r < c1 && ok; ++r, ++li) {
                const int rs = s == 0 ? NST - 1 : s - 1;             // the stage this tile came from
                const uint32_t rs_phase = s == 0 ? rph ^ 1u : rph;
                A acc[2][4];
                if constexpr (HALF) {
                    lookup(0, 2);
                    mma_part<NCLS, 0, 4, true>(B, w0, w1, acc);
                    if constexpr (BLK == 8) {
                        lookup(2, 2);
                        mma_part<NCLS, 4, 4, false>(B, w0, w1, acc);
                    }
                } else {
                    mma_tile<NCLS, HALVES, BLK>(B, w0, w1, acc);
                }
                if (r + 1 < c1) fetch();
                float *park = s_park + (((r - c0) * RG + rg) * SL + slice) * EF + lane * (HALF ? 4 : 1);
                if constexpr (HALF) {
                    float4 *q = reinterpret_cast<float4 *>(park);
                    float4 o = make_float4(fmaf(acc[0][0] + acc[1][0], ka, -kc), fmaf(acc[0][1] + acc[1][1], kb, -kd),
                                           fmaf(acc[0][2] + acc[1][2], ka, -kc), fmaf(acc[0][3] + acc[1][3], kb, -kd));
                    if (jj > 0) { const float4 p = *q; o.x += p.x; o.y += p.y; o.z += p.z; o.w += p.w; }
                    *q = o;
                } else {
                    float lo = fmaf((float)(acc[0][0] + acc[1][0]), ka, fmaf((float)(acc[0][1] + acc[1][1]), kb, -kc));
                    float hi = fmaf((float)(acc[0][2] + acc[1][2]), ka, fmaf((float)(acc[0][3] + acc[1][3]), kb, -kc));
                    if (jj > 0) { lo += park[0]; hi += park[32]; }
                    park[0] = lo;
                    park[32] = hi;
                }
                // that stage takes what comes NST further on in the walk, once every warp has read it
                if (((li ^ warp) & (NW - 1)) == 0 && li + NST < total && ok) {
                    ok = mbar_wait(bar_empty(rs), rs_phase, s_abort, batch.status);
                    if (ok && lane == 0) issue(li + NST, rs);
                }
            }
        }
        if (P.mu && g == 0 && rg == 0) {
            if constexpr (HALF) { s_sx[slice * 8 + 2 * t] = sx0; s_sx[slice * 8 + 2 * t + 1] = sx1; }
            else s_sx[slice * 8 + t] = sx0;
        }
        // ---- the slices meet: add them in a fixed order, apply alpha (and mu), store
        __syncthreads();
        const bool fine = ok && !*s_abort;
        {
            auto finish = [&](int m, int n, float dot, float sx, float al, float mu) {
                float yv = al * dot + mu * sx;
                if (P.acc) yv += reinterpret_cast<const float *>(P.y)[(size_t)m * P.N + n];
                store_from_float(P.y, P.y_dt, (size_t)m * P.N + n, yv);
            };
            // sum over the slices of an output's partial results (integer form: output q of this thread; fp16 form: a lane's four)
            auto half_src = [&](int q) { return reinterpret_cast<float4 *>(s_park) + (size_t)((((tid + (q >> 1) * CT) >> 5)) << sl2) * 32 + lane; };
            auto half_sum = [&](int q) {
                float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
                const float4 *src = half_src(q);
                for (int w = 0; w < SL; w += 4)
#pragma unroll
                    for (int i = 0; i < 4; ++i) { const float4 p = src[(w + i) * 32]; d.x += p.x; d.y += p.y; d.z += p.z; d.w += p.w; }
                return d;
            };
            auto int_sum = [&](int q, int m) {           // tile row -> lane group g
                const int rl = out_row(q);
                const float2 *src = reinterpret_cast<const float2 *>(s_park + ((rl >> 4) << sl2) * EF + ((rl >> 3) & 1) * 32 + ((rl & 3) * 2 + ((rl >> 2) & 1)) * 4 + 2 * m);
                float d4[4] = {0.f, 0.f, 0.f, 0.f};
                for (int w = 0; w < SL; w += 4)
#pragma unroll
                    for (int i = 0; i < 4; ++i) { const float2 p = src[(w + i) * (EF / 2)]; d4[i] += p.x + p.y; }
                return (d4[0] + d4[1]) + (d4[2] + d4[3]);
            };
            auto half_finish = [&](int q, const float4 &d, float sxa, float sxb) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int n = c0 * SROWS + out_row(q + i);
                    if (n < P.N) {
                        const float al = lo_half(am_reg[q + i]), mu = lo_half(am_reg[q + i] >> 16);
                        finish(2 * t, n, i ? d.z : d.x, sxa, al, mu);
                        if (2 * t + 1 < M) finish(2 * t + 1, n, i ? d.w : d.y, sxb, al, mu);
                    }
                }
            };
            // sum of x of a row: over the slices (fp16 form: column c; integer form: c = 2 m, two columns)
            auto sx_sum = [&](int c) {
                float sx = 0.f;
                for (int w = 0; w < SL; ++w) sx += HALF ? s_sx[w * 8 + c] : s_sx[w * 8 + c] + s_sx[w * 8 + c + 1];
                return sx;
            };
            if (!SPLIT || kw == 1) {                     // (with kw == 1 every CTA of the cluster comes this way)
                if (fine) {
#pragma unroll
                    for (int q = 0; q < OPT; q += HALF ? 2 : 1) {
                        if constexpr (HALF) {
                            if (((tid + (q >> 1) * CT) >> 5) * 16 < nrows && 2 * t < M)
                                half_finish(q, half_sum(q), P.mu ? sx_sum(2 * t) : 0.f, P.mu ? sx_sum(2 * t + 1) : 0.f);
                        } else {
                            const int m = tid + q * CT >= nrows ? 1 : 0, rl = out_row(q), n = c0 * SROWS + rl;
                            if (m < M && rl < nrows && n < P.N)
                                finish(m, n, int_sum(q, m), P.mu ? sx_sum(2 * m) : 0.f, lo_half(am_reg[q]), lo_half(am_reg[q] >> 16));
                        }
                    }
                }
            } else if constexpr (SPLIT) {
                // this CTA's sums go to the entry of slice 0 (read by the same thread alone); a warp's outputs are finished by one CTA
                float *s_sxt = reinterpret_cast<float *>(smem + L.misc + MISC_SXT);
#pragma unroll
                for (int q = 0; q < OPT; q += 2)
                    if (((tid + (q >> 1) * CT) >> 5) * 16 < nrows && 2 * t < M) *half_src(q) = half_sum(q);
                if (P.mu && tid < M) s_sxt[tid] = sx_sum(tid);
                cluster_sync();
                auto peers = [&](uint32_t a) {           // (in the order of the CTAs)
                    float f[8], r = 0.f;
#pragma unroll
                    for (int k = 0; k < 8; ++k) f[k] = k < kw ? peer_ld(peer_addr(a, k)) : 0.f;
#pragma unroll
                    for (int k = 0; k < 8; ++k) r += f[k];
                    return r;
                };
                const uint32_t sxt = sbase + L.misc + MISC_SXT;
#pragma unroll
                for (int q = 0; q < OPT; q += 2) {
                    const int tl = (tid + (q >> 1) * CT) >> 5;
                    if (!fine || tl % kw != kq || tl * 16 >= nrows || 2 * t >= M) continue;
                    const uint32_t a = smem_addr(half_src(q));
                    float4 d = make_float4(0.f, 0.f, 0.f, 0.f), p[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) p[k] = k < kw ? peer_ld4(peer_addr(a, k)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int k = 0; k < 8; ++k) { d.x += p[k].x; d.y += p[k].y; d.z += p[k].z; d.w += p[k].w; }
                    half_finish(q, d, P.mu ? peers(sxt + 8 * t) : 0.f, P.mu && 2 * t + 1 < M ? peers(sxt + 8 * t + 4) : 0.f);
                }
                cluster_sync();                          // (nobody goes on while its sums are being read)
            }
        }
        if ((!SPLIT || kw == 1) && c1 < ghi) __syncthreads();        // the next chunk overwrites what was just read
    }
    // A CTA that gave up on a wait may still have copies in flight into its shared memory: let them land before it goes.
    if (*s_abort) {
        const long long t0 = clock64();
        while (clock64() - t0 < 400000LL) __nanosleep(1000);
        __syncthreads();
    }
}

// Which kernel: classes per block (v / 4 rounded up), table form, index bits (0: 16-bit containers), warps, fp32 activations.
struct Pick { int ncls, tab, ib, nw; bool x32; };

// grid > 0: launches in clusters of `cluster` CTAs.  grid == 0: writes the number of such clusters that fit the device at once.
template <int NCLS, bool HALF, int TAB, int IB, int NW, bool X32, bool SPLIT>
int launch_kernel(const Batch &b, int grid, int cluster, int *fit, cudaStream_t s)
{
    auto kern = gemv_kernel<NCLS, HALF, TAB, IB, NW, X32, SPLIT>;
    // the attribute is set once per device to all a CTA may ask for; which launch needs how much is the planner's business
    constexpr int most = NW == 8 ? 113 * 1024 : 227 * 1024;
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e);
    if (dev >= 64 || !((done.load(std::memory_order_relaxed) >> dev) & 1u)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess) return cuda_fail(e);
        if (dev < 64) done.fetch_or(uint64_t(1) << dev, std::memory_order_relaxed);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(NW * 32);
    cfg.dynamicSmemBytes = (size_t)b.L.total;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    if (grid == 0) {
        static std::atomic<int> known[16][9];
        int n = dev < 16 ? known[dev][cluster].load(std::memory_order_relaxed) : 0;
        if (!n) {
            cfg.gridDim = dim3((unsigned)cluster);
            cfg.dynamicSmemBytes = most;
            cfg.attrs = at + 1;
            cfg.numAttrs = 1;
            e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
            if (e != cudaSuccess) return cuda_fail(e);
            if (dev < 16) known[dev][cluster].store(n, std::memory_order_relaxed);
        }
        *fit = n;
        return BTC_OK;
    }
    e = cudaLaunchKernelEx(&cfg, kern, b);
    return e == cudaSuccess ? BTC_OK : cuda_fail(e);
}

// (one translation unit each)
int launch_int(const Batch &b, const Pick &k, int grid, int cluster, int *fit, cudaStream_t s);
int launch_half(const Batch &b, const Pick &k, int grid, int cluster, int *fit, cudaStream_t s);
int launch_half_split(const Batch &b, const Pick &k, int grid, int cluster, int *fit, cudaStream_t s);

template <bool HALF, bool SPLIT>
int dispatch(const Batch &b, const Pick &k, int grid, int cluster, int *fit, cudaStream_t s)
{
// (dense rows are read by no other kernel, so their forms go down to v = 4: 12 and 13 bits mean more than 2048 codewords, some of
// them repeated where v is 10 or less)
#define GV_CASE(C, T, I, W) if (k.ncls == C && k.tab == T && k.ib == I && k.nw == W) return launch_kernel<C, HALF, T, I, W, false, SPLIT>(b, grid, cluster, fit, s)
#define GV_TABLES(C, T) GV_CASE(C, T, 0, 8); GV_CASE(C, T, 0, 16)
#define GV_PACKED(C, T) GV_CASE(C, T, 12, 8); GV_CASE(C, T, 13, 8)
    if constexpr (HALF) {
#define GV_HALF(C, X) GV_CASE_X(C, TAB_WORDS, 0, X); GV_CASE_X(C, TAB_HEAD, 0, X)
#define GV_HALF_PACKED(C, X) GV_CASE_X(C, TAB_WORDS, 12, X); GV_CASE_X(C, TAB_WORDS, 13, X)
#define GV_CASE_X(C, T, I, X) if (k.ncls == C && k.tab == T && k.ib == I && k.x32 == X) return launch_kernel<C, true, T, I, 16, X, SPLIT>(b, grid, cluster, fit, s)
        GV_HALF(1, false); GV_HALF(2, false); GV_HALF(3, false); GV_HALF(4, false); GV_HALF(5, false); GV_HALF(6, false);
        GV_HALF(1, true); GV_HALF(2, true); GV_HALF(3, true); GV_HALF(4, true); GV_HALF(5, true);
        GV_HALF_PACKED(1, false); GV_HALF_PACKED(2, false); GV_HALF_PACKED(3, false); GV_HALF_PACKED(4, false);
        GV_HALF_PACKED(1, true); GV_HALF_PACKED(2, true); GV_HALF_PACKED(3, true); GV_HALF_PACKED(4, true);
#undef GV_CASE_X
#undef GV_HALF
#undef GV_HALF_PACKED
    } else {
        GV_TABLES(2, TAB_HALVES); GV_TABLES(3, TAB_HALVES); GV_TABLES(4, TAB_HALVES);
        GV_TABLES(5, TAB_WORDS); GV_CASE(5, TAB_HEAD, 0, 16);
        GV_PACKED(2, TAB_HALVES); GV_PACKED(3, TAB_HALVES); GV_PACKED(4, TAB_HALVES);
    }
#undef GV_TABLES
#undef GV_PACKED
#undef GV_CASE
    return BTC_ERR_UNSUPPORTED;
}

}  // namespace gv
}  // namespace btc
