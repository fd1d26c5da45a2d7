// Binary codebook construction (paper Section 4.1 "Flash and Accurate Binary Codebook"; loop of the appendix
// Algorithm "Binary Codebook Optimization"): initial centroids = the most frequent distinct vectors, then
//   E-step  z_i = argmin_k d_H(b_i, c_k)      (||b - c||^2 = 4 d_H; smallest k among equals)
//   M-step  c_k = element-wise majority of the vectors assigned to k  (ties -> +1; an empty cluster keeps its centroid)
// until no assignment changes or max_iter E-steps have run.
//
// Everything is done in the space of the 2^v possible patterns (v <= 20: the paper's range; 65536 of them at v = 16), not
// per vector: identical vectors have identical nearest centroids, so one histogram pass over the n vectors (the only pass
// that streams them, besides the final look-up of z) reduces every later step to at most 2^v weighted patterns.
//
// One cooperative launch, a CTA per SM, the steps separated by a barrier over the grid:
//   histogram  each CTA counts its vectors in shared memory as 16-bit counters (v <= 16: 128 KB; a hot pattern is a few
//              per cent of all vectors, and that many atomics on one address of L2 serialise), then adds the non-zero ones
//   ranking    rank(p) = #{q : (cnt[q], -q) > (cnt[p], -p)}, centroid rank(p) = p when rank(p) < c: a counting sort by frequency
//              (a histogram of the frequencies per part and in total; where a frequency's patterns of a part start is added
//              up once per frequency, and the part's patterns draw their places from there in word order; frequencies past the
//              last bin are ranked pairwise).  A CTA takes one part of the patterns, its
//              frequencies in shared memory, or several in turn where few SMs share 2^20 patterns
//   E-step     the Hamming distance is a sum over the bits, so min over k of (distance, k) for ALL patterns at once is a
//              separable min-plus convolution: start from key(c_k) = (0, k), and for every bit b
//              key(p) = min(key(p), key(p ^ 2^b) + (1, 0)).  v 2^v steps instead of distinct patterns x centroids (1 M
//              instead of 487 M for a 4096 x 4096 layer at v = 16 with 8192 centroids).  The low nine bits within 512
//              neighbouring patterns, the others on columns of four, with a grid barrier between.
//   M-step     every occurring pattern whose cluster is another than in the round before moves cnt[p] (total and counts of
//              its set bits, several counts to a 64-bit atomic) from that one's votes to the new one's, so that rounds in which
//              few move cast few votes and the one that finds nothing changed none; then one thread per centroid.  Where many
//              patterns share few centroids up to 32 copies of the votes are kept, and a warp per centroid adds them up
//   assign     z through the label table in shared memory (v <= 16)
// Bound: latency.  1 048 576 vectors, v = 16, 8192 centroids, two rounds: 46.0 us a call (50.4 us where a warp added up
// the parts before, and counted the equals before, for every pattern that it ranked; 58.7 us where in addition the round behind an
// M-step that changed no centroid was run to find that nothing changes: two barriers and both halves of its E-step).
// Clock stamps of the first CTA in thousands: clearing 2.3, histogram 12.9, patterns per frequency 2.8, suffix sums 1.6, ranking 5.6, E-step
// 2.8 + 9.6 with all votes cast, M-step 4.7, assignment 6.7; the six grid barriers, with the wait for the slowest CTA, 3.6 to 6.6 each.
// A move is two atomics per word where casting anew is one, so a round in which more than half of the patterns move costs more
// than that; on few centroids, where the votes are most of the call, the copies more than make up for it.  Two rounds, in the second
// of which three quarters of 65 536 patterns move: 16 centroids 331 us with all votes cast anew, 391 as differences in one copy,
// 65 in 32; 64 centroids 125, 142, 91; 256 centroids 80, 81, 74; 1024 centroids (one copy) 83.1, 83.6.  A run that converges
// in R rounds casts fewer votes than anew unless more than (R - 1) / 2 times the patterns move after the first.
// Integer arithmetic only; results are bit-exact against the definition.
#include <cuda.h>
#include <atomic>
#include "btc_internal.cuh"

namespace btc {

constexpr int KM_VMAX = 20;                  // longest vector: the steps keep tables of 2^v entries
constexpr int KM_THREADS = 1024;
constexpr int KM_BINS = 2048;                // frequencies 0 .. 2046, and all larger ones together
constexpr int KM_MAX_CTAS = 256;
constexpr int KM_LOW = 9;                    // bits of the first half of an E-step: 512 patterns
constexpr uint32_t KM_NONE = (255u << 16) | 0xffffu;
constexpr int KM_MAX_WORDS = 11;             // 64-bit words that hold 21 counts of 32 bits, two each
constexpr size_t KM_SMEM = 128 * 1024;
constexpr int KM_PART = 8192;                // most patterns per part of the ranking
// Patterns per centroid and copy of the votes.  v = 16, 256 centroids, three rounds (us): 98.9 at 32, 97.4 at 64, 100.3 at 128 and
// 109.2 in one copy; 1024 centroids: 105.4, 99.1, 99.1 and 98.6 (copies have to be cleared and summed).
constexpr int KM_CROWD = 64;
constexpr int KM_COPIES = 32;                // at most: a warp sums them up, one per lane
static_assert((1 << KM_VMAX) / KM_PART <= KM_MAX_CTAS && (3 * KM_BINS + 1 + 2 * KM_PART) * 4 <= KM_SMEM && KM_PART < 65536,
              "parts fit the columns, their frequencies and places shared memory, their counts 16 bits");

__device__ int g_km_status = 0;

struct KmState {                             // zeroed by the host, with the frequencies that follow it
    unsigned arrived;     // grid barrier
    int changed[2];       // set by the E-step of round i in slot i & 1
    int moved[2];         // the same for a centroid changed by the M-step of round i
    int n_over;           // patterns whose frequency is past the last bin
};

struct KmArgs {
    const uint32_t *vecs;
    size_t n;
    int v, Kc, max_iter;
    uint32_t *C;
    uint16_t *z;
    int *info;
    KmState *st;
    uint32_t *cnt;        // [P] frequencies
    uint32_t *seed;       // [P] key (0, k) at the centroids
    uint32_t *key;        // [P] after the low bits
    uint16_t *label;      // [P] assignment of the last E-step
    uint32_t *bins;       // [KM_BINS] patterns per frequency
    uint16_t *cols;       // [KM_BINS][KM_MAX_CTAS] the same per part
    uint2 *over;          // [P] (frequency, pattern) past the last bin
    unsigned long long *votes;   // [Kc][words]
    int words, fields;    // 64-bit words per centroid, counts per word
    int parts;            // of the patterns in the ranking: a CTA each, or several where there are few CTAs
};

__host__ __device__ inline size_t km_align(size_t x) { return (x + 255) & ~(size_t)255; }

// Carves the workspace (ws may be null: returns the bytes needed).
static size_t km_carve(KmArgs &a, void *ws, int v, int Kc, size_t n)
{
    const size_t P = (size_t)1 << v;
    size_t o = 0;
    auto take = [&](size_t bytes) { void *p = static_cast<char *>(ws) + o; o += km_align(bytes); return p; };
    a.fields = n < (1u << 21) ? 3 : 2;       // counts of 21 or 32 bits
    a.words = (v + 1 + a.fields - 1) / a.fields;
    a.st = static_cast<KmState *>(take(sizeof(KmState)));
    a.cnt = static_cast<uint32_t *>(take(P * 4));
    a.seed = static_cast<uint32_t *>(take(P * 4));
    a.key = static_cast<uint32_t *>(take(P * 4));
    a.label = static_cast<uint16_t *>(take(P * 2));
    a.bins = static_cast<uint32_t *>(take(KM_BINS * 4));
    a.cols = static_cast<uint16_t *>(take((size_t)KM_BINS * KM_MAX_CTAS * 2));
    a.over = static_cast<uint2 *>(take(P * 8));
    a.votes = static_cast<unsigned long long *>(take((size_t)Kc * a.words * 8));
    return o;
}

static size_t km_workspace_bytes(int v, int Kc)
{
    KmArgs a;
    return km_carve(a, nullptr, v, Kc, (size_t)1 << 31);   // (the wider counts)
}

// Barrier over the grid (co-resident: cooperative launch).  Bounded: false once about 2 s have passed.
__device__ __forceinline__ bool km_sync(KmState *st, unsigned &target, int *s_ok)
{
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned seen;
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(&st->arrived) : "memory");
        const long long t0 = clock64();
        int ok = 1;
        for (;;) {
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&st->arrived) : "memory");
            if ((int)(seen - target) >= 0) break;
            if (clock64() - t0 > 4000000000LL) {
                atomicExch(&g_km_status, (int)BTC_ERR_TIMEOUT);
                ok = 0;
                break;
            }
        }
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

// f(i, word) for every vector of [begin, end), or f4(i, four words) for four neighbours: 16-byte loads, four in flight.
template <typename F, typename F4>
__device__ __forceinline__ void km_stream(const uint32_t *__restrict__ vecs, size_t begin, size_t end, F f, F4 f4)
{
    if ((reinterpret_cast<uintptr_t>(vecs) & 15u) == 0) {   // (begin is a multiple of 4, or the end)
        const uint4 *src = reinterpret_cast<const uint4 *>(vecs);
        const size_t q1 = end / 4;
        for (size_t q0 = begin / 4; q0 < q1; q0 += 4 * KM_THREADS) {
            uint4 w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const size_t q = q0 + threadIdx.x + u * KM_THREADS;
                if (q < q1) w[u] = __ldg(src + q);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const size_t q = q0 + threadIdx.x + u * KM_THREADS;
                if (q < q1) f4(4 * q, w[u]);
            }
        }
        begin = max(begin, end & ~(size_t)3);                // (an empty share may start inside the last four)
    }
    for (size_t i = begin + threadIdx.x; i < end; i += KM_THREADS) f(i, __ldg(vecs + i));
}

template <typename F>
__device__ __forceinline__ void km_stream(const uint32_t *__restrict__ vecs, size_t begin, size_t end, F f)
{
    km_stream(vecs, begin, end, f, [&](size_t i, const uint4 &w) { f(i, w.x); f(i + 1, w.y); f(i + 2, w.z); f(i + 3, w.w); });
}

// CROWDED: there may be patterns enough per centroid for copies of the votes.
template <bool CROWDED>
__global__ void __launch_bounds__(KM_THREADS, 1)
km_kernel(const KmArgs a)
{
    extern __shared__ __align__(16) unsigned char km_smem[];
    __shared__ int s_ok;
    __shared__ uint32_t s_warp[32];
    __shared__ int s_listed, s_overs;
    uint32_t *sm = reinterpret_cast<uint32_t *>(km_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int G = gridDim.x, b = blockIdx.x, v = a.v, P = 1 << v, Kc = a.Kc;
    const uint32_t mask = (uint32_t)P - 1u;
    const int gid = b * KM_THREADS + tid, gthreads = G * KM_THREADS;
    unsigned target = 0;

    // ---- clear what the steps after the next barrier add to (the frequencies and the state arrive cleared)
    for (int i = gid; i < P; i += gthreads) a.seed[i] = KM_NONE;
    for (int i = gid; i < KM_BINS; i += gthreads) a.bins[i] = 0u;
    for (int i = gid; i < Kc; i += gthreads) a.C[i] = 0u;
    for (int i = gid; i < KM_BINS * KM_MAX_CTAS / 8; i += gthreads) reinterpret_cast<uint4 *>(a.cols)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (size_t i = gid; i < (size_t)Kc * a.words; i += gthreads) a.votes[i] = 0ull;

    // ---- histogram
    const size_t share = ((a.n + G - 1) / G + 3) & ~(size_t)3;
    const size_t v0 = min(a.n, share * b), v1 = min(a.n, share * (b + 1));
    if (v <= 16) {
        const int hw = max(P / 2, 1);
        for (int i = tid; i < hw; i += KM_THREADS) sm[i] = 0u;
        constexpr size_t MOST = 65532;                       // (16-bit counters; a multiple of 4)
        for (size_t c0 = v0; c0 < v1; c0 += MOST) {
            __syncthreads();
            km_stream(a.vecs, c0, min(v1, c0 + MOST), [&](size_t, uint32_t w) { w &= mask; atomicAdd(sm + (w >> 1), 1u << (16 * (w & 1u))); });
            __syncthreads();
            for (int i = tid; i < hw; i += KM_THREADS) {
                const uint32_t w = sm[i];
                if (w & 0xffffu) atomicAdd(a.cnt + 2 * i, w & 0xffffu);
                if (w >> 16) atomicAdd(a.cnt + 2 * i + 1, w >> 16);
                sm[i] = 0u;
            }
        }
    } else {
        km_stream(a.vecs, v0, v1, [&](size_t, uint32_t w) { atomicAdd(a.cnt + (w & mask), 1u); });
    }
    if (!km_sync(a.st, target, &s_ok)) return;

    // ---- patterns per frequency: part by part, the frequencies of the last one kept in shared memory
    const int per = (P + a.parts - 1) / a.parts;
    uint32_t *s_bins = sm, *s_cnt = sm + KM_BINS + 1;
    for (int q = b; q < a.parts; q += G) {
        const int p0 = min(P, per * q), p1 = min(P, p0 + per);
        for (int i = tid; i < KM_BINS; i += KM_THREADS) s_bins[i] = 0u;
        __syncthreads();
        for (int p = p0 + tid; p < p1; p += KM_THREADS) {
            const uint32_t c = __ldcg(a.cnt + p);
            s_cnt[p - p0] = c;
            if (c) atomicAdd(s_bins + min(c, (uint32_t)KM_BINS - 1u), 1u);
            if (c >= KM_BINS - 1) a.over[atomicAdd(&a.st->n_over, 1)] = make_uint2(c, (uint32_t)p);
        }
        __syncthreads();
        for (int i = tid; i < KM_BINS; i += KM_THREADS) {        // (the thread that clears the bin for the next part)
            const uint32_t h = s_bins[i];
            if (h) { a.cols[(size_t)i * KM_MAX_CTAS + q] = (uint16_t)h; atomicAdd(a.bins + i, h); }
        }
    }
    if (!km_sync(a.st, target, &s_ok)) return;

    // ---- suffix sums: s_bins[i] = patterns of frequency bin >= i
    {
        uint32_t x1 = __ldcg(a.bins + KM_BINS - 1 - 2 * tid), x0 = __ldcg(a.bins + KM_BINS - 2 - 2 * tid);   // (from the top)
        if (tid == KM_BINS / 2 - 1) x0 = 0u;                 // (frequency 0 does not occur)
        uint32_t s = x1 + x0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, s, o); if (lane >= o) s += t; }
        if (lane == 31) s_warp[warp] = s;
        __syncthreads();
        if (warp == 0) {
            uint32_t w = s_warp[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, w, o); if (lane >= o) w += t; }
            s_warp[lane] = w;
        }
        __syncthreads();
        if (warp) s += s_warp[warp - 1];
        s_bins[KM_BINS - 2 - 2 * tid] = s;
        s_bins[KM_BINS - 1 - 2 * tid] = s - x0;
        if (tid == 0) s_bins[KM_BINS] = 0u;
        __syncthreads();
    }
    const int n_unique = (int)s_bins[1], kc = min(Kc, n_unique);

    // ---- ranks: centroids, and the seeds of the first E-step.  A part lists the frequencies that can rank below c, a warp adds up each
    //      one's patterns in the parts before (a 16-byte load per lane, four in flight), and the part's own patterns then draw their
    //      places from that start, 32 at a time in word order, those of a frequency found by a match over the warp.
    uint32_t *s_next = s_cnt + KM_PART, *s_list = s_next + KM_BINS;     // next free rank of a frequency; the frequencies listed
    uint32_t *s_over = s_list + KM_BINS;                                // patterns of the part past the last bin
    constexpr uint32_t UNSEEN = 0xffffffffu, LISTED = 0xfffffffeu;
    for (int q = b; q < a.parts; q += G) {
        const int p0 = min(P, per * q), np = min(P, p0 + per) - p0;
        __syncthreads();
        for (int i = tid; i < KM_BINS; i += KM_THREADS) s_next[i] = UNSEEN;
        if (tid == 0) s_listed = s_overs = 0;
        if (a.parts > G)                                     // (several parts: their frequencies again)
            for (int i = tid; i < np; i += KM_THREADS) s_cnt[i] = __ldcg(a.cnt + p0 + i);
        __syncthreads();
        auto ranked = [&](uint32_t c) { return c != 0u && c < KM_BINS - 1 && s_bins[c + 1] < (uint32_t)Kc; };
        for (int i = tid; i < np; i += KM_THREADS) {
            const uint32_t c = s_cnt[i];
            if (ranked(c) && atomicExch(s_next + c, LISTED) == UNSEEN) s_list[atomicAdd(&s_listed, 1)] = c;
            if (c >= KM_BINS - 1) s_over[atomicAdd(&s_overs, 1)] = (uint32_t)i;
        }
        __syncthreads();
        for (int i0 = warp; i0 < s_listed; i0 += 4 * (KM_THREADS / 32)) {
            uint4 col[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + u * (KM_THREADS / 32);
                if (i < s_listed) col[u] = __ldcg(reinterpret_cast<const uint4 *>(a.cols + (size_t)s_list[i] * KM_MAX_CTAS) + lane);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + u * (KM_THREADS / 32);
                if (i >= s_listed) continue;
                const uint32_t w[4] = {col[u].x, col[u].y, col[u].z, col[u].w};
                uint32_t r = 0;
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (8 * lane + k < q) r += (w[k >> 1] >> (16 * (k & 1))) & 0xffffu;
                r = __reduce_add_sync(0xffffffffu, r);
                if (lane == 0) s_next[s_list[i]] = r + s_bins[s_list[i] + 1];
            }
        }
        __syncthreads();
        for (int i0 = 0; i0 < np; i0 += KM_THREADS) {        // (uniform)
            const int i = i0 + tid;
            const uint32_t p = (uint32_t)(p0 + i), c = i < np ? s_cnt[i] : 0u;
            const bool mine = ranked(c);
            const uint32_t same = __match_any_sync(0xffffffffu, mine ? c : 0u);
            const int first = __ffs(same) - 1;
            uint32_t r = 0;
            // (counted ahead: with the end of the part looked at in each turn 30 clk more a turn, 222 of them at v = 20.  That takes 93 us for
            // 5000 vectors, 156 where each pattern was ranked by itself; turns only for warps that have a pattern to rank 82, but 42.1 -> 43.2 and
            // 46.2 -> 47.8 for 300 000 and 1 048 576 vectors at v = 16)
            const int warps = min(KM_THREADS / 32, (np - i0 + 31) / 32);
            for (int w = 0; w < warps; ++w) {
                if (w == warp && mine && lane == first) { r = s_next[c]; s_next[c] = r + __popc(same); }
                __syncthreads();
            }
            r = __shfl_sync(0xffffffffu, r, first) + __popc(same & ((1u << lane) - 1u));
            if (mine && r < (uint32_t)Kc) { a.C[r] = p; a.seed[p] = r; }
        }
        // past the last bin: pairwise, a warp per pattern (4 194 304 vectors, where most patterns are past it: v = 10, 256 centroids
        // 45 us a call, v = 12, 777 47; 61 and 60 where a warp took those among its 32 neighbours one after another)
        for (int i = warp; i < s_overs; i += KM_THREADS / 32) {
            const uint32_t c = s_cnt[s_over[i]], p = (uint32_t)p0 + s_over[i];
            uint32_t before = 0;
            for (int j = lane; j < (int)s_bins[KM_BINS - 1]; j += 32) {
                const uint2 o = __ldcg(a.over + j);
                before += (o.x > c || (o.x == c && o.y < p)) ? 1u : 0u;
            }
            before = __reduce_add_sync(0xffffffffu, before);
            if (lane == 0 && before < (uint32_t)Kc) { a.C[before] = p; a.seed[p] = before; }
        }
    }
    if (!km_sync(a.st, target, &s_ok)) return;

    // ---- where many patterns share few centroids, their votes go to several copies: the atomics on one address follow one another
    const int copy = kc * a.words;
    int copies = 1;
    unsigned long long *votes = a.votes, *mine = votes;
    if (CROWDED && n_unique >= 2 * KM_CROWD * kc && P >= 2 * copy) {
        copies = min(min(KM_COPIES, P / copy), n_unique / (KM_CROWD * kc));
        votes = reinterpret_cast<unsigned long long *>(a.over);                  // (2^v words, last read before the barrier just passed)
        mine = votes + b % copies * copy;
        for (int i = gid; i < copy * copies; i += gthreads) votes[i] = 0ull;     // (a barrier before the first is cast)
    }

    const int low = min(v, KM_LOW), high = v - low;
    int it = 0, done = 0;
    while (it < a.max_iter && !done) {
        // ---- E-step, low bits: 512 neighbouring patterns per half CTA
        for (int u0 = 2 * b; u0 < (P >> low); u0 += 2 * G) {
            const int half = tid >> KM_LOW, u = u0 + half, e = tid & ((1 << KM_LOW) - 1);
            const bool live = u < (P >> low) && e < (1 << low);
            uint32_t k = KM_NONE;
            const int p = (u << low) + e;
            if (live) { k = __ldcg(a.seed + p); a.seed[p] = KM_NONE; }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1)
                if (o < (1 << low)) k = min(k, __shfl_xor_sync(0xffffffffu, k, o) + 0x10000u);
#pragma unroll
            for (int o = 32; o < (1 << KM_LOW); o <<= 1)
                if (o < (1 << low)) {                        // (uniform)
                    __syncthreads();
                    sm[tid] = k;
                    __syncthreads();
                    k = min(k, sm[tid ^ o] + 0x10000u);
                }
            if (live) a.key[p] = k;
        }
        if (!km_sync(a.st, target, &s_ok)) return;
        // ---- E-step, high bits, on columns of four patterns; labels and votes
        const int cols = min(4, 1 << low), E = cols << high, sh = __ffs(cols) - 1;
        int changed = 0;
        for (int u = b; u < (1 << low) / cols; u += G) {
            __syncthreads();
            for (int e = tid; e < E; e += KM_THREADS) sm[e] = __ldcg(a.key + ((e >> sh) << low) + u * cols + (e & (cols - 1)));
            for (int h = 0; h < high; ++h) {
                __syncthreads();
                const int o = cols << h;
                for (int q = tid; q < E / 2; q += KM_THREADS) {
                    const int e = (q & (o - 1)) | ((q & ~(o - 1)) << 1);
                    const uint32_t x = sm[e], y = sm[e + o];
                    sm[e] = min(x, y + 0x10000u);
                    sm[e + o] = min(y, x + 0x10000u);
                }
            }
            __syncthreads();
            for (int e = tid; e < E; e += KM_THREADS) {
                const int p = ((e >> sh) << low) + u * cols + (e & (cols - 1));
                const uint32_t c = __ldcg(a.cnt + p);
                if (!c) continue;
                const uint32_t z = sm[e] & 0xffffu;
                const uint32_t was = it == 0 ? KM_NONE : a.label[p];         // (this thread wrote it in the round before)
                if (was == z) continue;                      // its votes stand
                changed = 1;
                a.label[p] = (uint16_t)z;
                unsigned long long *vote = mine + (size_t)z * a.words, *old = it ? mine + (size_t)was * a.words : vote;
                const int bits = a.fields == 3 ? 21 : 32;
                uint32_t pat = ((uint32_t)p << 1) | 1u;      // count 0: the total; count 1 + t: element t is +1
                for (int w = 0; w < a.words; ++w) {
                    unsigned long long add = 0ull;
                    for (int f = 0; f < a.fields; ++f) {
                        if (pat & 1u) add |= (unsigned long long)c << (bits * f);
                        pat >>= 1;
                    }
                    if (!add) continue;
                    atomicAdd(vote + w, add);
                    if (it) atomicAdd(old + w, 0ull - add);  // (borrows between the counts of a word cancel in its total)
                }
            }
        }
        if (__syncthreads_or(changed) && tid == 0) a.st->changed[it & 1] = 1;
        if (gid == 0) a.st->changed[(it + 1) & 1] = 0;       // (last read before the barrier just passed)
        if (!km_sync(a.st, target, &s_ok)) return;
        done = *reinterpret_cast<volatile int *>(&a.st->changed[it & 1]) == 0;
        ++it;
        if (done) break;                                     // (nothing changed, so no votes were cast: no M-step)
        // ---- M-step, and the seeds of the next E-step
        const int bits = a.fields == 3 ? 21 : 32;
        const unsigned long long fmask = (1ull << bits) - 1ull;
        int moved = 0;
        auto elect = [&](int k, unsigned long long (&x)[KM_MAX_WORDS], bool write) {
            const uint32_t tot = (uint32_t)(x[0] & fmask);
            uint32_t pat = 0u;                                           // bit 0: the total, bit 1 + t: element t
            int bit = 0;
#pragma unroll
            for (int w = 0; w < KM_MAX_WORDS; ++w)
                if (w < a.words) {
                    for (int f = 0; f < a.fields; ++f, ++bit) {
                        const uint32_t o = (uint32_t)(x[w] & fmask);
                        x[w] >>= bits;
                        if (o >= tot - o) pat |= 1u << bit;              // at least as many +1 as -1: sign(0) = +1
                    }
                }
            if (!write) return;
            uint32_t c = (pat >> 1) & mask;
            const uint32_t before = __ldcg(a.C + k);
            if (!tot) c = before;                                        // (an empty cluster keeps its centroid)
            if (c != before) { a.C[k] = c; moved = 1; }
            if (it < a.max_iter) atomicMin(a.seed + c, (uint32_t)k);
        };
        unsigned long long x[KM_MAX_WORDS];
        if (!CROWDED || copies == 1) {
            for (int k = tid * G + b; k < kc; k += gthreads) {           // (spread over the SMs)
                const unsigned long long *vote = votes + (size_t)k * a.words;
#pragma unroll
                for (int w = 0; w < KM_MAX_WORDS; ++w)
                    if (w < a.words) x[w] = __ldcg(vote + w);
                elect(k, x, true);
            }
        } else {
            for (int k = warp * G + b; k < kc; k += gthreads / 32) {     // (a warp per centroid, a copy per lane)
                const unsigned long long *vote = votes + (size_t)k * a.words + lane * copy;
#pragma unroll
                for (int w = 0; w < KM_MAX_WORDS; ++w)
                    if (w < a.words) x[w] = lane < copies ? __ldcg(vote + w) : 0ull;
#pragma unroll
                for (int w = 0; w < KM_MAX_WORDS; ++w)
                    if (w < a.words)
                        for (int o = 16; o; o >>= 1) x[w] += __shfl_xor_sync(0xffffffffu, x[w], o);
                elect(k, x, lane == 0);
            }
        }
        if (it < a.max_iter) {
            // the same centroids give the same assignments, so a round behind an M-step that changed none is not run but only counted
            const int slot = (it - 1) & 1;
            if (__syncthreads_or(moved) && tid == 0) a.st->moved[slot] = 1;
            if (gid == 0) a.st->moved[slot ^ 1] = 0;         // (last read before the barrier of the E-step)
            if (!km_sync(a.st, target, &s_ok)) return;
            done = *reinterpret_cast<volatile int *>(&a.st->moved[slot]) == 0;
            it += done;
        }
    }

    // ---- assignments
    if (v <= 16) {
        __syncthreads();
        uint16_t *tab = reinterpret_cast<uint16_t *>(km_smem);
        if (P >= 8) {
            for (int i = tid; i < P / 8; i += KM_THREADS) reinterpret_cast<uint4 *>(tab)[i] = __ldcg(reinterpret_cast<const uint4 *>(a.label) + i);
        } else if (tid < P) {
            tab[tid] = __ldcg(a.label + tid);
        }
        __syncthreads();
        auto one = [&](size_t i, uint32_t w) { a.z[i] = tab[w & mask]; };
        if ((reinterpret_cast<uintptr_t>(a.z) & 7u) == 0)    // four assignments to a store
            km_stream(a.vecs, v0, v1, one, [&](size_t i, const uint4 &w) {
                *reinterpret_cast<uint2 *>(a.z + i) = make_uint2(tab[w.x & mask] | (uint32_t)tab[w.y & mask] << 16, tab[w.z & mask] | (uint32_t)tab[w.w & mask] << 16);
            });
        else
            km_stream(a.vecs, v0, v1, one);
    } else {
        km_stream(a.vecs, v0, v1, [&](size_t i, uint32_t w) { a.z[i] = __ldcg(a.label + (w & mask)); });
    }
    if (gid == 0) { a.info[0] = it; a.info[1] = kc; a.info[2] = n_unique; a.info[3] = done; }
}

int km_status_reset()
{
    const int zero = 0;
    cudaError_t e = cudaMemcpyToSymbol(g_km_status, &zero, sizeof(int));
    return e == cudaSuccess ? BTC_OK : cuda_fail(e);
}

int km_status_read(int *out)
{
    int v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_km_status, sizeof(int));
    if (e != cudaSuccess) return cuda_fail(e);
    *out = v;
    return BTC_OK;
}

static const void *const KM_KERNELS[2] = {reinterpret_cast<const void *>(km_kernel<false>), reinterpret_cast<const void *>(km_kernel<true>)};

// SMs that a cooperative launch on the stream can count on, a CTA each: the device's or, on a stream of a green context, that
// context's share of them.
static cudaError_t km_sms(cudaStream_t s, int *out)
{
    static std::atomic<int> sms_of[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int sms = dev < 64 ? sms_of[dev].load(std::memory_order_relaxed) : 0;
    if (!sms) {
        int per_sm = 0;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        for (const void *kern : KM_KERNELS) {
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)KM_SMEM);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, KM_THREADS, KM_SMEM);
            if (e == cudaSuccess && per_sm < 1) e = cudaErrorCooperativeLaunchTooLarge;
        }
        if (e != cudaSuccess) return e;
        if (sms > KM_MAX_CTAS) sms = KM_MAX_CTAS;
        if (dev < 64) sms_of[dev].store(sms, std::memory_order_relaxed);
    }
    typedef CUresult (*green_fn)(CUstream, CUgreenCtx *);
    typedef CUresult (*resource_fn)(CUgreenCtx, CUdevResource *, CUdevResourceType);
    struct Driver { green_fn green; resource_fn resource; };
    static const Driver driver = [] {                        // (a driver without green contexts has neither)
        auto find = [](const char *name) {
            void *p = nullptr;
            cudaDriverEntryPointQueryResult r;
            const bool ok = cudaGetDriverEntryPoint(name, &p, cudaEnableDefault, &r) == cudaSuccess && r == cudaDriverEntryPointSuccess;
            return ok ? p : nullptr;
        };
        Driver d;
        d.green = reinterpret_cast<green_fn>(find("cuStreamGetGreenCtx"));
        d.resource = reinterpret_cast<resource_fn>(find("cuGreenCtxGetDevResource"));
        return d;
    }();
    CUgreenCtx ctx = nullptr;
    CUdevResource r = {};
    if (driver.green && driver.resource && driver.green(s, &ctx) == CUDA_SUCCESS && ctx &&
        driver.resource(ctx, &r, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS && r.sm.smCount >= 1 && (int)r.sm.smCount < sms)
        sms = (int)r.sm.smCount;
    *out = sms;
    return cudaSuccess;
}

}  // namespace btc

using namespace btc;

extern "C" BTC_API size_t btc_codebook_kmeans_workspace_bytes(int v, int Kc)
{
    if (v < 1 || v > KM_VMAX || Kc < 1 || Kc > 65536) return 0;
    return km_workspace_bytes(v, Kc);
}

extern "C" BTC_API int btc_codebook_kmeans(const uint32_t *vecs, size_t n, int v, int Kc, int max_iter, uint32_t *C_words,
                                           uint16_t *z, int *info, void *workspace, size_t workspace_bytes, void *stream)
{
    if (!vecs || !C_words || !z || !info || !workspace) return BTC_ERR_NULL;
    if (Kc < 1 || Kc > 65536 || n < 1 || n > 0x7fffffffull || max_iter < 1 || max_iter > 4096 || v < 1 || v > 32) return BTC_ERR_SHAPE;
    if (v > KM_VMAX) return BTC_ERR_UNSUPPORTED;             // the pattern-space steps keep 2^v entries
    if (workspace_bytes < km_workspace_bytes(v, Kc)) return BTC_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(workspace) % 256) return BTC_ERR_ALIGN;
    cudaStream_t s = (cudaStream_t)stream;
    KmArgs a;
    km_carve(a, workspace, v, Kc, n);
    a.vecs = vecs; a.n = n; a.v = v; a.Kc = Kc; a.max_iter = max_iter; a.C = C_words; a.z = z; a.info = info;
    int sms = 0;
    cudaError_t e = km_sms(s, &sms);
    if (e != cudaSuccess) return cuda_fail(e);
    // a CTA per SM, fewer where there is little to do (a barrier costs more the more of them there are)
    const size_t want = (n + 1023) / 1024 > (size_t)((1 << v) + 511) / 512 ? (n + 1023) / 1024 : (size_t)((1 << v) + 511) / 512;
    int grid = want < (size_t)sms ? (int)want : sms;
    const int parts = ((1 << v) + KM_PART - 1) / KM_PART;
    e = cudaMemsetAsync(a.st, 0, km_align(sizeof(KmState)) + ((size_t)4 << v), s);
    if (e != cudaSuccess) return cuda_fail(e);
    // (there are at most as many patterns as vectors; the form without copies saves 0.3 to 0.9 us where there are too few for them)
    const void *kern = KM_KERNELS[(n < (size_t)1 << v ? n : (size_t)1 << v) >= (size_t)2 * KM_CROWD * Kc];
    void *params[] = {&a};
    for (;;) {
        a.parts = grid > parts ? grid : parts;
        e = cudaLaunchCooperativeKernel(kern, dim3((unsigned)grid), dim3(KM_THREADS), params, KM_SMEM, s);
        if (e != cudaErrorCooperativeLaunchTooLarge || grid == 1) break;
        (void)cudaGetLastError();                            // (some other share of the device: as many as are let in)
        grid -= (grid + 7) / 8;
    }
    return e == cudaSuccess ? BTC_OK : cuda_fail(e);
}
