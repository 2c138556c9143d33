// sort.cu -- stable LSD radix sort of (key, value) u32 pairs in S independent segments, on many
// CTAs: per 8-bit pass, (1) every 2,048-element tile counts its digits, (2) the (digit, tile)
// counts of each segment are scanned, a long segment by several CTAs, (3) every tile scatters its
// elements in a stable order (warp match on the digit, then per-digit prefix over the tile's warps).
// Segments of at most 8,192 pairs are sorted by one CTA each, in one launch.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "internal.cuh"

namespace aiwcrf {

constexpr int kSortThreads = 256;
constexpr int kSortSub = 8;
constexpr int kSortTile = kSortThreads * kSortSub;

__global__ void __launch_bounds__(kSortThreads) sort_hist_kernel(const uint32_t *__restrict__ keys, int64_t n,
                                                                 int64_t stride, int shift, int nb,
                                                                 uint32_t *__restrict__ hist)
{
    __shared__ uint32_t h[256];
    const int b = blockIdx.x, seg = blockIdx.y, tid = threadIdx.x;
    h[tid] = 0u;
    __syncthreads();
    const uint32_t *k = keys + (size_t)seg * (size_t)stride;
    const int64_t end = min(n, (int64_t)(b + 1) * kSortTile);
    for (int64_t i = (int64_t)b * kSortTile + tid; i < end; i += kSortThreads) atomicAdd(&h[(k[i] >> shift) & 255u], 1u);
    __syncthreads();
    hist[((size_t)seg * 256 + tid) * (size_t)nb + b] = h[tid];
}

// exclusive scan of one segment's 256 * nb counts, digit-major, into scan: CTA (part, segment)
// scans the counts [part * per4, ...) (16-byte words). It first sums every count before its own
// part, which lets the parts run side by side without waiting for one another (the counts are
// read-only, a few hundred KB in L2); then every thread sums a contiguous run of its part, one
// block scan of the run sums, and every thread writes its run from its own prefix. (A segment
// starts 1,024 * nb bytes after the 16-byte aligned base, and 256 * nb counts are whole words.)
// Sorting 1,000,000 keys, one CTA per segment took 28 us a pass, the parts take 10 (cold caches).
constexpr int kScanPartThreads = 512;
__global__ void __launch_bounds__(kScanPartThreads) sort_scan_kernel(const uint32_t *__restrict__ hist,
                                                                     uint32_t *__restrict__ scan, int nb, int64_t per4)
{
    __shared__ uint32_t warp_tmp[32];
    __shared__ uint32_t before;
    const size_t seg = (size_t)blockIdx.y * 256 * (size_t)nb;
    const uint4 *h4 = reinterpret_cast<const uint4 *>(hist + seg);
    uint4 *o4 = reinterpret_cast<uint4 *>(scan + seg);
    const int64_t total4 = 64 * (int64_t)nb;
    const int64_t p0 = (int64_t)blockIdx.x * per4, p1 = min(total4, p0 + per4);
    uint32_t pre = 0;
#pragma unroll 4
    for (int64_t i = threadIdx.x; i < p0; i += kScanPartThreads) {
        const uint4 v = __ldg(&h4[i]);
        pre += v.x + v.y + v.z + v.w;
    }
    const int64_t per = (p1 - p0 + kScanPartThreads - 1) / kScanPartThreads;
    const int64_t lo = min(p1, p0 + (int64_t)threadIdx.x * per), hi = min(p1, lo + per);
    uint32_t sum = 0;
#pragma unroll 4
    for (int64_t i = lo; i < hi; ++i) {
        const uint4 v = __ldg(&h4[i]);
        sum += v.x + v.y + v.z + v.w;
    }
    uint32_t tot;
    if (blockIdx.x) {
        block_incl_scan(pre, warp_tmp, tot);
        if (threadIdx.x == 0) before = tot;
    } else if (threadIdx.x == 0) {
        before = 0u;
    }
    uint32_t run = block_incl_scan(sum, warp_tmp, tot) - sum;     // its barriers publish `before`
    run += before;
#pragma unroll 4
    for (int64_t i = lo; i < hi; ++i) {
        const uint4 v = __ldg(&h4[i]);
        uint4 o;
        o.x = run; run += v.x;
        o.y = run; run += v.y;
        o.z = run; run += v.z;
        o.w = run; run += v.w;
        o4[i] = o;
    }
}

// Stable scatter of one tile. A warp owns kSortSub consecutive runs of 32 elements, loaded at once.
// It ranks each run's elements among the warp's earlier ones of the same digit (match, and a count
// per digit that is the warp's own); then one pass over the tile's warps turns the counts into
// positions within the tile. The tile is put in digit order in shared memory first, so that its
// writes go out as runs of consecutive addresses (8 elements of a digit on average) instead of one
// 32-byte sector per 4-byte word. Latency bounds it (a tile is a chain of kSortSub ranked runs and
// a few barriers), so tiles are small enough for six CTAs per SM.
// Measured, a fit's rank phase (111,000 rows x 32 columns) / 1,000,000 queries with their walk:
// barriers after every 256 elements of a 4,096-element tile, scattered writes 282 us / 4.33 ms;
// this, tiles of 2,048 261 us / 4.33 ms; of 4,096 274 / 4.31; of 1,024 288 / 4.36; eight ballots for
// the match 287 / 4.33.
__global__ void __launch_bounds__(kSortThreads) sort_scatter_kernel(const uint32_t *__restrict__ kin,
                                                                    const uint32_t *__restrict__ vin,
                                                                    uint32_t *__restrict__ kout,
                                                                    uint32_t *__restrict__ vout, int64_t n,
                                                                    int64_t stride, int shift, int nb,
                                                                    const uint32_t *__restrict__ scan)
{
    constexpr int kWarps = kSortThreads / 32;
    __shared__ uint32_t wcnt[kWarps][256];
    __shared__ uint32_t to[256];            // global position of a digit's element minus its tile position
    __shared__ uint32_t warp_tmp[32];
    __shared__ uint32_t sk[kSortTile], sv[kSortTile];
    const int b = blockIdx.x, seg = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const size_t off = (size_t)seg * (size_t)stride;
    const int64_t t0 = (int64_t)b * kSortTile;
    const int count = (int)min((int64_t)kSortTile, n - t0);
    const int i0 = warp * (32 * kSortSub) + lane;
    uint32_t k[kSortSub], v[kSortSub], rank[kSortSub];
#pragma unroll
    for (int u = 0; u < kSortSub; ++u) {
        const bool valid = i0 + 32 * u < count;
        k[u] = valid ? kin[off + t0 + i0 + 32 * u] : 0u;
        v[u] = valid ? vin[off + t0 + i0 + 32 * u] : 0u;
    }
    const uint32_t base = scan[((size_t)seg * 256 + tid) * (size_t)nb + b];
#pragma unroll
    for (int w = 0; w < 8; ++w) wcnt[warp][32 * w + lane] = 0u;
    __syncwarp();
#pragma unroll
    for (int u = 0; u < kSortSub; ++u) {
        const bool valid = i0 + 32 * u < count;
        const uint32_t d = (k[u] >> shift) & 255u;
        const uint32_t peers = __match_any_sync(kFull, valid ? d : (256u + lane));
        const uint32_t before = __popc(peers & lanemask_lt());
        const uint32_t old = valid ? wcnt[warp][d] : 0u;
        rank[u] = old + before;
        __syncwarp();
        if (valid && before == 0) wcnt[warp][d] = old + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    uint32_t tot = 0, all;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) tot += wcnt[w][tid];
    uint32_t run = block_incl_scan(tot, warp_tmp, all) - tot;     // the digit's start within the tile
    to[tid] = base - run;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const uint32_t c = wcnt[w][tid];
        wcnt[w][tid] = run;
        run += c;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kSortSub; ++u) {
        if (i0 + 32 * u < count) {
            const uint32_t pos = wcnt[warp][(k[u] >> shift) & 255u] + rank[u];
            sk[pos] = k[u];
            sv[pos] = v[u];
        }
    }
    __syncthreads();
#pragma unroll 4
    for (int i = tid; i < count; i += kSortThreads) {
        const uint32_t key = sk[i];
        const uint32_t pos = to[(key >> shift) & 255u] + (uint32_t)i;
        kout[off + pos] = key;
        vout[off + pos] = sv[i];
    }
}

// A whole sort of a segment that fits one CTA's shared memory: the scatter's ranking with the segment as
// its one tile, a pass after the other in shared memory. It is a chain of barriers and matches, where the
// passes above are three launches each whatever the size. Measured, the rank phase of a fit of 32 columns,
// passes / this: 2,220 rows 138 / 98 us, 4,440 145 / 115, 6,660 146 / 110; 8,192 keys are the most whose
// tile (with 16 KB of counts) leaves a thread its eight pairs in registers.
constexpr int kSmallSortThreads = 1024;
constexpr int64_t kSmallSortMax = 8192;

template <int SUB>
__global__ void __launch_bounds__(kSmallSortThreads) sort_small_kernel(uint32_t *__restrict__ keys, uint32_t *__restrict__ vals,
                                                                       int n, int64_t stride, int passes)
{
    constexpr int kWarps = kSmallSortThreads / 32;
    extern __shared__ uint32_t sort_sm[];
    uint32_t *sk = sort_sm, *sv = sk + kSmallSortThreads * SUB;
    uint16_t(*wcnt)[256] = reinterpret_cast<uint16_t(*)[256]>(sv + kSmallSortThreads * SUB);
    __shared__ uint32_t warp_tmp[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t *gk = keys + (size_t)blockIdx.x * (size_t)stride, *gv = vals + (size_t)blockIdx.x * (size_t)stride;
    const int i0 = warp * (32 * SUB) + lane;
    uint32_t k[SUB], v[SUB], rank[SUB];
#pragma unroll
    for (int u = 0; u < SUB; ++u) {
        const bool valid = i0 + 32 * u < n;
        k[u] = valid ? gk[i0 + 32 * u] : 0u;
        v[u] = valid ? gv[i0 + 32 * u] : 0u;
    }
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = 8 * pass;
#pragma unroll
        for (int w = 0; w < 8; ++w) wcnt[warp][32 * w + lane] = 0u;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < SUB; ++u) {
            const bool valid = i0 + 32 * u < n;
            const uint32_t d = (k[u] >> shift) & 255u;
            const uint32_t peers = __match_any_sync(kFull, valid ? d : (256u + lane));
            const uint32_t before = __popc(peers & lanemask_lt());
            const uint32_t old = valid ? wcnt[warp][d] : 0u;
            rank[u] = old + before;
            __syncwarp();
            if (valid && before == 0) wcnt[warp][d] = (uint16_t)(old + __popc(peers));
            __syncwarp();
        }
        __syncthreads();
        uint32_t tot = 0, all;
        if (tid < 256) {
#pragma unroll
            for (int w = 0; w < kWarps; ++w) tot += wcnt[w][tid];
        }
        uint32_t run = block_incl_scan(tot, warp_tmp, all) - tot;
        if (tid < 256) {
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const uint32_t c = wcnt[w][tid];
                wcnt[w][tid] = (uint16_t)run;
                run += c;
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < SUB; ++u) {
            if (i0 + 32 * u < n) {
                const uint32_t pos = wcnt[warp][(k[u] >> shift) & 255u] + rank[u];
                sk[pos] = k[u];
                sv[pos] = v[u];
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < SUB; ++u) {
            if (i0 + 32 * u < n) { k[u] = sk[i0 + 32 * u]; v[u] = sv[i0 + 32 * u]; }
        }
    }
#pragma unroll
    for (int u = 0; u < SUB; ++u) {
        if (i0 + 32 * u < n) { gk[i0 + 32 * u] = k[u]; gv[i0 + 32 * u] = v[u]; }
    }
}

template <int SUB>
int sort_small(uint32_t *keys, uint32_t *vals, int64_t n, int S, int64_t stride, int passes, cudaStream_t s)
{
    const int smem = kSmallSortThreads * SUB * 8 + (kSmallSortThreads / 32) * 512;
    cudaError_t e = cudaFuncSetAttribute(sort_small_kernel<SUB>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) {
        sort_small_kernel<SUB><<<(unsigned)S, kSmallSortThreads, (size_t)smem, s>>>(keys, vals, (int)n, stride, passes);
        count_launches(1);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? AIWCRF_OK : cuda_fail(e, "radix sort launch");
}

size_t radix_sort_hist_words(int64_t n, int S)
{
    const int64_t nb = (n + kSortTile - 1) / kSortTile;
    return 2 * (size_t)S * 256 * (size_t)(nb > 0 ? nb : 1) + 1;      // the counts and their scan
}

int radix_sort_segments(uint32_t *keys_a, uint32_t *vals_a, uint32_t *keys_b, uint32_t *vals_b, int64_t n,
                        int S, int64_t stride, uint32_t *hist, cudaStream_t s, int bits, bool *in_b)
{
    if (in_b) *in_b = false;
    if (n <= 0 || S <= 0) return AIWCRF_OK;
    if (n <= kSmallSortMax) {
        const int passes = (bits + 7) / 8;
        return n <= 2 * kSmallSortThreads   ? sort_small<2>(keys_a, vals_a, n, S, stride, passes, s)
               : n <= 4 * kSmallSortThreads ? sort_small<4>(keys_a, vals_a, n, S, stride, passes, s)
                                            : sort_small<8>(keys_a, vals_a, n, S, stride, passes, s);
    }
    const int nb = (int)((n + kSortTile - 1) / kSortTile);
    const dim3 grid((unsigned)nb, (unsigned)S);
    uint32_t *scan = hist + (size_t)S * 256 * (size_t)nb;
    // parts of the count scan: a few thousand counts each, so that one long segment is spread over
    // SMs; short segments (and many of them) are one part each
    const int parts = (int)std::max<int64_t>(1, std::min<int64_t>(32, 64 * (int64_t)nb / 512));
    const int64_t per4 = (64 * (int64_t)nb + parts - 1) / parts;
    uint32_t *ki = keys_a, *vi = vals_a, *ko = keys_b, *vo = vals_b;
    const int passes = (bits + 7) / 8;
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = 8 * pass;
        sort_hist_kernel<<<grid, kSortThreads, 0, s>>>(ki, n, stride, shift, nb, hist);
        sort_scan_kernel<<<dim3((unsigned)parts, (unsigned)S), kScanPartThreads, 0, s>>>(hist, scan, nb, per4);
        sort_scatter_kernel<<<grid, kSortThreads, 0, s>>>(ki, vi, ko, vo, n, stride, shift, nb, scan);
        count_launches(3);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "radix sort launch");
        uint32_t *t = ki; ki = ko; ko = t;
        t = vi; vi = vo; vo = t;
    }
    if (in_b) *in_b = (passes & 1) != 0;
    return AIWCRF_OK;
}

}  // namespace aiwcrf
