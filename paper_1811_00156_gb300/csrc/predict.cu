// predict.cu -- forest queries (Sec. I, Sec. V) and device selection (Sec. VI).
//
// code_queries_kernel turns every query feature into its rank code c(x) = #{training values of
// the feature < x}; the forest keeps a copy of its nodes whose thresholds are the ranks of the
// training values they are, and x <= threshold  <=>  c(x) <= rank, so the walk is exact.
// predict_kernel: one CTA owns 256 * QPT queries whose codes (one byte per feature when every
// column has at most 255 values) it stages once in shared memory. It then walks a part of the trees for
// all its queries, QPT independent walks per thread: every tree, or, where that leaves the chip idle or
// its last wave nearly empty, one of several shares (tree_parts). Trees stream through two shared-memory
// slots with 1-D bulk asynchronous copies (cp.async.bulk, completion counted on an mbarrier):
// while the CTA walks tree t from one slot, tree t + 1 is landing in the other. A tree larger
// than a slot is walked straight from global memory. Per-query sums are exact int64 (plus an
// exact 128-bit sum of squares for the variance), so the result does not depend on any order.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <vector>

#include "internal.cuh"

namespace aiwcrf {

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

constexpr int kPredThreads = 256;
constexpr uint32_t kWaitLimit = 1u << 24;     // try_wait polls before giving up

// stage tree t into slot (or just complete the phase if it does not fit)
__device__ __forceinline__ void issue_tree(const uint64_t *nodes, const int64_t *tree_off, int t,
                                           int tree_cap, uint64_t *slot, uint64_t *bar)
{
    const int64_t a = tree_off[t], nn = tree_off[t + 1] - a;
    if (nn <= tree_cap) {
        const uint32_t bytes = (uint32_t)nn * 8u;
        fence_proxy_async();
        mbar_arrive_expect_tx(bar, bytes);
        bulk_g2s(slot, nodes + a, bytes, bar);
    } else {
        mbar_arrive(bar);
    }
}

// The tile's code rows (words 32-bit words, 16-byte aligned at both ends) into shared memory: whole
// 16-byte units by one bulk copy that completes on bar, the rest by plain loads.
__device__ __forceinline__ void stage_rows(uint32_t *dst, const uint32_t *src, int64_t words, uint64_t *bar)
{
    const int64_t whole = words & ~(int64_t)3;
    if (threadIdx.x == 0) {
        mbar_arrive_expect_tx(bar, (uint32_t)whole * 4u);
        if (whole) bulk_g2s(dst, src, (uint32_t)whole * 4u, bar);
    }
    if (threadIdx.x < words - whole) dst[whole + threadIdx.x] = src[whole + threadIdx.x];
}

// Every thread of the CTA: wait for stage_rows' copy on bar[2]. On a wait that gives up, flag it,
// give the first trees' copies (bar[0], bar[1]) a bounded chance to land, and return false.
__device__ __forceinline__ bool rows_landed(uint64_t *bar, int T, uint32_t *err)
{
    bool ok = false;
    for (uint32_t it = 0; it < kWaitLimit && !ok; ++it) ok = mbar_try_wait(&bar[2], 0);
    if (!__syncthreads_or(!ok)) return true;
    if (threadIdx.x == 0) atomicOr(err, kErrTimeout);
    for (int b = 0; b < min(T, 2); ++b)
        for (uint32_t it = 0; it < kWaitLimit; ++it)
            if (mbar_try_wait(&bar[b], 0)) break;
    return false;
}

__device__ __forceinline__ int64_t leaf_value(uint64_t nd)
{
    return ((int64_t)(nd << 1)) >> 1;
}

// Rank codes of queries: c(x) = #{table values < x}; NaN goes right of every threshold
// (c = table size). A CTA codes kCodeQueries queries into rows in shared memory, one lane per
// query and kCodeWarps warps side by side over the features, then writes its rows, which are
// contiguous in global memory, with 16-byte stores, so that every byte of the code matrix is
// written once, whole sectors at a time. A row is row_words 4-byte words; its padding is zero.
// What bounds it is the searches' chain of dependent table loads (L1 hits: a warp's lanes search
// one table). A thread searches kCodeGroup features side by side, so 32 features are one chain of
// `steps` loads per thread; one thread per query walked eight such chains one after the other.
// 2,220 queries 58 -> 11 us, 111,000 47 -> 23, 1,000,000 196 -> 177 (148 values per column; cold).
constexpr int kCodeQueries = 32;
constexpr int kCodeWarps = 8;
constexpr int kCodeThreads = 32 * kCodeWarps;
constexpr int kCodeGroup = 4;

// this lane's codes c[f] of the features f < nf that are its warp's, x(f) their values
template <typename CT, typename Value>
__device__ __forceinline__ void code_columns(int nf, const float *__restrict__ fvals, int64_t fstride,
                                             const uint32_t *__restrict__ fcard, int steps, int warp, CT *c, const Value &value)
{
    for (int f0 = warp; f0 < nf; f0 += kCodeWarps * kCodeGroup) {
        float x[kCodeGroup];
        uint32_t n[kCodeGroup], pos[kCodeGroup];
        const float *tab[kCodeGroup];
#pragma unroll
        for (int u = 0; u < kCodeGroup; ++u) {
            const int f = f0 + u * kCodeWarps;
            x[u] = f < nf ? value(f) : 0.0f;
            n[u] = f < nf ? __ldg(&fcard[f]) : 0u;
            tab[u] = fvals + (size_t)(f < nf ? f : 0) * (size_t)fstride;
            pos[u] = 0u;
        }
        if constexpr (sizeof(CT) == 1) {
            // lower bound by halving powers of two: pos + bit values are below x if the last of
            // them is (tables are sorted; a position past the table, or a NaN, never is)
            for (uint32_t bit = 1u << (steps - 1); bit; bit >>= 1) {
#pragma unroll
                for (int u = 0; u < kCodeGroup; ++u) {
                    const uint32_t at = pos[u] + bit;
                    if (at <= n[u] && __ldg(&tab[u][at - 1]) < x[u]) pos[u] = at;
                }
            }
        } else {
            // larger tables (over 255 values): halves of what is left, whose probes spread over L1's sets;
            // those at powers of two meet in a few. 700,000 queries x 32 columns of 6,660 values 434 ->
            // 325 us, 400,000 of 111,000 values 810 -> 355; small tables are faster the other way.
            uint32_t len[kCodeGroup];
#pragma unroll
            for (int u = 0; u < kCodeGroup; ++u) len[u] = n[u];
            for (int it = 0; it < steps; ++it) {
#pragma unroll
                for (int u = 0; u < kCodeGroup; ++u) {
                    const uint32_t half = len[u] >> 1;
                    const bool below = len[u] != 0u && __ldg(&tab[u][pos[u] + half]) < x[u];
                    pos[u] += below ? half + 1u : 0u;
                    len[u] = below ? len[u] - half - 1u : half;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kCodeGroup; ++u) {
            const int f = f0 + u * kCodeWarps;
            if (f < nf) c[f] = (CT)(x[u] != x[u] ? n[u] : pos[u]);
        }
    }
}

template <typename CT>
__global__ void __launch_bounds__(kCodeThreads) code_queries_kernel(const float *__restrict__ Xq, int64_t Q, int F,
                                                                   const float *__restrict__ fvals, int64_t fstride,
                                                                   const uint32_t *__restrict__ fcard,
                                                                   CT *__restrict__ codes, int row_words, int steps,
                                                                   unsigned long long *zero, int64_t nzero)
{
    extern __shared__ __align__(16) uint32_t code_rows[];         // kCodeQueries * row_words words
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t q0 = (int64_t)blockIdx.x * kCodeQueries, q = q0 + lane;
    for (int64_t i = (int64_t)blockIdx.x * kCodeThreads + tid; i < nzero; i += (int64_t)gridDim.x * kCodeThreads)
        zero[i] = 0ull;                                            // the walk's sums and tickets
    CT *c = reinterpret_cast<CT *>(code_rows + (size_t)lane * (size_t)row_words);   // odd row_words: distinct banks
    for (int f = F + warp; f < row_words * 4 / (int)sizeof(CT); f += kCodeWarps) c[f] = (CT)0;
    // features are read once: streaming loads (evict first in L1 and L2) leave the codes written here
    // resident in L2 for the key and walk kernels that read them
    if (q < Q)
        code_columns<CT>(F, fvals, fstride, fcard, steps, warp, c,
                         [&](int f) { return __ldcs(&Xq[(size_t)f * (size_t)Q + q]); });
    __syncthreads();
    const int64_t n = min((int64_t)kCodeQueries, Q - q0);
    const int words = (int)n * row_words;
    uint32_t *dst = reinterpret_cast<uint32_t *>(codes) + (size_t)q0 * (size_t)row_words;
    const int vec = (reinterpret_cast<uintptr_t>(dst) & 15u) == 0 ? words >> 2 : 0;
    for (int i = tid; i < vec; i += kCodeThreads)
        reinterpret_cast<uint4 *>(dst)[i] = reinterpret_cast<const uint4 *>(code_rows)[i];
    for (int i = 4 * vec + tid; i < words; i += kCodeThreads) dst[i] = code_rows[i];
}

// Rank codes of a device selection's queries (k, j) = kernel k's features, device ids[j], one size
// class: a CTA codes the features of kCodeQueries kernels as above, the devices and the size once,
// and writes every kernel's row for every device. (Expanding the queries first read and searched
// every feature once per device.)
template <typename CT>
__device__ __forceinline__ CT code_of(float x, const float *__restrict__ tab, uint32_t n, int steps)
{
    uint32_t pos = 0u;
    for (uint32_t bit = 1u << (steps - 1); bit; bit >>= 1) {
        const uint32_t at = pos + bit;
        if (at <= n && __ldg(&tab[at - 1]) < x) pos = at;
    }
    return (CT)(x != x ? n : pos);
}

template <typename CT>
__global__ void __launch_bounds__(kCodeThreads) code_selection_kernel(
    const float *__restrict__ kfeat, int32_t K, int32_t size_class, DeviceIds ids, int32_t D, int F,
    const float *__restrict__ fvals, int64_t fstride, const uint32_t *__restrict__ fcard, CT *__restrict__ codes,
    int row_words, int steps, unsigned long long *zero, int64_t nzero)
{
    extern __shared__ __align__(16) uint32_t code_rows[];         // kCodeQueries kernels' rows
    __shared__ uint32_t dcode[kSelectMaxDevices];
    __shared__ uint32_t scode;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t k0 = (int64_t)blockIdx.x * kCodeQueries, k = k0 + lane;
    for (int64_t i = (int64_t)blockIdx.x * kCodeThreads + tid; i < nzero; i += (int64_t)gridDim.x * kCodeThreads) zero[i] = 0ull;
    CT *c = reinterpret_cast<CT *>(code_rows + (size_t)lane * (size_t)row_words);
    // the device's and the size's places and the padding: zero here, put in as the rows are written
    for (int f = F - 2 + warp; f < row_words * 4 / (int)sizeof(CT); f += kCodeWarps) c[f] = (CT)0;
    code_columns<CT>(F - 2, fvals, fstride, fcard, steps, warp, c,
                     [&](int f) { return k < K ? __ldg(&kfeat[(size_t)f * (size_t)K + k]) : 0.0f; });
    if (tid < D) dcode[tid] = code_of<CT>((float)ids[tid], fvals + (size_t)(F - 2) * (size_t)fstride, __ldg(&fcard[F - 2]), steps);
    if (tid == kCodeThreads - 1)
        scode = code_of<CT>((float)size_class, fvals + (size_t)(F - 1) * (size_t)fstride, __ldg(&fcard[F - 1]), steps);
    __syncthreads();
    constexpr int kPer = 4 / (int)sizeof(CT);
    const int dw = (F - 2) / kPer, ds = (F - 2) % kPer * 8 * (int)sizeof(CT);
    const int sw = (F - 1) / kPer, ss = (F - 1) % kPer * 8 * (int)sizeof(CT);
    const int rows = (int)min((int64_t)kCodeQueries, K - k0) * D, words = rows * row_words;
    uint32_t *dst = reinterpret_cast<uint32_t *>(codes) + (size_t)k0 * (size_t)D * (size_t)row_words;
    for (int i = tid; i < words; i += kCodeThreads) {
        const int r = i / row_words, w = i - r * row_words, kk = r / D, j = r - kk * D;
        uint32_t v = code_rows[kk * row_words + w];
        if (w == dw) v |= dcode[j] << ds;
        if (w == sw) v |= scode << ss;
        dst[i] = v;
    }
}

// bytes of one feature's code for a forest: one when every value table has at most 255 values
__host__ __forceinline__ int code_bytes_of(const aiwcrf_forest *f)
{
    return f->max_card <= 255u ? 1 : (f->max_card <= 65535u ? 2 : 4);
}

// Words of one query's code row: F codes rounded up to whole words, made odd so that rows
// staged side by side in shared memory start on distinct banks.
__host__ __forceinline__ int code_row_words(int F, int code_bytes)
{
    int w = (F * code_bytes + 3) / 4;
    if ((w & 1) == 0) ++w;
    return w;
}

// codes of Q queries (row_words words per query) on the stream; zero: nzero 8-byte words to clear
template <typename CT>
cudaError_t launch_code_queries(const aiwcrf_forest *f, const float *dXq, int64_t Q, CT *d_codes, int row_words,
                                cudaStream_t s, unsigned long long *zero = nullptr, int64_t nzero = 0)
{
    if (Q == 0) return cudaSuccess;
    const size_t smem = (size_t)kCodeQueries * (size_t)row_words * 4;        // <= 16.5 KB (F <= 128)
    const int steps = 32 - __builtin_clz(f->max_card | 1u);               // bit width of the largest table
    code_queries_kernel<CT><<<(unsigned)((Q + kCodeQueries - 1) / kCodeQueries), kCodeThreads, smem, s>>>(
        dXq, Q, f->F, f->d_fvals, f->fstride, f->d_fcard, d_codes, row_words, steps, zero, nzero);
    count_launches(1);
    return cudaGetLastError();
}

// One step of QPT independent walks through one tree (coded thresholds).
template <typename CT, int QPT, typename NodePtr>
__device__ __forceinline__ void walk_tree(NodePtr tn, const CT *const (&xr)[QPT], int64_t (&acc)[QPT],
                                          u128_t (&sq)[QPT], bool var, uint32_t nn)
{
    uint32_t j[QPT];
#pragma unroll
    for (int i = 0; i < QPT; ++i) j[i] = 0u;
    for (;;) {
        bool more = false;
#pragma unroll
        for (int i = 0; i < QPT; ++i) {
            const uint64_t nd = tn[j[i]];
            const uint32_t hi = (uint32_t)(nd >> 32);
            const bool leaf = (int32_t)hi < 0;
            const uint32_t f = leaf ? 0u : ((hi >> 24) & 0x7Fu);
            const uint32_t c = (uint32_t)xr[i][f];
            const uint32_t nxt = (hi & 0xFFFFFFu) + (c > ((uint32_t)nd & 0xFFFFFFu) ? 1u : 0u);
            j[i] = leaf ? j[i] : AIWCRF_IDX(nxt, nn, kBoundWalk);
            more |= !leaf;
        }
        if (!more) break;
    }
#pragma unroll
    for (int i = 0; i < QPT; ++i) {
        const int64_t v = leaf_value(tn[j[i]]);
        acc[i] += v;
        if (var) sq[i] += (u128_t)((i128_t)v * (i128_t)v);
    }
}

// Split of the trees over CTAs. CTA (tile, part) walks trees [part * per, ...) for its tile of
// queries; with more than one part, each CTA adds its queries' partial sums (and sums of squares)
// into sum / sq, and the last CTA of a tile to arrive (ticket) writes the results: exact integers,
// so the order does not matter. sum, sq and ticket are zero on entry (the coding kernel clears
// them). A square sum keeps all its 128 bits, as an unsplit walk's does: the low words are added first,
// and whoever's addition wraps carries into the high word.
// Adding costs the last CTA one read per query; summing the parts' separate sums there instead
// took 35 us of a 2,220-query call with 128 parts.
struct TreeParts {
    int per;                     // trees of one part
    unsigned long long *sum;     // one per query position (whole tiles)
    unsigned long long *sq;      // two per query position, for the variance
    uint32_t *ticket;            // one per tile
};

__device__ __forceinline__ void write_query(int64_t q, int64_t acc, u128_t sq, int64_t total_trees, int64_t *out_sum,
                                            int64_t *out_pred, uint64_t *out_var)
{
    if (out_sum) out_sum[q] = acc;
    if (out_pred) {
        if (total_trees <= 0xFFFFFFFFll) {
            out_pred[q] = round_mean(acc, (uint32_t)total_trees);
        } else {
            const i128_t num = (i128_t)2 * acc + total_trees, den = (i128_t)2 * total_trees;
            i128_t d = num / den;
            if (num % den != 0 && num < 0) d -= 1;
            out_pred[q] = (int64_t)d;
        }
    }
    if (out_var) {
        const u128_t V = (u128_t)total_trees * sq - (u128_t)((i128_t)acc * (i128_t)acc);
        out_var[2 * q] = (uint64_t)V;
        out_var[2 * q + 1] = (uint64_t)(V >> 64);
    }
}

// The end of both walk kernels: the thread's QPT queries' sums to the outputs, or to the parts
// and, from the tile's last CTA, to the outputs. Query at tile position i is perm[i] with PERM.
template <int QPT, bool VAR, bool PERM>
__device__ __forceinline__ void finish_tile(const TreeParts &tp, int64_t (&acc)[QPT], u128_t (&sq)[QPT], int64_t q0,
                                            int64_t Q, int64_t total_trees, int64_t *out_sum, int64_t *out_pred,
                                            uint64_t *out_var, const uint32_t *__restrict__ perm)
{
    const int tid = threadIdx.x;
    if (gridDim.y > 1) {
        __shared__ uint32_t last;
#pragma unroll
        for (int i = 0; i < QPT; ++i) {
            const size_t k = (size_t)q0 + (size_t)(tid + i * kPredThreads);
            atomicAdd(&tp.sum[k], (unsigned long long)acc[i]);
            if (VAR) {
                const unsigned long long lo = (unsigned long long)sq[i], was = atomicAdd(&tp.sq[2 * k], lo);
                atomicAdd(&tp.sq[2 * k + 1], (unsigned long long)(sq[i] >> 64) + (was + lo < lo ? 1ull : 0ull));
            }
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) last = atomicAdd(&tp.ticket[blockIdx.x], 1u) == gridDim.y - 1 ? 1u : 0u;
        __syncthreads();
        if (!last) return;
        __threadfence();
#pragma unroll
        for (int i = 0; i < QPT; ++i) {
            const size_t k = (size_t)q0 + (size_t)(tid + i * kPredThreads);
            acc[i] = (int64_t)__ldcg(&tp.sum[k]);
            if (VAR) sq[i] = (u128_t)__ldcg(&tp.sq[2 * k]) | ((u128_t)__ldcg(&tp.sq[2 * k + 1]) << 64);
        }
    }
#pragma unroll
    for (int i = 0; i < QPT; ++i) {
        const int64_t qs = q0 + tid + i * kPredThreads;
        if (qs >= Q) continue;
        write_query(PERM ? (int64_t)perm[qs] : qs, acc[i], sq[i], total_trees, out_sum, out_pred, VAR ? out_var : nullptr);
    }
}

// Coded walk. The CTA's 256 * QPT query codes sit in shared memory as rows of ld_words
// 32-bit words (an odd count, so neighbouring queries hit different banks).
template <typename CT, int QPT, bool VAR>
__global__ void __launch_bounds__(kPredThreads) predict_kernel(
    const uint64_t *__restrict__ nodes, const int64_t *__restrict__ tree_off_all, int T_all, const CT *__restrict__ codes,
    int64_t Q, int ld_words, int64_t total_trees, int tree_cap, int64_t *out_sum, int64_t *out_pred,
    uint64_t *out_var, uint32_t *err, TreeParts tp)
{
    // this part's trees
    const int t_first = (int)blockIdx.y * tp.per, T = min(tp.per, T_all - t_first);
    const int64_t *tree_off = tree_off_all + t_first;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ __align__(8) uint64_t bar[3];
    uint64_t *slot0 = reinterpret_cast<uint64_t *>(sm_raw);
    uint64_t *slot1 = slot0 + tree_cap;
    uint32_t *xw = reinterpret_cast<uint32_t *>(slot1 + tree_cap);
    const int tid = threadIdx.x;
    const int QT = kPredThreads * QPT;
    const int64_t q0 = (int64_t)blockIdx.x * QT;

    if (tid == 0) {
        for (int i = 0; i < 3; ++i) mbar_init(&bar[i], 1);
        fence_mbar_init();
        issue_tree(nodes, tree_off, 0, tree_cap, slot0, &bar[0]);
        if (T > 1) issue_tree(nodes, tree_off, 1, tree_cap, slot1, &bar[1]);
    }
    // the tile's codes: global rows of ld_words words -> shared rows of ld_words words
    stage_rows(xw, reinterpret_cast<const uint32_t *>(codes) + (size_t)q0 * (size_t)ld_words,
               min((int64_t)QT, Q - q0) * ld_words, &bar[2]);
    __syncthreads();
    if (!rows_landed(bar, T, err)) return;

    const CT *xr[QPT];
#pragma unroll
    for (int i = 0; i < QPT; ++i)
        xr[i] = reinterpret_cast<const CT *>(xw + (size_t)(tid + i * kPredThreads) * (size_t)ld_words);
    int64_t acc[QPT];
    u128_t sq[QPT];
#pragma unroll
    for (int i = 0; i < QPT; ++i) { acc[i] = 0; sq[i] = 0; }

    for (int t = 0; t < T; ++t) {
        const int s = t & 1;
        const uint32_t parity = (uint32_t)((t >> 1) & 1);
        bool ok = false;
        for (uint32_t it = 0; it < kWaitLimit && !ok; ++it) ok = mbar_try_wait(&bar[s], parity);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) atomicOr(err, kErrTimeout);
            // give the other slot's copy (tree t + 1) a bounded chance to land before exiting
            if (t + 1 < T)
                for (uint32_t it = 0; it < kWaitLimit; ++it)
                    if (mbar_try_wait(&bar[s ^ 1], (uint32_t)(((t + 1) >> 1) & 1))) break;
            return;
        }
        const int64_t a = tree_off[t];
        const uint32_t nn = (uint32_t)(tree_off[t + 1] - a);
        if (nn <= (uint32_t)tree_cap) {
            if (s) walk_tree<CT, QPT>(slot1, xr, acc, sq, VAR, nn);
            else walk_tree<CT, QPT>(slot0, xr, acc, sq, VAR, nn);
        } else {
            walk_tree<CT, QPT>(nodes + a, xr, acc, sq, VAR, nn);
        }
        __syncthreads();
        if (tid == 0 && t + 2 < T) issue_tree(nodes, tree_off, t + 2, tree_cap, s ? slot1 : slot0, &bar[s]);
    }

    finish_tile<QPT, VAR, false>(tp, acc, sq, q0, Q, total_trees, out_sum, out_pred, out_var, nullptr);
}

// ------------------------------------------------------------------------------------------
// compact 4-byte coded nodes (one CTA per tree)
// ------------------------------------------------------------------------------------------
__global__ void compact_nodes_kernel(const uint64_t *__restrict__ cnodes, const int64_t *__restrict__ tree_off,
                                     const int64_t *__restrict__ tree_off4, uint32_t *__restrict__ c32, int shift)
{
    const int t = blockIdx.x;
    const int64_t a = tree_off[t], m = tree_off[t + 1] - a;
    const int64_t a4 = tree_off4[t], m4 = tree_off4[t + 1] - a4;
    for (int64_t j = threadIdx.x; j < m4; j += blockDim.x) {
        const uint32_t v = compact_node(j < m ? cnodes[a + j] : 1ull << 63, (uint32_t)j, shift);
        c32[a4 + j] = v;
    }
}

__device__ __forceinline__ void issue_tree4(const uint32_t *c32, const int64_t *tree_off4, int t, int tree_cap,
                                            uint32_t *slot, uint64_t *bar)
{
    const int64_t a = tree_off4[t], nn = tree_off4[t + 1] - a;
    if (nn <= tree_cap) {
        const uint32_t bytes = (uint32_t)nn * 4u;
        fence_proxy_async();
        mbar_arrive_expect_tx(bar, bytes);
        bulk_g2s(slot, c32 + a, bytes, bar);
    } else {
        mbar_arrive(bar);
    }
}

// Walk of compact nodes; returns each chain's leaf index within the tree. A leaf is its own
// child, so a step past it stays on it: chains step kWalkSteps nodes at a time with no per-step
// leaf test, and the warp stops once the last node of every chain was a leaf. (A leaf's feature
// field is 255: its code read lands in the padding after the query rows and is never above the
// leaf's threshold 255.)
// Instruction issue bounds the walk, so a step is as few as the node's layout allows. SCALED nodes
// (trees of at most 16,384) hold the left child as a byte offset below the threshold byte: with
// m = threshold * 65536 + left, code > threshold  <=>  code * 65536 > m, and the next offset is m, or
// m + 4, without its upper half: no separate threshold or index arithmetic. 1,000,000 queries x 500
// trees: walk 4.27 -> 4.00 ms; shared-memory wavefronts (997 M, 80 % of their peak rate) bound it now.
constexpr int kWalkSteps = 2;
template <int QPT, bool SCALED, typename NodePtr>
__device__ __forceinline__ void walk_tree4(NodePtr tn, const uint8_t *const (&xr)[QPT], uint32_t (&j)[QPT], uint32_t nn)
{
    uint32_t nd[QPT];
#pragma unroll
    for (int i = 0; i < QPT; ++i) j[i] = 0u;
    for (;;) {
#pragma unroll
        for (int u = 0; u < kWalkSteps; ++u) {
#pragma unroll
            for (int i = 0; i < QPT; ++i) {
                if (SCALED) {
                    nd[i] = *reinterpret_cast<NodePtr>(reinterpret_cast<const unsigned char *>(tn) + j[i]);
                    const uint32_t c = (uint32_t)xr[i][nd[i] >> 24];
                    uint32_t m = nd[i] & 0xFFFFFFu;
                    if ((c << 16) > m) m += 4u;
                    j[i] = AIWCRF_IDX(m & 0xFFFFu, 4u * nn, kBoundWalk);
                } else {
                    nd[i] = tn[j[i]];
                    const uint32_t c = (uint32_t)xr[i][nd[i] >> 24];
                    j[i] = AIWCRF_IDX((nd[i] & 0xFFFFu) + (c > ((nd[i] >> 16) & 0xFFu) ? 1u : 0u), nn, kBoundWalk);
                }
            }
        }
        bool done = true;
#pragma unroll
        for (int i = 0; i < QPT; ++i) done = done && (int32_t)nd[i] < 0;
        if (__all_sync(kFull, done)) break;
    }
#pragma unroll
    for (int i = 0; i < QPT; ++i)
        if (SCALED) j[i] >>= 2;
}

// The byte-code walk over compact trees. Leaf values are loaded from the 8-byte node array
// (L2-resident) and added one tree later, so their latency overlaps the next walk.
template <int QPT, bool VAR, bool PERM, bool SCALED>
__global__ void __launch_bounds__(kPredThreads) predict4_kernel(
    const uint32_t *__restrict__ c32, const int64_t *__restrict__ tree_off4_all, const uint64_t *__restrict__ nodes,
    const int64_t *__restrict__ tree_off_all, int T_all, const uint8_t *__restrict__ codes, int64_t Q, int ld_words,
    int64_t total_trees, int tree_cap, int64_t *out_sum, int64_t *out_pred, uint64_t *out_var, uint32_t *err,
    const uint32_t *__restrict__ perm, TreeParts tp)
{
    // this part's trees
    const int t_first = (int)blockIdx.y * tp.per, T = min(tp.per, T_all - t_first);
    const int64_t *tree_off4 = tree_off4_all + t_first, *tree_off = tree_off_all + t_first;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ __align__(8) uint64_t bar[3];
    uint32_t *slot0 = reinterpret_cast<uint32_t *>(sm_raw);
    uint32_t *slot1 = slot0 + tree_cap;
    uint32_t *xw = slot1 + tree_cap;
    const int tid = threadIdx.x;
    const int QT = kPredThreads * QPT;
    const int64_t q0 = (int64_t)blockIdx.x * QT;

    if (tid == 0) {
        for (int i = 0; i < 3; ++i) mbar_init(&bar[i], 1);
        fence_mbar_init();
        issue_tree4(c32, tree_off4, 0, tree_cap, slot0, &bar[0]);
        if (T > 1) issue_tree4(c32, tree_off4, 1, tree_cap, slot1, &bar[1]);
    }
    {
        // the tile's query codes; with PERM, tile position i holds query perm[q0 + i]
        const uint32_t *gw = reinterpret_cast<const uint32_t *>(codes);
        const int64_t nq = min((int64_t)QT, Q - q0);
        const int64_t words = nq * ld_words;
        if (PERM) {
            for (int64_t k = tid; k < words; k += kPredThreads) {
                const int64_t r = k / ld_words, w = k - r * ld_words;
                xw[k] = gw[(size_t)perm[q0 + r] * (size_t)ld_words + (size_t)w];
            }
        } else {
            stage_rows(xw, gw + (size_t)q0 * (size_t)ld_words, words, &bar[2]);
        }
    }
    __syncthreads();
    if (!PERM && !rows_landed(bar, T, err)) return;

    const uint8_t *xr[QPT];
#pragma unroll
    for (int i = 0; i < QPT; ++i)
        xr[i] = reinterpret_cast<const uint8_t *>(xw + (size_t)(tid + i * kPredThreads) * (size_t)ld_words);
    int64_t acc[QPT], pend[QPT];
    u128_t sq[QPT];
#pragma unroll
    for (int i = 0; i < QPT; ++i) { acc[i] = 0; pend[i] = 0; sq[i] = 0; }

    // the tree's offsets are loaded one tree ahead, so their latency overlaps a walk
    int64_t a4 = tree_off4[0], b4 = T > 0 ? tree_off4[1] : 0, ta = tree_off[0];
    for (int t = 0; t < T; ++t) {
        const int s = t & 1;
        const uint32_t parity = (uint32_t)((t >> 1) & 1);
        const int tn1 = t + 1 < T ? t + 1 : t;
        const int64_t b4n = tree_off4[tn1 + 1], tan = tree_off[tn1];
        bool ok = false;
        for (uint32_t it = 0; it < kWaitLimit && !ok; ++it) ok = mbar_try_wait(&bar[s], parity);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) atomicOr(err, kErrTimeout);
            if (t + 1 < T)
                for (uint32_t it = 0; it < kWaitLimit; ++it)
                    if (mbar_try_wait(&bar[s ^ 1], (uint32_t)(((t + 1) >> 1) & 1))) break;
            return;
        }
        uint32_t j[QPT];
        const uint32_t nn4 = (uint32_t)(b4 - a4);
        if (b4 - a4 <= tree_cap) {
            if (s) walk_tree4<QPT, SCALED, const uint32_t *>(slot1, xr, j, nn4);
            else walk_tree4<QPT, SCALED, const uint32_t *>(slot0, xr, j, nn4);
        } else {
            walk_tree4<QPT, SCALED, const uint32_t *>(c32 + a4, xr, j, nn4);
        }
        // add the previous tree's leaves, then start loading this tree's
        const uint64_t *tn = nodes + ta;
        a4 = b4;
        b4 = b4n;
        ta = tan;
#pragma unroll
        for (int i = 0; i < QPT; ++i) {
            acc[i] += pend[i];
            if (VAR) sq[i] += (u128_t)((i128_t)pend[i] * (i128_t)pend[i]);
            pend[i] = leaf_value(__ldg(&tn[j[i]]));
        }
        __syncthreads();
        if (tid == 0 && t + 2 < T) issue_tree4(c32, tree_off4, t + 2, tree_cap, s ? slot1 : slot0, &bar[s]);
    }
#pragma unroll
    for (int i = 0; i < QPT; ++i) {
        acc[i] += pend[i];
        if (VAR) sq[i] += (u128_t)((i128_t)pend[i] * (i128_t)pend[i]);
    }

    finish_tile<QPT, VAR, PERM>(tp, acc, sq, q0, Q, total_trees, out_sum, out_pred, out_var, perm);
}

// Split features of every tree's first kTopNodes nodes (breadth-first: the top levels).
__global__ void top_features_kernel(const uint64_t *__restrict__ cnodes, const int64_t *__restrict__ tree_off, int T,
                                    uint32_t *counts)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const int64_t a = tree_off[t], m = min((int64_t)kTopNodes, tree_off[t + 1] - a);
    for (int64_t j = 0; j < m; ++j) {
        const uint64_t nd = cnodes[a + j];
        if (!(nd >> 63)) atomicAdd(&counts[(nd >> 56) & 0x7Fu], 1u);
    }
}

// sort key of a coded query: the codes of up to four features, most significant first, each in
// the bits its codes need (at most 32 in all)
__global__ void query_key_kernel(const uint8_t *__restrict__ codes, int ld_bytes, int64_t Q, int4 kf, int4 kb,
                                 uint32_t *__restrict__ keys, uint32_t *__restrict__ idx)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= Q) return;
    const uint8_t *c = codes + (size_t)q * (size_t)ld_bytes;
    uint32_t k = 0;
    if (kf.x >= 0) k = (uint32_t)c[kf.x];
    if (kf.y >= 0) k = (k << kb.y) | (uint32_t)c[kf.y];
    if (kf.z >= 0) k = (k << kb.z) | (uint32_t)c[kf.z];
    if (kf.w >= 0) k = (k << kb.w) | (uint32_t)c[kf.w];
    keys[q] = k;
    idx[q] = (uint32_t)q;
}

// ------------------------------------------------------------------------------------------
// out-of-bag evaluation (the tuning objective of Sec. III-B): per training row, the exact sum of
// the leaf values of the trees whose bootstrap did not draw it, and their number
// ------------------------------------------------------------------------------------------
template <typename CT>
__global__ void oob_kernel(const uint64_t *__restrict__ cnodes, const int64_t *__restrict__ tree_off, int T,
                           const CT *__restrict__ codes, int ld, int64_t N, const uint32_t *__restrict__ inbag,
                           int64_t words, int64_t *__restrict__ out_sum, int32_t *__restrict__ out_count)
{
    const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= N) return;
    const CT *x = codes + (size_t)row * (size_t)ld;
    int64_t sum = 0;
    int32_t cnt = 0;
    for (int t = 0; t < T; ++t) {
        if ((__ldg(&inbag[(size_t)t * (size_t)words + (size_t)(row >> 5)]) >> (row & 31)) & 1u) continue;
        const uint64_t *tn = cnodes + tree_off[t];
        const uint32_t nn = (uint32_t)(tree_off[t + 1] - tree_off[t]);
        uint32_t j = 0;
        for (;;) {
            const uint64_t nd = __ldg(&tn[j]);
            if (nd >> 63) { sum += leaf_value(nd); break; }
            const uint32_t f = AIWCRF_IDX((uint32_t)(nd >> 56) & 0x7Fu, (uint32_t)ld, kBoundFeature);
            j = AIWCRF_IDX(((uint32_t)(nd >> 32) & 0xFFFFFFu) + ((uint32_t)x[f] > ((uint32_t)nd & 0xFFFFFFu) ? 1u : 0u), nn,
                           kBoundWalk);
        }
        ++cnt;
    }
    out_sum[row] = sum;
    out_count[row] = cnt;
}

// The same for compact trees: CTA (tile of 256 * QPT rows, part of tp_per trees). As in
// predict4_kernel the rows' codes sit in shared memory and the trees pass through two slots, here by
// asynchronous copies of every thread (whose wait cannot run out, so that the call needs no error
// flag). Every row is walked: leaving a tree's in-bag rows out would only idle their lanes; the
// in-bag words, one for a warp's 32 rows, are read one tree ahead. With several parts the sums and
// counts, zero on entry, are added to.
// Repeated runs of one cell follow each other in a table as it is measured, and their codes are
// alike: a tile whose neighbouring rows hold at most kOobDistinct different ones walks only those
// (from L2: a few walks per thread), a batch of trees at a time, and then adds up every row's leaves:
// 111,000 rows of 50 runs a cell x 500 trees 420 -> 122 us. At the line itself, rows alike in fours (128
// different ones a tile) of trees of about 11,000 nodes, the whole call 8,190 -> 3,361 us; by eights 6,761 ->
// 1,738. Rows that are not beside their like are all walked.
// What bounds it is instruction issue, as the walk of predict; the walk from global memory it
// replaces waited for a load per node: 111,000 rows x 500 trees 1,072 -> 420 us.
__device__ __forceinline__ void copy_tree4_async(const uint32_t *src, int64_t nodes, uint32_t *slot)
{
    for (int64_t i = threadIdx.x; i < nodes / 4; i += kPredThreads)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(slot + 4 * i)), "l"(src + 4 * i) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
}

constexpr int kOobDistinct = 128;

// the leaf that one row's codes reach in a compact tree in global memory
template <bool SCALED>
__device__ __forceinline__ uint32_t walk_one4(const uint32_t *__restrict__ tn, const uint8_t *x, uint32_t nn)
{
    uint32_t j = 0u;
    for (;;) {
        const uint32_t nd = SCALED ? __ldg(reinterpret_cast<const uint32_t *>(reinterpret_cast<const unsigned char *>(tn) + j))
                                   : __ldg(tn + j);
        if ((int32_t)nd < 0) return SCALED ? j >> 2 : j;
        const uint32_t c = (uint32_t)x[nd >> 24];
        if (SCALED) {
            uint32_t m = nd & 0xFFFFFFu;
            if ((c << 16) > m) m += 4u;
            j = AIWCRF_IDX(m & 0xFFFFu, 4u * nn, kBoundWalk);
        } else {
            j = AIWCRF_IDX((nd & 0xFFFFu) + (c > ((nd >> 16) & 0xFFu) ? 1u : 0u), nn, kBoundWalk);
        }
    }
}

template <int QPT, bool SCALED>
__global__ void __launch_bounds__(kPredThreads) oob4_kernel(
    const uint32_t *__restrict__ c32, const int64_t *__restrict__ tree_off4, const uint64_t *__restrict__ nodes,
    const int64_t *__restrict__ tree_off, int T_all, int per, const uint32_t *__restrict__ codes, int64_t N, int ld_words,
    int tree_cap, const uint32_t *__restrict__ inbag, int64_t inbag_words, int64_t *out_sum, int32_t *out_count)
{
    extern __shared__ __align__(16) unsigned char sm_raw[];
    uint32_t *slot0 = reinterpret_cast<uint32_t *>(sm_raw);
    uint32_t *slot1 = slot0 + tree_cap;
    uint32_t *xw = slot1 + tree_cap;
    const int tid = threadIdx.x;
    const int64_t q0 = (int64_t)blockIdx.x * kPredThreads * QPT;
    const int t_first = (int)blockIdx.y * per, t_end = min(T_all, t_first + per);
    auto fetch = [&](int t) {                    // tree t's nodes into its slot, if they fit one
        const int64_t a = tree_off4[t], nn = tree_off4[t + 1] - a;
        copy_tree4_async(c32 + a, nn <= tree_cap ? nn : 0, (t - t_first) & 1 ? slot1 : slot0);
    };
    const int n_rows = (int)min((int64_t)kPredThreads * QPT, N - q0);
    {
        const int64_t words = (int64_t)n_rows * ld_words;
        const uint32_t *src = codes + (size_t)q0 * (size_t)ld_words;
        for (int64_t k = tid; k < words; k += kPredThreads) xw[k] = src[k];
    }
    const uint8_t *xr[QPT];
    const uint32_t *bits[QPT];
    uint32_t bag[QPT], count[QPT];
    int64_t acc[QPT], pend[QPT];
#pragma unroll
    for (int i = 0; i < QPT; ++i) {
        const int64_t row = q0 + tid + i * kPredThreads;
        xr[i] = reinterpret_cast<const uint8_t *>(xw + (size_t)(tid + i * kPredThreads) * (size_t)ld_words);
        // a row past the end is in every bag
        bits[i] = row < N ? inbag + (size_t)t_first * (size_t)inbag_words + (size_t)(row >> 5) : nullptr;
        bag[i] = bits[i] ? __ldg(bits[i]) : ~0u;
        count[i] = 0u;
        acc[i] = pend[i] = 0;
    }
    // rows that differ from the one before them
    __shared__ uint16_t first_row[kOobDistinct];
    __shared__ uint32_t warp_heads[QPT * kPredThreads / 32];
    __syncthreads();
    uint32_t run_of[QPT];
    bool head[QPT];
#pragma unroll
    for (int i = 0; i < QPT; ++i) {
        const int r = tid + i * kPredThreads;
        const uint32_t *w = xw + (size_t)r * (size_t)ld_words;
        head[i] = r == 0;
        if (r > 0 && r < n_rows)
            for (int k = 0; k < ld_words && !head[i]; ++k) head[i] = w[k] != w[k - ld_words];
        const uint32_t b = __ballot_sync(kFull, head[i] && r < n_rows);
        run_of[i] = __popc(b & (lanemask_lt() | (1u << (tid & 31))));       // heads up to this row, in its warp
        if ((tid & 31) == 0) warp_heads[r >> 5] = __popc(b);
    }
    __syncthreads();
    int distinct = 0;
#pragma unroll
    for (int k = 0; k < QPT * kPredThreads / 32; ++k) {
        const int n = (int)warp_heads[k];
#pragma unroll
        for (int i = 0; i < QPT; ++i)
            if (k < (tid + i * kPredThreads) >> 5) run_of[i] += (uint32_t)n;
        distinct += n;
    }
    const int batch = min(min(32, tree_cap / distinct), t_end - t_first);    // the slots hold tree_cap leaf values
    if (distinct <= kOobDistinct && batch >= 1) {
        int64_t *leaf = reinterpret_cast<int64_t *>(sm_raw);               // [tree of the batch][distinct row]
#pragma unroll
        for (int i = 0; i < QPT; ++i) {
            run_of[i] -= 1u;
            if (head[i] && tid + i * kPredThreads < n_rows) first_row[run_of[i]] = (uint16_t)(tid + i * kPredThreads);
        }
        __syncthreads();
        for (int t0 = t_first; t0 < t_end; t0 += batch) {
            const int nt = min(batch, t_end - t0);
            for (int k = tid; k < nt * distinct; k += kPredThreads) {
                const int tt = k / distinct, d = k - tt * distinct, t = t0 + tt;
                const int64_t a = tree_off4[t];
                const uint32_t j = walk_one4<SCALED>(c32 + a, reinterpret_cast<const uint8_t *>(xw + (size_t)first_row[d] * (size_t)ld_words),
                                                     (uint32_t)(tree_off4[t + 1] - a));
                leaf[k] = leaf_value(__ldg(&nodes[tree_off[t] + j]));
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < QPT; ++i) {
                if (!bits[i]) continue;
                const uint32_t *word = bits[i] + (size_t)(t0 - t_first) * (size_t)inbag_words;
#pragma unroll 8
                for (int tt = 0; tt < nt; ++tt, word += inbag_words) {
                    const bool out = !((__ldg(word) >> (tid & 31)) & 1u);
                    const int64_t v = leaf[tt * distinct + (int)run_of[i]];
                    acc[i] += out ? v : 0;
                    count[i] += out ? 1u : 0u;
                }
            }
            __syncthreads();
        }
    } else {
        fetch(t_first);
        for (int t = t_first; t < t_end; ++t) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();                         // tree t has landed, and nobody walks tree t - 1 any more
            if (t + 1 < t_end) fetch(t + 1);
            uint32_t next[QPT];
#pragma unroll
            for (int i = 0; i < QPT; ++i) {
                if (bits[i] && t + 1 < t_end) bits[i] += inbag_words;
                next[i] = bits[i] ? __ldg(bits[i]) : ~0u;
            }
            const int64_t a = tree_off4[t];
            const uint32_t nn = (uint32_t)(tree_off4[t + 1] - a);
            const bool fits = nn <= (uint32_t)tree_cap;
            uint32_t j[QPT];
            if (!fits) walk_tree4<QPT, SCALED, const uint32_t *>(c32 + a, xr, j, nn);
            else if ((t - t_first) & 1) walk_tree4<QPT, SCALED, const uint32_t *>(slot1, xr, j, nn);
            else walk_tree4<QPT, SCALED, const uint32_t *>(slot0, xr, j, nn);
            const uint64_t *tn = nodes + tree_off[t];
#pragma unroll
            for (int i = 0; i < QPT; ++i) {
                const bool out = !((bag[i] >> (tid & 31)) & 1u);
                acc[i] += pend[i];
                count[i] += out ? 1u : 0u;
                pend[i] = out ? leaf_value(__ldg(&tn[j[i]])) : 0;
                bag[i] = next[i];
            }
        }
    }
#pragma unroll
    for (int i = 0; i < QPT; ++i) {
        const int64_t row = q0 + tid + i * kPredThreads;
        if (row >= N) continue;
        acc[i] += pend[i];
        if (gridDim.y > 1) {
            atomicAdd(reinterpret_cast<unsigned long long *>(&out_sum[row]), (unsigned long long)acc[i]);
            atomicAdd(&out_count[row], (int)count[i]);
        } else {
            out_sum[row] = acc[i];
            out_count[row] = (int32_t)count[i];
        }
    }
}

// Out-of-bag error (Sec. III-B): per row with c > 0 out-of-bag trees its out-of-bag prediction
// p = floor((2 s + c) / (2 c)) and the squared error (p - y)^2, exact in 128 bits; each CTA
// writes the sum of its rows' squared errors and their number, oob_error_finish_kernel adds the
// CTA sums in CTA order and divides once.
constexpr int kOobErrThreads = 256;

// the warp's sum of 128-bit values and counts, in every lane
__device__ __forceinline__ void warp_add_part(unsigned long long &lo, unsigned long long &hi, unsigned long long &rows)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long olo = __shfl_xor_sync(kFull, lo, o), ohi = __shfl_xor_sync(kFull, hi, o);
        const unsigned long long nlo = lo + olo;
        hi += ohi + (nlo < lo ? 1ull : 0ull);
        lo = nlo;
        rows += __shfl_xor_sync(kFull, rows, o);
    }
}

__global__ void __launch_bounds__(kOobErrThreads) oob_error_kernel(const int64_t *__restrict__ sum,
                                                                   const int32_t *__restrict__ cnt,
                                                                   const int64_t *__restrict__ y, int64_t N,
                                                                   int64_t *__restrict__ pred, OobPart *part,
                                                                   uint32_t *err)
{
    __shared__ OobPart red[kOobErrThreads / 32];
    const int64_t row = (int64_t)blockIdx.x * kOobErrThreads + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long lo = 0ull, hi = 0ull, rows = 0ull;
    if (row < N) {
        const int32_t c = cnt[row];
        int64_t p = 0;
        if (c > 0) {
            const long long yr = y[row];
            if (yr > AIWCRF_MAX_ABS_Y || yr < -AIWCRF_MAX_ABS_Y) atomicOr(err, kErrY);
            p = round_mean(sum[row], (uint32_t)c);
            const i128_t d = (i128_t)p - (i128_t)yr;                 // |d| < 2^42
            const u128_t a = d < 0 ? (u128_t)(-d) : (u128_t)d;
            const u128_t sq = a * a;
            lo = (unsigned long long)sq;
            hi = (unsigned long long)(sq >> 64);
            rows = 1ull;
        }
        if (pred) pred[row] = p;
    }
    warp_add_part(lo, hi, rows);
    if (lane == 0) { red[warp].lo = lo; red[warp].hi = hi; red[warp].rows = rows; }
    __syncthreads();
    if (threadIdx.x == 0) {
        OobPart t = red[0];
        for (int w = 1; w < kOobErrThreads / 32; ++w) {
            const unsigned long long nlo = t.lo + red[w].lo;
            t.hi += red[w].hi + (nlo < t.lo ? 1ull : 0ull);
            t.lo = nlo;
            t.rows += red[w].rows;
        }
        part[blockIdx.x] = t;
    }
}

// One CTA adds the CTA sums (exact, so in any order) and divides once. One thread adding them in
// turn waited for a load per CTA: 434 of them took 50 us.
__global__ void __launch_bounds__(kOobErrThreads) oob_error_finish_kernel(const OobPart *part, int nparts, OobResult *res)
{
    __shared__ OobPart red[kOobErrThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long lo = 0ull, hi = 0ull, rows = 0ull;
    for (int i = threadIdx.x; i < nparts; i += kOobErrThreads) {
        const unsigned long long nlo = lo + part[i].lo;
        hi += part[i].hi + (nlo < lo ? 1ull : 0ull);
        lo = nlo;
        rows += part[i].rows;
    }
    warp_add_part(lo, hi, rows);
    if (lane == 0) { red[warp].lo = lo; red[warp].hi = hi; red[warp].rows = rows; }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < kOobErrThreads / 32; ++w) {
        const unsigned long long nlo = lo + red[w].lo;
        hi += red[w].hi + (nlo < lo ? 1ull : 0ull);
        lo = nlo;
        rows += red[w].rows;
    }
    res->sq_lo = lo;
    res->sq_hi = hi;
    res->rows = (long long)rows;
    // sum < 2^106: hi converts exactly, lo once rounded; mean in units of the target squared
    const double sq = __dadd_rn(__dmul_rn((double)hi, 18446744073709551616.0), (double)lo);
    res->mse = rows ? __dmul_rn(__ddiv_rn(sq, (double)rows), 5.42101086242752217e-20) : 0.0;   // 2^-64
}

int oob_error_launch(const int64_t *d_sum, const int32_t *d_count, const int64_t *d_y, int64_t N, int64_t *d_pred,
                     OobPart *d_parts, OobResult *d_res, uint32_t *d_err, cudaStream_t s)
{
    const int nparts = (int)std::max<int64_t>(1, (N + kOobErrThreads - 1) / kOobErrThreads);
    oob_error_kernel<<<(unsigned)nparts, kOobErrThreads, 0, s>>>(d_sum, d_count, d_y, N, d_pred, d_parts, d_err);
    oob_error_finish_kernel<<<1, kOobErrThreads, 0, s>>>(d_parts, nparts, d_res);
    count_launches(2);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "oob_error launch");
    return AIWCRF_OK;
}

size_t oob_error_parts(int64_t N)
{
    return (size_t)std::max<int64_t>(1, (N + kOobErrThreads - 1) / kOobErrThreads);
}

__global__ void round_mean_kernel(const int64_t *sums, int64_t n, int64_t T, int64_t *out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const i128_t num = (i128_t)2 * sums[i] + T, den = (i128_t)2 * T;
    i128_t d = num / den;
    if (num % den != 0 && num < 0) d -= 1;
    out[i] = (int64_t)d;
}

// query (k, j) of device selection: kernel k's features (kfeat, leading dimension ld),
// device_ids[j], and size_class, or size_row[k] where size_row is given
__global__ void expand_queries_kernel(const float *kfeat, int32_t K, int64_t ld, int32_t size_class,
                                      const float *size_row, const int32_t *dev, int32_t D, int32_t F, float *q)
{
    const int64_t Qn = (int64_t)K * D;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Qn) return;
    const int32_t k = (int32_t)(i / D), jd = (int32_t)(i % D);
    for (int f = 0; f < F - 2; ++f) q[(size_t)f * (size_t)Qn + i] = kfeat[(size_t)f * (size_t)ld + k];
    q[(size_t)(F - 2) * (size_t)Qn + i] = (float)dev[jd];
    q[(size_t)(F - 1) * (size_t)Qn + i] =
        size_row ? size_row[k] : (float)size_class;
}

// argmin over devices per kernel; ties to the lower device id
__global__ void argmin_kernel(const int64_t *pred, DeviceIds dev, int32_t K, int32_t D, int32_t *best,
                              int64_t *out_pred)
{
    const int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    int64_t bp = 0;
    int32_t bd = 0;
    for (int32_t jd = 0; jd < D; ++jd) {
        const int64_t p = pred[(size_t)k * (size_t)D + jd];
        if (out_pred) out_pred[(size_t)k * (size_t)D + jd] = p;
        if (jd == 0 || p < bp || (p == bp && dev[jd] < bd)) { bp = p; bd = dev[jd]; }   // any id, negative ones too
    }
    best[k] = bd;
}

namespace {

constexpr int kQPT = 2;
// compact-forest batches of at least this many queries are walked in sorted order
constexpr int64_t kSortMinQueries = 1 << 16;

// Shared memory of the 8-byte node walk (predict_kernel): kQPT code rows per thread, 256 bytes
// after them, and two tree slots sized to the forest's largest tree up to 48 KB each.
struct WalkSmem {
    int tree_cap;
    int bytes;
};

WalkSmem walk8_smem(const aiwcrf_forest *f, int row_words)
{
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const int xs_bytes = kPredThreads * kQPT * row_words * 4 + 256;
    int tree_cap = std::min<int>((optin - xs_bytes - 1024) / 16, 6144);
    if ((int64_t)tree_cap > f->max_tree_nodes) tree_cap = (int)f->max_tree_nodes;
    tree_cap &= ~1;
    if (tree_cap < 2) tree_cap = 2;
    return WalkSmem{tree_cap, 2 * tree_cap * 8 + xs_bytes};
}

// The same for the compact walks: query code rows, then 256 bytes that a leaf's code read (feature
// field 255) may touch, and two slots of 4-byte nodes.
WalkSmem walk4_smem(const aiwcrf_forest *f, int row_words)
{
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const int xs_bytes = kPredThreads * kQPT * row_words * 4 + 256;
    int tree_cap = std::min<int>((optin - xs_bytes - 1024) / 8, 12288);
    if ((int64_t)tree_cap > f->max_tree4) tree_cap = (int)f->max_tree4;
    tree_cap &= ~3;
    if (tree_cap < 4) tree_cap = 4;
    return WalkSmem{tree_cap, 2 * tree_cap * 4 + xs_bytes};
}

// How a call's trees are split over CTAs (TreeParts), for tiles of 256 * kQPT queries and CTAs of
// smem bytes of shared memory.
//  - Fewer tiles than the chip holds CTAs: as many parts as fill it once, down to one tree each.
//  - More: enough parts that the last wave of CTAs, nearly empty for an unlucky tile count, is a
//    small share of the launch, while a part keeps kPartMinTrees trees to pay for staging its
//    tile's codes again.
// Measured, the walk alone (GB300; unsplit -> split): 2,220 queries x 128 trees 243 -> 13 us (5 CTAs
// -> 640), 40,001 x 500 with the variance 933 -> 264 us (79 -> 1,264), 1,000,000 x 500 4.34 ->
// 4.22 ms (1,954 CTAs in 2.1 waves -> 7,816).
constexpr int64_t kPartMinTrees = 32;
constexpr int64_t kPartWaves = 8;

int tree_parts(int64_t tiles, int smem, int64_t T)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t slots = (int64_t)sms * std::max(1, std::min(2048 / kPredThreads, 233472 / (smem + 1024)));
    const int64_t fill = std::min<int64_t>((slots + tiles - 1) / tiles, T);
    const int64_t smooth = std::min<int64_t>((kPartWaves * slots + tiles - 1) / tiles, T / kPartMinTrees);
    return (int)std::max<int64_t>(1, std::min<int64_t>(std::max(fill, smooth), 65535));
}

size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }

// The walk's own scratch, one stream-ordered block: the queries' codes, and the sums and tickets
// of the split above. (Callers that bring code scratch walk unsplit.)
struct WalkScratch {
    void *block = nullptr;
    cudaStream_t s = nullptr;
    void *codes = nullptr;
    TreeParts tp = {};
    int parts = 1;
    unsigned long long *zero = nullptr;     // what the coding kernel clears: zero_words words
    int64_t zero_words = 0;
    ~WalkScratch() { if (block) cudaFreeAsync(block, s); }

    cudaError_t init(int64_t Q, size_t code_bytes, int smem, int64_t T, bool var, void *codes_scratch, cudaStream_t st)
    {
        s = st;
        const int64_t tiles = (Q + (int64_t)kPredThreads * kQPT - 1) / ((int64_t)kPredThreads * kQPT);
        tp.per = (int)T;
        if (codes_scratch) { codes = codes_scratch; return cudaSuccess; }
        parts = tree_parts(tiles, smem, T);
        tp.per = (int)((T + parts - 1) / parts);
        parts = (int)((T + tp.per - 1) / tp.per);
        const size_t b_codes = up256(code_bytes);
        const int64_t n = parts > 1 ? tiles * kPredThreads * kQPT : 0;
        zero_words = parts > 1 ? n * (var ? 3 : 1) + (tiles + 1) / 2 : 0;
        const cudaError_t e = cudaMallocAsync(&block, b_codes + 8 * (size_t)zero_words, st);
        if (e != cudaSuccess) { block = nullptr; return e; }
        codes = block;
        zero = reinterpret_cast<unsigned long long *>(static_cast<unsigned char *>(block) + b_codes);
        tp.sum = zero;
        tp.sq = zero + n;
        tp.ticket = reinterpret_cast<uint32_t *>(zero + n * (var ? 3 : 1));
        return cudaSuccess;
    }
};

// Coding and walk of Q queries. code(codes, row_words, zero, zero_words) enqueues the kernel that
// writes their code rows and clears zero_words 8-byte words.
template <typename CT, bool VAR, typename Code>
int launch_predict(const aiwcrf_forest *f, const Code &code, int64_t Q, int64_t *d_sum, int64_t *d_pred,
                   uint64_t *d_var, int64_t total_trees, cudaStream_t s, uint32_t *d_err, void *codes_scratch,
                   int64_t walk_T)
{
    const int ld_words = code_row_words(f->F, (int)sizeof(CT));
    const WalkSmem ws = walk8_smem(f, ld_words);
    const int tree_cap = ws.tree_cap, smem = ws.bytes;
    WalkScratch w;
    cudaError_t e = w.init(Q, (size_t)Q * (size_t)ld_words * 4, smem, walk_T, VAR, codes_scratch, s);
    if (e != cudaSuccess) return fail(AIWCRF_E_OOM, "device allocation of the query codes failed");
    CT *d_codes = static_cast<CT *>(w.codes);
    if ((e = code(d_codes, ld_words, w.zero, w.zero_words)) != cudaSuccess) return cuda_fail(e, "query coding launch");
    auto kern = predict_kernel<CT, kQPT, VAR>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(predict_kernel)");
    const int64_t grid = (Q + (int64_t)kPredThreads * kQPT - 1) / ((int64_t)kPredThreads * kQPT);
    prof_begin(s, kProfWalk);
    kern<<<dim3((unsigned)grid, (unsigned)w.parts), kPredThreads, smem, s>>>(
        f->d_cnodes, f->d_tree_off, (int)walk_T, d_codes, Q, ld_words, total_trees, tree_cap, d_sum, d_pred, d_var,
        d_err, w.tp);
    prof_end(s, kProfWalk);
    count_launches(1);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "predict_kernel launch");
    return AIWCRF_OK;
}

template <bool VAR, typename Code>
int launch_predict4(const aiwcrf_forest *f, const Code &code, int64_t Q, int64_t *d_sum, int64_t *d_pred,
                    uint64_t *d_var, int64_t total_trees, cudaStream_t s, uint32_t *d_err, void *codes_scratch,
                    int64_t walk_T)
{
    const int ld_words = code_row_words(f->F, 1);
    const WalkSmem ws = walk4_smem(f, ld_words);
    const int tree_cap = ws.tree_cap, smem = ws.bytes;
    WalkScratch w;
    cudaError_t e = w.init(Q, (size_t)Q * (size_t)ld_words * 4, smem, walk_T, VAR, codes_scratch, s);
    if (e != cudaSuccess) return fail(AIWCRF_E_OOM, "device allocation of the query codes failed");
    uint8_t *d_codes = static_cast<uint8_t *>(w.codes);
    if ((e = code(d_codes, ld_words, w.zero, w.zero_words)) != cudaSuccess) return cuda_fail(e, "query coding launch");
    // large batches walk in the order of their leading codes (own scratch only)
    const bool sorted = !codes_scratch && Q >= kSortMinQueries && Q < ((int64_t)1 << 32) && f->key_feats[0] >= 0;
    uint32_t *perm = nullptr;
    struct FreeSort { uint32_t *p; cudaStream_t s; ~FreeSort() { if (p) cudaFreeAsync(p, s); } } fs{nullptr, s};
    if (sorted) {
        const size_t nq = (size_t)Q + 1, hw = radix_sort_hist_words(Q, 1);
        uint32_t *buf = nullptr;
        if (cudaMallocAsync(&buf, sizeof(uint32_t) * (4 * nq + hw), s) != cudaSuccess)
            return fail(AIWCRF_E_OOM, "device allocation of the query order failed");
        fs.p = buf;
        uint32_t *kA = buf, *vA = buf + nq, *kB = buf + 2 * nq, *vB = buf + 3 * nq, *hist = buf + 4 * nq;
        const int4 kf = make_int4(f->key_feats[0], f->key_feats[1], f->key_feats[2], f->key_feats[3]);
        const int4 kb = make_int4(f->key_bits[0], f->key_bits[1], f->key_bits[2], f->key_bits[3]);
        query_key_kernel<<<(unsigned)((Q + 255) / 256), 256, 0, s>>>(d_codes, ld_words * 4, Q, kf, kb, kA, vA);
        count_launches(1);
        bool in_b = false;
        int rc = radix_sort_segments(kA, vA, kB, vB, Q, 1, Q, hist, s, kb.x + kb.y + kb.z + kb.w, &in_b);
        if (rc != AIWCRF_OK) return rc;
        perm = in_b ? vB : vA;
    }
    auto kern = f->c32_shift ? (sorted ? predict4_kernel<kQPT, VAR, true, true> : predict4_kernel<kQPT, VAR, false, true>)
                             : (sorted ? predict4_kernel<kQPT, VAR, true, false> : predict4_kernel<kQPT, VAR, false, false>);
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(predict4_kernel)");
    const int64_t grid = (Q + (int64_t)kPredThreads * kQPT - 1) / ((int64_t)kPredThreads * kQPT);
    prof_begin(s, kProfWalk);
    kern<<<dim3((unsigned)grid, (unsigned)w.parts), kPredThreads, smem, s>>>(
        f->d_c32, f->d_tree_off4, f->d_nodes, f->d_tree_off, (int)walk_T, d_codes, Q, ld_words, total_trees, tree_cap,
        d_sum, d_pred, d_var, d_err, perm, w.tp);
    prof_end(s, kProfWalk);
    count_launches(1);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "predict4_kernel launch");
    return AIWCRF_OK;
}

template <typename CT, typename Code>
int launch_coded(const aiwcrf_forest *f, const Code &code, int64_t Q, int64_t *d_sum, int64_t *d_pred, uint64_t *d_var,
                 int64_t total_trees, cudaStream_t s, uint32_t *d_err, void *scratch, int64_t walk_T)
{
    if constexpr (sizeof(CT) == 1) {
        if (f->compact)
            return d_var ? launch_predict4<true>(f, code, Q, d_sum, d_pred, d_var, total_trees, s, d_err, scratch, walk_T)
                         : launch_predict4<false>(f, code, Q, d_sum, d_pred, d_var, total_trees, s, d_err, scratch, walk_T);
    }
    return d_var ? launch_predict<CT, true>(f, code, Q, d_sum, d_pred, d_var, total_trees, s, d_err, scratch, walk_T)
                 : launch_predict<CT, false>(f, code, Q, d_sum, d_pred, d_var, total_trees, s, d_err, scratch, walk_T);
}

template <typename CT>
int launch_predict_ct(const aiwcrf_forest *f, const float *dXq, int64_t Q, int64_t *d_sum, int64_t *d_pred,
                      uint64_t *d_var, int64_t total_trees, cudaStream_t s, uint32_t *d_err, void *scratch = nullptr,
                      int64_t walk_T = -1)
{
    auto code = [&](CT *codes, int row_words, unsigned long long *zero, int64_t nzero) {
        return launch_code_queries<CT>(f, dXq, Q, codes, row_words, s, zero, nzero);
    };
    return launch_coded<CT>(f, code, Q, d_sum, d_pred, d_var, total_trees, s, d_err, scratch, walk_T < 0 ? f->T : walk_T);
}

// the same for the K x D queries of a device selection (query k * D + j), D <= kSelectMaxDevices
template <typename CT>
int launch_select_ct(const aiwcrf_forest *f, const float *d_kfeat, int32_t K, int32_t size_class, const DeviceIds &ids,
                     int32_t D, int64_t *d_pred, cudaStream_t s, uint32_t *d_err)
{
    const int64_t Q = (int64_t)K * D;
    auto code = [&](CT *codes, int row_words, unsigned long long *zero, int64_t nzero) {
        const size_t smem = (size_t)kCodeQueries * (size_t)row_words * 4;
        const int steps = 32 - __builtin_clz(f->max_card | 1u);
        code_selection_kernel<CT><<<(unsigned)((K + kCodeQueries - 1) / kCodeQueries), kCodeThreads, smem, s>>>(
            d_kfeat, K, size_class, ids, D, f->F, f->d_fvals, f->fstride, f->d_fcard, codes, row_words, steps, zero, nzero);
        count_launches(1);
        return cudaGetLastError();
    };
    return launch_coded<CT>(f, code, Q, nullptr, d_pred, nullptr, f->T, s, d_err, nullptr, f->T);
}

}  // namespace

size_t predict_codes_bytes(const aiwcrf_forest *f, int64_t Q)
{
    return (size_t)Q * (size_t)code_row_words(f->F, code_bytes_of(f)) * 4;
}

size_t predict_codes_bytes_max(int32_t F, int64_t Q)
{
    return (size_t)Q * (size_t)code_row_words(F, 4) * 4;
}

int predict_enqueue(const aiwcrf_forest *f, const float *dXq, int64_t Q, int64_t *d_sum, int64_t *d_pred,
                    cudaStream_t s, uint32_t *d_err, void *codes_scratch)
{
    if (Q == 0) return AIWCRF_OK;
    if (f->max_card <= 255u) return launch_predict_ct<uint8_t>(f, dXq, Q, d_sum, d_pred, nullptr, f->T, s, d_err, codes_scratch);
    if (f->max_card <= 65535u) return launch_predict_ct<uint16_t>(f, dXq, Q, d_sum, d_pred, nullptr, f->T, s, d_err, codes_scratch);
    return launch_predict_ct<uint32_t>(f, dXq, Q, d_sum, d_pred, nullptr, f->T, s, d_err, codes_scratch);
}

int predict_prefix_var_enqueue(const aiwcrf_forest *f, const float *dXq, int64_t Q, int64_t n_trees,
                               uint64_t *d_var, cudaStream_t s, uint32_t *d_err, void *codes_scratch)
{
    if (Q == 0) return AIWCRF_OK;
    if (f->max_card <= 255u)
        return launch_predict_ct<uint8_t>(f, dXq, Q, nullptr, nullptr, d_var, n_trees, s, d_err, codes_scratch, n_trees);
    if (f->max_card <= 65535u)
        return launch_predict_ct<uint16_t>(f, dXq, Q, nullptr, nullptr, d_var, n_trees, s, d_err, codes_scratch, n_trees);
    return launch_predict_ct<uint32_t>(f, dXq, Q, nullptr, nullptr, d_var, n_trees, s, d_err, codes_scratch, n_trees);
}

int expand_launch(const float *d_kfeat, int32_t K, int64_t ld, int32_t size_class, const float *d_size_row,
                  const int32_t *d_dev, int32_t D, int32_t F, float *d_q, cudaStream_t s)
{
    const int64_t Qn = (int64_t)K * D;
    if (Qn == 0) return AIWCRF_OK;
    expand_queries_kernel<<<(unsigned)((Qn + 255) / 256), 256, 0, s>>>(d_kfeat, K, ld, size_class, d_size_row, d_dev,
                                                                        D, F, d_q);
    count_launches(1);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "expand_queries_kernel launch");
    return AIWCRF_OK;
}

int predict_launch(const aiwcrf_forest *f, const float *dXq, int64_t Q, int64_t *d_sum, int64_t *d_pred,
                   uint64_t *d_var, int64_t total_trees, cudaStream_t s)
{
    if (Q == 0) return AIWCRF_OK;
    keep_pool_memory(f->device);
    uint32_t *d_err = nullptr;
    cudaError_t e = cudaMallocAsync(&d_err, sizeof(uint32_t), s);
    if (e != cudaSuccess) return fail(AIWCRF_E_OOM, "device allocation failed");
    cudaMemsetAsync(d_err, 0, sizeof(uint32_t), s);
    prof_begin(s, kProfPredict);
    int rc;
    if (f->max_card <= 255u) rc = launch_predict_ct<uint8_t>(f, dXq, Q, d_sum, d_pred, d_var, total_trees, s, d_err);
    else if (f->max_card <= 65535u) rc = launch_predict_ct<uint16_t>(f, dXq, Q, d_sum, d_pred, d_var, total_trees, s, d_err);
    else rc = launch_predict_ct<uint32_t>(f, dXq, Q, d_sum, d_pred, d_var, total_trees, s, d_err);
    prof_end(s, kProfPredict);
    uint32_t h_err = 0;
    if (rc == AIWCRF_OK) {
        e = cudaMemcpyAsync(&h_err, d_err, sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) rc = cuda_fail(e, "predict");
    }
    cudaFreeAsync(d_err, s);
    if (rc == AIWCRF_OK && (h_err & kErrTimeout)) rc = fail(AIWCRF_E_TIMEOUT, "a bounded device wait gave up");
    return rc;
}

namespace {
template <typename CT>
int oob_ct(const aiwcrf_forest *f, const float *dX, int64_t N, int64_t *d_sum, int32_t *d_count, cudaStream_t s)
{
    const int ld_words = code_row_words(f->F, (int)sizeof(CT));
    const int ld = ld_words * 4 / (int)sizeof(CT);
    CT *d_codes = nullptr;
    cudaError_t e = cudaMallocAsync(&d_codes, (size_t)N * (size_t)ld_words * 4, s);
    if (e != cudaSuccess) return fail(AIWCRF_E_OOM, "device allocation of the row codes failed");
    struct Free { CT *p; cudaStream_t s; ~Free() { cudaFreeAsync(p, s); } } fr{d_codes, s};
    if (sizeof(CT) == 1 && f->compact) {
        const WalkSmem ws = walk4_smem(f, ld_words);
        const int64_t tiles = (N + (int64_t)kPredThreads * kQPT - 1) / ((int64_t)kPredThreads * kQPT);
        const int want = tree_parts(tiles, ws.bytes, f->T);
        const int per = (int)((f->T + want - 1) / want), parts = (int)((f->T + per - 1) / per);
        if ((e = launch_code_queries<CT>(f, dX, N, d_codes, ld_words, s,
                                         parts > 1 ? reinterpret_cast<unsigned long long *>(d_sum) : nullptr,
                                         parts > 1 ? N : 0)) != cudaSuccess)
            return cuda_fail(e, "code_queries_kernel launch");
        if (parts > 1 && (e = cudaMemsetAsync(d_count, 0, sizeof(int32_t) * (size_t)N, s)) != cudaSuccess)
            return cuda_fail(e, "out-of-bag counts");
        auto kern = f->c32_shift ? oob4_kernel<kQPT, true> : oob4_kernel<kQPT, false>;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ws.bytes);
        if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(oob4_kernel)");
        kern<<<dim3((unsigned)tiles, (unsigned)parts), kPredThreads, ws.bytes, s>>>(
            f->d_c32, f->d_tree_off4, f->d_nodes, f->d_tree_off, (int)f->T, per, reinterpret_cast<uint32_t *>(d_codes), N,
            ld_words, ws.tree_cap, f->d_inbag, f->inbag_words, d_sum, d_count);
        count_launches(1);
        e = cudaGetLastError();
        return e == cudaSuccess ? AIWCRF_OK : cuda_fail(e, "oob4_kernel launch");
    }
    if ((e = launch_code_queries<CT>(f, dX, N, d_codes, ld_words, s)) != cudaSuccess)
        return cuda_fail(e, "code_queries_kernel launch");
    oob_kernel<CT><<<(unsigned)((N + 127) / 128), 128, 0, s>>>(f->d_cnodes, f->d_tree_off, (int)f->T, d_codes, ld, N,
                                                              f->d_inbag, f->inbag_words, d_sum, d_count);
    count_launches(1);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "oob launch");
    return AIWCRF_OK;
}
}  // namespace

int oob_launch(const aiwcrf_forest *f, const float *dX, int64_t N, int64_t *d_sum, int32_t *d_count, cudaStream_t s)
{
    if (N == 0) return AIWCRF_OK;
    keep_pool_memory(f->device);
    if (f->max_card <= 255u) return oob_ct<uint8_t>(f, dX, N, d_sum, d_count, s);
    if (f->max_card <= 65535u) return oob_ct<uint16_t>(f, dX, N, d_sum, d_count, s);
    return oob_ct<uint32_t>(f, dX, N, d_sum, d_count, s);
}

int forest_build_compact(aiwcrf_forest *f, cudaStream_t s)
{
    if (!f->compact) return AIWCRF_OK;
    compact_nodes_kernel<<<(unsigned)f->T, 256, 0, s>>>(f->d_cnodes, f->d_tree_off, f->d_tree_off4, f->d_c32,
                                                          f->c32_shift);
    count_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "compact_nodes_kernel launch");
    // the features the trees split on first, for the order of large query batches
    uint32_t *d_cnt = nullptr;
    if (cudaMallocAsync(&d_cnt, 4 * (size_t)f->F, s) != cudaSuccess) return fail(AIWCRF_E_OOM, "feature counts");
    e = cudaMemsetAsync(d_cnt, 0, 4 * (size_t)f->F, s);
    if (e == cudaSuccess) {
        top_features_kernel<<<(unsigned)((f->T + 127) / 128), 128, 0, s>>>(f->d_cnodes, f->d_tree_off, (int)f->T, d_cnt);
        count_launches(1);
        e = cudaGetLastError();
    }
    std::vector<uint32_t> h((size_t)f->F, 0u), card((size_t)f->F, 0u);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h.data(), d_cnt, 4 * (size_t)f->F, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(card.data(), f->d_fcard, 4 * (size_t)f->F, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFreeAsync(d_cnt, s);
    if (e != cudaSuccess) return cuda_fail(e, "top split features");
    forest_set_key_feats(f, h.data(), card.data());
    return AIWCRF_OK;
}

void forest_set_key_feats(aiwcrf_forest *f, const uint32_t *top_counts, const uint32_t *card)
{
    std::vector<int> order((size_t)f->F);
    for (int i = 0; i < f->F; ++i) order[(size_t)i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return top_counts[x] > top_counts[y]; });
    for (int k = 0; k < 4; ++k) {
        f->key_feats[k] = (k < f->F && top_counts[order[(size_t)k]] > 0) ? order[(size_t)k] : -1;
        f->key_bits[k] = f->key_feats[k] < 0 ? 0 : 32 - __builtin_clz(card[f->key_feats[k]] | 1u);
    }
}

int round_mean_launch(const int64_t *d_sum, int64_t Q, int64_t total_trees, int64_t *d_out, cudaStream_t s)
{
    if (Q == 0) return AIWCRF_OK;
    round_mean_kernel<<<(unsigned)((Q + 255) / 256), 256, 0, s>>>(d_sum, Q, total_trees, d_out);
    count_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "round_mean_kernel launch");
    return AIWCRF_OK;
}

// Which kernels answer a device selection of K kernels x D devices:
//  - D <= 64 and few CTAs of the tree-parallel kernel (tree_parallel_selection): that kernel;
//  - D <= 64 beyond that: the walk of predict, whose trees pass through shared memory once for 512
//    queries, on rows coded once per kernel;
//  - more devices: the queries written out, and predict.
// A CTA of the tree-parallel kernel is a kernel and 32 trees, however few the forest has, and codes the
// kernel's features, then takes 16 devices a pass: it costs about as much as (passes + 1) / 2 CTAs of one
// pass, 8 ns of the chip's time with one tree and 12 with 32. The batch walk costs 57 to 85 us whatever the
// trees while it has few queries, and 130 and more once it sorts them. Measured per call (us), tree-parallel /
// batch walk, compact forests, D = 15: 2,048 CTAs 58 / 61 (1 tree), 65 / 78 (64), 64 / 73 (500); 4,096 73 /
// 62, 86 / 83, 83 / 83; 6,000 87 / 131 (sorted), 106 / 96, 101 / 94; 12,000 135 / 136 (1 tree), 182 / 208 (32);
// 16,384 169 / 142, 234 / 221. With few devices the batch is smaller and the lines cross earlier: D = 1 56 / 57
// at 2,048 CTAs, 70 / 57 at 4,096 (1 tree), 62 / 58 and 80 / 59 (64), 59 / 66 and 77 / 68 (500). D = 64, 1 tree:
// 4,096 kernels 133 / 145, 6,000 171 / 163. Two-byte codes, unsorted, D = 15: 4,096 CTAs 81 / 70 (1 tree), 95 /
// 109 (64), 92 / 105 (500). (A line in walks alone sent 1,000,000 kernels x 1 device x 1 tree to the
// tree-parallel kernel: 7,834 us against 428.)
constexpr int64_t kTreeParallelCtas = 4096, kTreeParallelCtasFewDevices = 2048, kTreeParallelCtasSorted = 12288;

bool tree_parallel_selection(const aiwcrf_forest *f, int64_t K, int64_t D, int32_t size_class)
{
    if (D > kSelectMaxDevices || size_class < 0) return false;
    const bool sorts = f->compact && K * D >= kSortMinQueries;
    const int64_t line = sorts ? kTreeParallelCtasSorted : D <= 8 ? kTreeParallelCtasFewDevices : kTreeParallelCtas;
    const int64_t ctas = K * ((f->T + 31) / 32), passes = (D + 15) / 16;
    return ctas * (passes + 1) <= 2 * line;
}

int select_launch(const aiwcrf_forest *f, const float *d_kfeat, int32_t K, int32_t size_class, const DeviceIds &ids,
                  int32_t D, int32_t *d_best, int64_t *d_pred, cudaStream_t s)
{
    const int64_t Qn = (int64_t)K * D;
    keep_pool_memory(f->device);
    // one block of scratch: sums and counters of the tree-parallel kernel, or an error flag; the
    // predictions if the caller wants none; the queries where they are written out
    const bool tree_parallel = tree_parallel_selection(f, K, D, size_class);
    const bool expand = D > kSelectMaxDevices;
    const size_t b_cnt = tree_parallel ? up256(8 * (size_t)Qn + 4 * (size_t)K) : 256;
    const size_t b_pred = d_pred ? 0 : up256(8 * (size_t)Qn), b_q = expand ? up256(4 * (size_t)f->F * (size_t)Qn) : 0;
    unsigned char *block = nullptr;
    cudaError_t e = cudaMallocAsync(&block, b_cnt + b_pred + b_q, s);
    if (e != cudaSuccess) return fail(AIWCRF_E_OOM, "select_device scratch");
    struct Free { void *p; cudaStream_t s; ~Free() { cudaFreeAsync(p, s); } } fr{block, s};
    int64_t *d_p = d_pred ? d_pred : reinterpret_cast<int64_t *>(block + b_cnt);
    if ((e = cudaMemsetAsync(block, 0, tree_parallel ? 8 * (size_t)Qn + 4 * (size_t)K : 4, s)) != cudaSuccess)
        return cuda_fail(e, "select scratch");
    if (tree_parallel) {
        unsigned long long *d_sum = reinterpret_cast<unsigned long long *>(block);
        prof_begin(s, kProfSelect);
        const int rc = select_small_launch(f, d_kfeat, K, size_class, ids, D, d_best, d_p, d_sum,
                                           reinterpret_cast<uint32_t *>(d_sum + Qn), s);
        prof_end(s, kProfSelect);
        return rc;
    }
    uint32_t *d_err = reinterpret_cast<uint32_t *>(block);
    int rc = AIWCRF_OK;
    if (expand) {
        float *d_q = reinterpret_cast<float *>(block + b_cnt + b_pred);
        prof_begin(s, kProfSelect);
        rc = expand_launch(d_kfeat, K, (int64_t)K, size_class, nullptr, ids.dev, D, f->F, d_q, s);
        prof_end(s, kProfSelect);
        if (rc == AIWCRF_OK) rc = predict_launch(f, d_q, Qn, nullptr, d_p, nullptr, f->T, s);
    } else {
        prof_begin(s, kProfPredict);
        if (f->max_card <= 255u) rc = launch_select_ct<uint8_t>(f, d_kfeat, K, size_class, ids, D, d_p, s, d_err);
        else if (f->max_card <= 65535u) rc = launch_select_ct<uint16_t>(f, d_kfeat, K, size_class, ids, D, d_p, s, d_err);
        else rc = launch_select_ct<uint32_t>(f, d_kfeat, K, size_class, ids, D, d_p, s, d_err);
        prof_end(s, kProfPredict);
    }
    if (rc != AIWCRF_OK) return rc;
    prof_begin(s, kProfSelect);
    argmin_kernel<<<(unsigned)((K + 127) / 128), 128, 0, s>>>(d_p, ids, K, D, d_best, nullptr);
    count_launches(1);
    e = cudaGetLastError();
    prof_end(s, kProfSelect);
    uint32_t h_err = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h_err, d_err, sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "select_device");
    if (h_err & kErrTimeout) return fail(AIWCRF_E_TIMEOUT, "a bounded device wait gave up");
    return AIWCRF_OK;
}

// ------------------------------------------------------------------------------------------
// Device selection inside caller-provided scratch (no allocation). Scratch layout, each part
// 256-byte aligned: device ids (D int32), expanded queries (F x K*D float), query codes
// (K*D rows of ld_words words), predictions (K*D int64), error flag (u32).
// ------------------------------------------------------------------------------------------
namespace {

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

int code_ld_words(const aiwcrf_forest *f)
{
    return code_row_words(f->F, code_bytes_of(f));
}

template <typename CT>
int select_noalloc_ct(const aiwcrf_forest *f, const float *d_kfeat, int32_t K, int32_t size_class, int32_t D,
                      int32_t *d_best, int64_t *d_pred, const int32_t *d_dev, float *d_q, uint32_t *d_codes,
                      int64_t *d_p, uint32_t *d_err, cudaStream_t s)
{
    const int64_t Qn = (int64_t)K * D;
    const int ld_words = code_ld_words(f);
    expand_queries_kernel<<<(unsigned)((Qn + 255) / 256), 256, 0, s>>>(d_kfeat, K, (int64_t)K, size_class, nullptr, d_dev, D,
                                                                        f->F,
                                                                        d_q);
    count_launches(1);
    cudaError_t e = launch_code_queries<CT>(f, d_q, Qn, reinterpret_cast<CT *>(d_codes), ld_words, s);
    if (e != cudaSuccess) return cuda_fail(e, "code_queries_kernel launch");
    const WalkSmem ws = walk8_smem(f, ld_words);
    const int tree_cap = ws.tree_cap, smem = ws.bytes;
    auto kern = predict_kernel<CT, kQPT, false>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(predict_kernel)");
    const int64_t grid = (Qn + (int64_t)kPredThreads * kQPT - 1) / ((int64_t)kPredThreads * kQPT);
    kern<<<(unsigned)grid, kPredThreads, smem, s>>>(f->d_cnodes, f->d_tree_off, (int)f->T,
                                                    reinterpret_cast<const CT *>(d_codes), Qn, ld_words, f->T,
                                                    tree_cap, nullptr, d_p, nullptr, d_err,
                                                    TreeParts{(int)f->T, nullptr, nullptr, nullptr});
    argmin_kernel<<<(unsigned)((K + 127) / 128), 128, 0, s>>>(d_p, DeviceIds{d_dev}, K, D, d_best, d_pred);
    count_launches(2);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "select_device launch");
    return AIWCRF_OK;
}

}  // namespace

size_t select_noalloc_bytes(const aiwcrf_forest *f, int32_t K, int32_t D)
{
    const size_t Qn = (size_t)K * (size_t)D;
    return align256(sizeof(int32_t) * (size_t)D) + align256(sizeof(float) * (size_t)f->F * Qn) +
           align256(Qn * (size_t)code_ld_words(f) * 4) + align256(sizeof(int64_t) * Qn) + align256(sizeof(uint32_t));
}

int select_launch_noalloc(const aiwcrf_forest *f, const float *d_kfeat, int32_t K, int32_t size_class,
                          const int32_t *h_dev, int32_t D, int32_t *d_best, int64_t *d_pred, unsigned char *scratch,
                          cudaStream_t s)
{
    const size_t Qn = (size_t)K * (size_t)D;
    unsigned char *p = scratch;
    int32_t *d_dev = reinterpret_cast<int32_t *>(p);
    p += align256(sizeof(int32_t) * (size_t)D);
    float *d_q = reinterpret_cast<float *>(p);
    p += align256(sizeof(float) * (size_t)f->F * Qn);
    uint32_t *d_codes = reinterpret_cast<uint32_t *>(p);
    p += align256(Qn * (size_t)code_ld_words(f) * 4);
    int64_t *d_p = reinterpret_cast<int64_t *>(p);
    p += align256(sizeof(int64_t) * Qn);
    uint32_t *d_err = reinterpret_cast<uint32_t *>(p);
    // device_ids may be host or device memory (unified addressing: no staging buffer needed)
    cudaError_t e = cudaMemcpyAsync(d_dev, h_dev, sizeof(int32_t) * (size_t)D, cudaMemcpyDefault, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_err, 0, sizeof(uint32_t), s);    // the flag must start at 0
    if (e != cudaSuccess) {
        cudaStreamSynchronize(s);     // nothing this call enqueued may still use the shared array
        return cuda_fail(e, "select_device scratch set-up");
    }
    prof_begin(s, kProfSelect);
    int rc;
    if (f->max_card <= 255u)
        rc = select_noalloc_ct<uint8_t>(f, d_kfeat, K, size_class, D, d_best, d_pred, d_dev, d_q, d_codes, d_p, d_err, s);
    else if (f->max_card <= 65535u)
        rc = select_noalloc_ct<uint16_t>(f, d_kfeat, K, size_class, D, d_best, d_pred, d_dev, d_q, d_codes, d_p, d_err, s);
    else
        rc = select_noalloc_ct<uint32_t>(f, d_kfeat, K, size_class, D, d_best, d_pred, d_dev, d_q, d_codes, d_p, d_err, s);
    prof_end(s, kProfSelect);
    if (rc != AIWCRF_OK) {
        cudaStreamSynchronize(s);     // kernels enqueued before the failure finish with the array
        return rc;
    }
    uint32_t h_err = 0;
    e = cudaMemcpyAsync(&h_err, d_err, sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "select_device");
    if (h_err & kErrTimeout) return fail(AIWCRF_E_TIMEOUT, "a bounded device wait gave up");
    return AIWCRF_OK;
}

}  // namespace aiwcrf

namespace aiwcrf {
AIWCRF_BOUNDS_READER(bounds_flags_predict)
}  // namespace aiwcrf
