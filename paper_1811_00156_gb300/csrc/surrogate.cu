// surrogate.cu -- a small MLP distilled from the forest's own predictions (not in the paper; the
// paper's model is the forest, Sec. III-B). Inputs: the AIWC columns standardised (log2 first
// for columns spanning orders of magnitude), one-hot device and size class, padded to 64;
// layers 64 -> 256 -> 256 -> 1 with GELU; BF16 weights and activations, FP32 accumulation.
//
// Training (Adam, MSE on the forest's log10-time predictions) runs five kernels per batch: encoding
// with layer 1, layer 2, the backward pass to both pre-activations, the weight gradients (the batch
// as K, split over CTAs), and fixed-order sums with Adam and the BF16 weight copies.
// Inference is one persistent fused kernel: both weight matrices stay in shared memory; for
// every 128 queries the encoded tile is written straight into the MMA operand layout, layer 1
// accumulates into TMEM columns 0..255 and layer 2 into 256..511, and the epilogues apply bias
// and GELU (and the final dot product) from tcgen05.ld registers while the MMAs of the next part run.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "internal.cuh"
#include "tc.cuh"

namespace aiwcrf {

using bf16 = __nv_bfloat16;

constexpr int kIn = 64;
constexpr int kHid = 256;
constexpr int oW1 = 0;
constexpr int ob1 = oW1 + kHid * kIn;
constexpr int oW2 = ob1 + kHid;
constexpr int ob2 = oW2 + kHid * kHid;
constexpr int ow3 = ob2 + kHid;
constexpr int ob3 = ow3 + kHid;
constexpr int kParams = ob3 + 1;

// GELU of the inference epilogues, two values at a time: the packed FP32 instructions halve those
// of the polynomials.
__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ float neg_abs_clamped(float x)      // max(-|x|, -6), NaN stays NaN
{
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(-fabsf(x)), "f"(-6.0f));
    return r;
}

__device__ __forceinline__ float exp2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Layer 1: 0.5 x (1 + erf(x / sqrt 2)) with erf by the rational-exponential approximation of
// Abramowitz & Stegun, Handbook of Mathematical Functions, formula 7.1.26 (absolute error at most
// 1.5e-7 for x >= 0, extended as an odd function): 1 - (a1 t + a2 t^2 + a3 t^3 + a4 t^4 + a5 t^5)
// exp(-x^2), t = 1 / (1 + p x), with the approximate reciprocal and exponential: the absolute error
// stays below 1e-6. Its result is rounded to BF16, where another formula's last bits would move an
// activation by a whole BF16 unit now and then, so the first layer keeps this one.
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ uint64_t gelu2_layer1(uint64_t x)
{
    auto both = [](float c) { return pack2(c, c); };
    float x0, x1, a, b;
    const uint64_t xs = mul2(x, both(0.70710678118654752f));
    unpack2(xs, x0, x1);
    const uint64_t ax = pack2(fabsf(x0), fabsf(x1));
    unpack2(fma2(both(0.3275911f), ax, both(1.0f)), a, b);
    const uint64_t t = pack2(rcp_approx(a), rcp_approx(b));
    uint64_t poly = fma2(both(-1.061405429f), t, both(1.453152027f));      // the polynomial's negative
    poly = fma2(poly, t, both(-1.421413741f));
    poly = fma2(poly, t, both(0.284496736f));
    poly = fma2(poly, t, both(-0.254829592f));
    poly = mul2(poly, t);
    // exp(-ax^2) = 2^(-ax^2 log2 e)
    unpack2(mul2(mul2(ax, ax), both(-1.44269504088896341f)), a, b);
    const uint64_t ex = pack2(exp2_approx(a), exp2_approx(b));
    unpack2(fma2(poly, ex, both(1.0f)), a, b);
    const uint64_t erf = pack2(copysignf(a, x0), copysignf(b, x1));
    return mul2(mul2(both(0.5f), x), add2(both(1.0f), erf));
}

// Layer 2, whose GELU stays in FP32: x Phi(x) = max(x, 0) - |x| Phi(-|x|), and log2 Phi(-t) is so
// smooth on [0, 6] that a degree-8 polynomial q (a weighted minimax fit, here in s = -t) gives
// |2^q - Phi(-t)| <= 7.6e-9; evaluated in FP32 it stays below 4e-8, and the exponential adds at most
// 2^-22 of a value below 1/2 (formula 7.1.26 leaves 7e-8 on the same scale before rounding). Beyond 6,
// Phi(-t) < 1e-9 is taken as Phi(-6), for minus infinity too (GELU's limit there; x times 1 + erf would be
// NaN). One exponential and nine multiply-adds a value. NaN stays NaN.
__device__ __forceinline__ uint64_t gelu2(uint64_t x)
{
    constexpr float kQ[9] = {-1.0f, 1.1511057615280151f, -0.45920491218566895f, 0.052505023777484894f,
                             0.007075459696352482f, 0.00014585882308892906f, -0.0001825532381189987f,
                             -3.8622158172074705e-05f, -2.7721882815967547e-06f};
    float x0, x1;
    unpack2(x, x0, x1);
    const uint64_t s = pack2(neg_abs_clamped(x0), neg_abs_clamped(x1));
    uint64_t q = fma2(pack2(kQ[8], kQ[8]), s, pack2(kQ[7], kQ[7]));
#pragma unroll
    for (int i = 6; i >= 0; --i) q = fma2(q, s, pack2(kQ[i], kQ[i]));
    float q0, q1;
    unpack2(q, q0, q1);
    return fma2(s, pack2(exp2_approx(q0), exp2_approx(q1)), pack2(fmaxf(x0, 0.0f), fmaxf(x1, 0.0f)));
}

// two floats as BF16 (round to nearest even) in one word, the first in the low half
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// Of a row's features a network's inputs: standardised AIWC columns, one-hot device, one-hot size, zeros.
struct Encoder {
    const float *mu, *sd;
    const uint8_t *logf;
    int n_aiwc, n_dev, n_size;
};

// ------------------------------------------------------------------------------------------
// training kernels
// ------------------------------------------------------------------------------------------
// One step (forward, backward, gradient sums) is five kernels. A tile is 128 rows of the batch; its
// BF16 matrices (inputs, activations, pre-activation gradients) live in global memory in the core
// matrix order of the MMA operands, so that the next kernel fetches a tile with bulk copies and reads
// it as it lies: by rows as a K-major operand, or transposed as an MN-major one for the weight
// gradients. What bounds a step at 4,096 rows is latency: 2 GFLOP are a microsecond of the tensor
// cores, and as twenty kernels (a GEMM, its elementwise work and every sum apart) it took 209 us of
// device time and a 4,096-row gradient 223 us; this takes 53 (cold caches) and 77, the launches and
// the wait now about half of it.
// FP32 values per row and column are stored [tile][column][row]: a warp's lanes are 32 rows.
constexpr int kTrainThreads = 512;               // 16 warps: four per TMEM lane quarter, 16 columns each
constexpr int kSlices = 4;                       // CTAs of a tile, 64 of the 256 columns each
constexpr int kSliceCols = kHid / kSlices;
constexpr int kTileX = 128 * kIn * 2, kTileH = 128 * kHid * 2;      // bytes of a tile's matrices
constexpr int kMaxSplits = 64;                   // of the batch's tiles, for the weight gradients

// byte offset of element (row, col) of a 128 x C tile
template <int C>
__host__ __device__ constexpr uint32_t tile_offset(uint32_t row, uint32_t col)
{
    return ((row >> 3) * (uint32_t)(C / 8) + (col >> 3)) * tc::kCoreBytes + (row & 7u) * 16u + (col & 7u) * 2u;
}

struct TrainArgs {
    Encoder e;
    const float *X;              // F x ld inputs
    int64_t ld;
    const uint32_t *perm;        // row order, or null
    int64_t r0;
    const float *yall;
    const int64_t *step;         // when set, the batch starts at row (*step mod spe) * B of the order
    int64_t spe;
    int B;
    const float *P;              // parameters
    const bf16 *W1b, *W2b;
    unsigned char *xt, *ht, *dz2t, *dz1t;        // BF16 tiles: inputs, layer-1 activations, gradients
    float *yb;                   // B targets
    float *g1, *g2, *h2;         // GELU'(z1), GELU'(z2), GELU(z2): [tile][column][row]
    float *dots;                 // B x 32 partial sums of the output dot
    float *db1, *db2, *dw3;      // [tile][column] sums over the tile's rows
    float *dloss;                // [tile][2]: sums of dout and of the loss
    float *w2part, *w1part;      // [split][256][256], [split][256][64]
    int splits;
    uint32_t *err;
};

__device__ __forceinline__ void gelu_both(float x, float &h, float &g)
{
    const float e = erff(x * 0.70710678118654752f);
    h = 0.5f * x * (1.0f + e);
    g = 0.5f * (1.0f + e) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// What the training kernels share: an mbarrier for MMAs and one for copies (or none), an accumulator of
// ncols TMEM columns, and an orderly end when a bounded wait runs out.
__device__ __forceinline__ void train_begin(uint64_t *bar_m, uint64_t *bar_c, uint32_t *tmem_base, uint32_t ncols)
{
    if (threadIdx.x < 32) {
        tc::tmem_alloc(tmem_base, ncols);
        tc::tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        tc::mbar_init(bar_m, 1);
        if (bar_c) tc::mbar_init(bar_c, 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
}

__device__ __forceinline__ void train_end(bool ok, uint32_t tbase, uint32_t ncols, uint32_t *err)
{
    if (!ok && threadIdx.x == 0) atomicOr(err, kErrTimeout);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (threadIdx.x < 32) tc::tmem_dealloc(tbase, ncols);
}

// every thread: the barrier's phase is complete (false for the whole CTA if a wait ran out)
__device__ __forceinline__ bool train_wait(uint64_t *bar, uint32_t phase)
{
    bool ok = __syncthreads_and(tc::mbar_wait(bar, phase));
    if (!ok) tc::mbar_wait(bar, phase);         // once more for what is still in flight, then give up
    tc::fence_after_sync();
    return ok;
}

// rows of a weight matrix stored [n][ld] as a K-major tile of 64 n x K (n of tile row r is row_of(r))
template <int K, typename RowOf>
__device__ __forceinline__ void stage_weights(unsigned char *dst, const bf16 *__restrict__ W, int ld, const RowOf &row_of)
{
    for (int i = threadIdx.x; i < kSliceCols * (K / 8); i += kTrainThreads) {
        const int r = i / (K / 8), k = (i % (K / 8)) * 8;
        *reinterpret_cast<uint4 *>(dst + tile_offset<K>((uint32_t)r, (uint32_t)k)) =
            __ldg(reinterpret_cast<const uint4 *>(W + (size_t)row_of(r) * (size_t)ld + k));
    }
}

// the tile's 128 x 64 accumulator columns [16 group, 16 group + 16) of this thread's row
__device__ __forceinline__ void train_acc(uint32_t tbase, int q4, int group, float (&x)[16])
{
    tc::tmem_ld16(tbase + ((uint32_t)(32 * q4) << 16) + 16u * group, x);
}

// CTA (slice, tile): encode the tile's rows, layer 1's columns [64 slice, ...): activations and GELU'.
__global__ void __launch_bounds__(kTrainThreads) train_layer1_kernel(TrainArgs a)
{
    __shared__ __align__(1024) unsigned char sX[kTileX];
    __shared__ __align__(1024) unsigned char sW[kSliceCols * kIn * 2];
    __shared__ __align__(8) uint64_t bar_m;
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, slice = blockIdx.x % kSlices;
    const int64_t tile = blockIdx.x / kSlices;
    train_begin(&bar_m, nullptr, &tmem_base, 64);
    {   // thread (row, part) encodes inputs [8 part, 8 part + 8) and [32 + 8 part, ...) of one row; the
        // row's values are loaded together before any is used
        const int row = tid & 127, part = tid >> 7;
        const int64_t r0 = a.step ? (*a.step % a.spe) * (int64_t)a.B : a.r0, at = r0 + tile * 128 + row;
        const int64_t src = a.perm ? (int64_t)a.perm[at] : at;
        float x[16], mu[16], sd[16];
        bool lg[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int k = (i < 8 ? 0 : 24) + 8 * part + i;
            x[i] = k < a.e.n_aiwc ? __ldg(&a.X[(size_t)k * (size_t)a.ld + src]) : 0.0f;
            mu[i] = k < a.e.n_aiwc ? __ldg(&a.e.mu[k]) : 0.0f;
            sd[i] = k < a.e.n_aiwc ? __ldg(&a.e.sd[k]) : 1.0f;
            lg[i] = k < a.e.n_aiwc && __ldg(&a.e.logf[k]);
        }
        const float dev = __ldg(&a.X[(size_t)a.e.n_aiwc * (size_t)a.ld + src]);
        const float size = __ldg(&a.X[(size_t)(a.e.n_aiwc + 1) * (size_t)a.ld + src]);
        if (slice == 0 && part == 0) a.yb[tile * 128 + row] = a.yall[src];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int k = (i < 8 ? 0 : 24) + 8 * part + i, d = k - a.e.n_aiwc, z = d - a.e.n_dev;
            if (d < 0) x[i] = ((lg[i] ? log2f(fmaxf(x[i], 1.0f)) : x[i]) - mu[i]) / sd[i];
            else x[i] = z < 0 ? (dev == (float)d ? 1.0f : 0.0f) : z < a.e.n_size && size == (float)z ? 1.0f : 0.0f;
        }
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const uint32_t off = tile_offset<kIn>((uint32_t)row, (uint32_t)(32 * g + 8 * part));
            const float *v = x + 8 * g;
            const uint4 w = make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]),
                                       pack_bf16x2(v[6], v[7]));
            *reinterpret_cast<uint4 *>(sX + off) = w;
            if (slice == 0) *reinterpret_cast<uint4 *>(a.xt + (size_t)tile * kTileX + off) = w;
        }
    }
    stage_weights<kIn>(sW, a.W1b + (size_t)slice * kSliceCols * kIn, kIn, [](int r) { return r; });
    tc::fence_smem_to_async();
    __syncthreads();
    const uint32_t tbase = tmem_base;
    if (tid == 0) {
        tc::fence_after_sync();
        const uint32_t a0 = tc::smem_addr(sX), w0 = tc::smem_addr(sW), idesc = tc::make_idesc_bf16(128, kSliceCols);
#pragma unroll
        for (int s = 0; s < kIn / 16; ++s)
            tc::mma_bf16(tbase, tc::make_desc(a0 + 256u * s, 128u, kIn / 8 * 128u), tc::make_desc(w0 + 256u * s, 128u, kIn / 8 * 128u),
                         idesc, s > 0 ? 1u : 0u);
        tc::mma_commit(&bar_m);
    }
    const bool ok = train_wait(&bar_m, 0u);
    if (ok) {
        const int q4 = warp & 3, group = warp >> 2, row = 32 * q4 + lane, col0 = kSliceCols * slice + 16 * group;
        float x[16], h[16];
        train_acc(tbase, q4, group, x);
        float *g1 = a.g1 + ((size_t)tile * kHid + col0) * 128 + row;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            float g;
            gelu_both(x[i] + __ldg(&a.P[ob1 + col0 + i]), h[i], g);
            g1[(size_t)i * 128] = g;
        }
#pragma unroll
        for (int p = 0; p < 2; ++p)
            *reinterpret_cast<uint4 *>(a.ht + (size_t)tile * kTileH + tile_offset<kHid>((uint32_t)row, (uint32_t)(col0 + 8 * p))) =
                make_uint4(pack_bf16x2(h[8 * p], h[8 * p + 1]), pack_bf16x2(h[8 * p + 2], h[8 * p + 3]),
                           pack_bf16x2(h[8 * p + 4], h[8 * p + 5]), pack_bf16x2(h[8 * p + 6], h[8 * p + 7]));
    }
    train_end(ok, tbase, 64, a.err);
}

// CTA (slice, tile): layer 2's columns n = 32 m + 8 slice + i (m, i < 8), in the order 8 i + m: GELU,
// GELU' and, for each 8 slice + i, the sum over m of GELU(z2) w3: one of the 32 partial sums of the output,
// in a fixed order.
constexpr int kLayer2Smem = kTileH + kSliceCols * kHid * 2;
__global__ void __launch_bounds__(kTrainThreads) train_layer2_kernel(TrainArgs a)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *sH = sm, *sW = sm + kTileH;
    __shared__ __align__(8) uint64_t bar_c, bar_m;
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, slice = blockIdx.x % kSlices;
    const int64_t tile = blockIdx.x / kSlices;
    train_begin(&bar_m, &bar_c, &tmem_base, 64);
    if (tid == 0) {
        tc::mbar_expect(&bar_c, kTileH);
        tc::bulk_load(sH, a.ht + (size_t)tile * kTileH, kTileH, &bar_c);
    }
    stage_weights<kHid>(sW, a.W2b, kHid, [slice](int r) { return 32 * (r & 7) + 8 * slice + (r >> 3); });
    tc::fence_smem_to_async();
    const uint32_t tbase = tmem_base;
    bool ok = train_wait(&bar_c, 0u);
    if (ok) {
        if (tid == 0) {
            const uint32_t a0 = tc::smem_addr(sH), w0 = tc::smem_addr(sW), idesc = tc::make_idesc_bf16(128, kSliceCols);
#pragma unroll
            for (int s = 0; s < kHid / 16; ++s)
                tc::mma_bf16(tbase, tc::make_desc(a0 + 256u * s, 128u, kHid / 8 * 128u),
                             tc::make_desc(w0 + 256u * s, 128u, kHid / 8 * 128u), idesc, s > 0 ? 1u : 0u);
            tc::mma_commit(&bar_m);
        }
        ok = train_wait(&bar_m, 0u);
    }
    if (ok) {
        const int q4 = warp & 3, group = warp >> 2, row = 32 * q4 + lane;
        float x[16];
        train_acc(tbase, q4, group, x);
        float *dots = a.dots + ((size_t)tile * 128 + row) * 32 + 8 * slice + 2 * group;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float dot = 0.0f;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int n = 32 * m + 8 * slice + 2 * group + i;
                float h, g;
                gelu_both(x[8 * i + m] + __ldg(&a.P[ob2 + n]), h, g);
                dot += h * __ldg(&a.P[ow3 + n]);
                const size_t at = ((size_t)tile * kHid + n) * 128 + row;
                a.h2[at] = h;
                a.g2[at] = g;
            }
            dots[i] = dot;
        }
    }
    train_end(ok, tbase, 64, a.err);
}

// sum of a tile column's 128 values v(row), by one warp
template <typename Value>
__device__ __forceinline__ float column_sum(int lane, const Value &v)
{
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) s += v(32 * k + lane);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    return s;
}

// CTA (slice, tile): the outputs and their errors, dz2 = dout w3 GELU'(z2) of the whole tile, and the
// columns k of [64 slice, ...) of dh1 = dz2 W2 and dz1 = dh1 GELU'(z1); sums over the tile's rows of dz2,
// GELU(z2) dout and dz1 for the slice's columns.
constexpr int kBackSmem = kTileH + kSliceCols * kHid * 2;
__global__ void __launch_bounds__(kTrainThreads) train_back_kernel(TrainArgs a)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *sZ = sm, *sW = sm + kTileH;       // dz2 (later dz1's columns in FP32), W2's columns
    __shared__ __align__(8) uint64_t bar_m;
    __shared__ uint32_t tmem_base;
    __shared__ float dout_s[128], w3s[kHid];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, slice = blockIdx.x % kSlices;
    const int64_t tile = blockIdx.x / kSlices;
    train_begin(&bar_m, nullptr, &tmem_base, 64);
    // thread (row, part) computes dz2 of one row's columns [64 part, ...): half of GELU' loaded ahead
    const int zrow = tid & 127, part = tid >> 7;
    const float *g2z = a.g2 + ((size_t)tile * kHid + kSliceCols * part) * 128 + zrow;
    float gz[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) gz[i] = __ldg(&g2z[(size_t)i * 128]);
    if (tid < 128) {
        // the 32 partial sums in the order of a warp's butterfly
        const float4 *d4 = reinterpret_cast<const float4 *>(a.dots + ((size_t)tile * 128 + tid) * 32);
        float s[32];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 v = d4[i];
            s[4 * i] = v.x; s[4 * i + 1] = v.y; s[4 * i + 2] = v.z; s[4 * i + 3] = v.w;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < o; ++i) s[i] += s[i + o];
        const float d = s[0] + a.P[ob3] - a.yb[tile * 128 + tid];
        dout_s[tid] = d / (float)a.B;
        if (slice == 0) {
            float sd = d / (float)a.B, sl = 0.5f * d * d;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                sd += __shfl_xor_sync(kFull, sd, o);
                sl += __shfl_xor_sync(kFull, sl, o);
            }
            if (lane == 0) { a.dloss[8 * tile + 2 * warp] = sd; a.dloss[8 * tile + 2 * warp + 1] = sl; }
        }
    } else if (tid - 128 < kHid) {
        w3s[tid - 128] = a.P[ow3 + tid - 128];
    }
    // W2[n][64 slice + c] with K = n: 16 bytes are 8 columns of one n
    for (int i = tid; i < kHid * (kSliceCols / 8); i += kTrainThreads) {
        const int n = i / (kSliceCols / 8), c = (i % (kSliceCols / 8)) * 8;
        *reinterpret_cast<uint4 *>(sW + tile_offset<kSliceCols>((uint32_t)n, (uint32_t)c)) =
            __ldg(reinterpret_cast<const uint4 *>(a.W2b + (size_t)n * kHid + kSliceCols * slice + c));
    }
    __syncthreads();
    {
        const float dout = dout_s[zrow];
#pragma unroll
        for (int c = 0; c < kSliceCols; c += 8) {
            float d[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                d[i] = dout * w3s[kSliceCols * part + c + i] * gz[(c + i) & 31];
                if (c < 32) gz[c + i] = __ldg(&g2z[(size_t)(32 + c + i) * 128]);
            }
            const uint4 v = make_uint4(pack_bf16x2(d[0], d[1]), pack_bf16x2(d[2], d[3]), pack_bf16x2(d[4], d[5]),
                                       pack_bf16x2(d[6], d[7]));
            const uint32_t off = tile_offset<kHid>((uint32_t)zrow, (uint32_t)(kSliceCols * part + c));
            *reinterpret_cast<uint4 *>(sZ + off) = v;
            if (part == slice) *reinterpret_cast<uint4 *>(a.dz2t + (size_t)tile * kTileH + off) = v;
        }
    }
    tc::fence_smem_to_async();
    __syncthreads();
    const uint32_t tbase = tmem_base;
    if (tid == 0) {
        tc::fence_after_sync();
        const uint32_t a0 = tc::smem_addr(sZ), w0 = tc::smem_addr(sW), idesc = tc::make_idesc_bf16(128, kSliceCols, false, true);
#pragma unroll
        for (int s = 0; s < kHid / 16; ++s)
            tc::mma_bf16(tbase, tc::make_desc(a0 + 256u * s, 128u, kHid / 8 * 128u),
                         tc::make_desc(w0 + 2u * (kSliceCols / 8 * 128u) * s, kSliceCols / 8 * 128u, 128u), idesc, s > 0 ? 1u : 0u);
        tc::mma_commit(&bar_m);
    }
    const int q4 = warp & 3, group = warp >> 2, row = 32 * q4 + lane, col0 = kSliceCols * slice + 16 * group;
    const float *g1 = a.g1 + ((size_t)tile * kHid + col0) * 128 + row;
    float x1[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x1[i] = __ldg(&g1[(size_t)i * 128]);
    // the slice's sums of dz2 and GELU(z2) dout, under the MMAs
#pragma unroll
    for (int u = 0; u < kSliceCols / (kTrainThreads / 32); ++u) {
        const int n = kSliceCols * slice + warp + u * (kTrainThreads / 32);
        const float *g2 = a.g2 + ((size_t)tile * kHid + n) * 128, *h2 = a.h2 + ((size_t)tile * kHid + n) * 128;
        const float s2 = column_sum(lane, [&](int b) { return dout_s[b] * w3s[n] * __ldg(&g2[b]); });
        const float s3 = column_sum(lane, [&](int b) { return __ldg(&h2[b]) * dout_s[b]; });
        if (lane == 0) { a.db2[tile * kHid + n] = s2; a.dw3[tile * kHid + n] = s3; }
    }
    const bool ok = train_wait(&bar_m, 0u);
    if (ok) {
        float *f = reinterpret_cast<float *>(sZ);    // [column of the slice][row]; the MMAs have read dz2
        float x[16];
        train_acc(tbase, q4, group, x);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            x[i] *= x1[i];
            f[(16 * group + i) * 128 + row] = x[i];
        }
#pragma unroll
        for (int p = 0; p < 2; ++p)
            *reinterpret_cast<uint4 *>(a.dz1t + (size_t)tile * kTileH + tile_offset<kHid>((uint32_t)row, (uint32_t)(col0 + 8 * p))) =
                make_uint4(pack_bf16x2(x[8 * p], x[8 * p + 1]), pack_bf16x2(x[8 * p + 2], x[8 * p + 3]),
                           pack_bf16x2(x[8 * p + 4], x[8 * p + 5]), pack_bf16x2(x[8 * p + 6], x[8 * p + 7]));
        __syncthreads();
        for (int c = warp; c < kSliceCols; c += kTrainThreads / 32) {
            const float s1 = column_sum(lane, [&](int row2) { return f[c * 128 + row2]; });
            if (lane == 0) a.db1[tile * kHid + kSliceCols * slice + c] = s1;
        }
    }
    train_end(ok, tbase, 64, a.err);
}

// CTA (half, split): rows [128 half, ...) of dW2 = dz2^T h1 and dW1 = dz1^T x over the split's tiles. Both
// operands are read transposed: a tile's rows are the MMA's K.
constexpr int kWgradSmem = kTileH / 2 + kTileH + kTileH / 2 + kTileX;
__global__ void __launch_bounds__(kTrainThreads) train_wgrad_kernel(TrainArgs a, int64_t *advance)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *sZ2 = sm, *sH = sZ2 + kTileH / 2, *sZ1 = sH + kTileH, *sX = sZ1 + kTileH / 2;
    __shared__ __align__(8) uint64_t bar_c, bar_m;
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, half = blockIdx.x, split = blockIdx.y;
    train_begin(&bar_m, &bar_c, &tmem_base, 512);
    const uint32_t tbase = tmem_base;
    if (advance && tid == 0 && half == 0 && split == 0) *advance += 1;     // nobody reads it in this kernel
    const int tiles = a.B / 128, per = (tiles + a.splits - 1) / a.splits;
    const int t0 = split * per, t1 = min(tiles, t0 + per);
    bool ok = true;
    uint32_t phase = 0;
    constexpr uint32_t kRowBlock = kHid / 8 * 128u, kHalfBlock = kRowBlock / 2;    // 8 rows of a tile, of half its columns
    for (int t = t0; t < t1 && ok; ++t) {
        if (tid == 0) {
            tc::mbar_expect(&bar_c, kWgradSmem);
            tc::bulk_load(sH, a.ht + (size_t)t * kTileH, kTileH, &bar_c);
            tc::bulk_load(sX, a.xt + (size_t)t * kTileX, kTileX, &bar_c);
            for (uint32_t b = 0; b < 16; ++b) {
                const size_t src = (size_t)t * kTileH + b * kRowBlock + half * kHalfBlock;
                tc::bulk_load(sZ2 + b * kHalfBlock, a.dz2t + src, kHalfBlock, &bar_c);
                tc::bulk_load(sZ1 + b * kHalfBlock, a.dz1t + src, kHalfBlock, &bar_c);
            }
        }
        ok = train_wait(&bar_c, phase);
        if (!ok) break;
        if (tid == 0) {
            const uint32_t z2 = tc::smem_addr(sZ2), h = tc::smem_addr(sH), z1 = tc::smem_addr(sZ1), x = tc::smem_addr(sX);
            const uint32_t id2 = tc::make_idesc_bf16(128, kHid, true, true), id1 = tc::make_idesc_bf16(128, kIn, true, true);
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                const uint32_t acc = t > t0 || s > 0 ? 1u : 0u;
                tc::mma_bf16(tbase, tc::make_desc(z2 + 2u * kHalfBlock * s, kHalfBlock, 128u),
                             tc::make_desc(h + 2u * kRowBlock * s, kRowBlock, 128u), id2, acc);
                tc::mma_bf16(tbase + kHid, tc::make_desc(z1 + 2u * kHalfBlock * s, kHalfBlock, 128u),
                             tc::make_desc(x + 2u * (kIn / 8 * 128u) * s, kIn / 8 * 128u, 128u), id1, acc);
            }
            tc::mma_commit(&bar_m);
        }
        ok = train_wait(&bar_m, phase);
        phase ^= 1u;
    }
    if (ok) {
        // 320 accumulator columns in 20 groups of 16, five a warp of a lane quarter
        const int q4 = warp & 3, n = 128 * half + 32 * q4 + lane;
        for (int g = warp >> 2; g < (kHid + kIn) / 16; g += 4) {
            float x[16];
            train_acc(tbase, q4, g, x);
            float *dst = g < kHid / 16 ? a.w2part + ((size_t)split * kHid + n) * kHid + 16 * g
                                       : a.w1part + ((size_t)split * kHid + n) * kIn + 16 * (g - kHid / 16);
#pragma unroll
            for (int i = 0; i < 16; i += 4) *reinterpret_cast<float4 *>(dst + i) = make_float4(x[i], x[i + 1], x[i + 2], x[i + 3]);
        }
    }
    train_end(ok, tbase, 512, a.err);
}

// Adam of one training step: the moments and, for steps counted on the device, the bias corrections
// c12[2 * step], c12[2 * step + 1] (the counter has been advanced).
struct AdamArgs {
    float *p, *m, *v;            // p null: gradients only
    bf16 *W1b, *W2b;             // BF16 copies of the weights
    float lr, beta1, beta2, eps;
    const float *c12;
    const int64_t *step;
};

// The gradient of every parameter: the splits' or tiles' sums in order; then Adam, if asked for.
constexpr int kReduceThreads = 128;
__global__ void __launch_bounds__(kReduceThreads) train_reduce_kernel(TrainArgs a, float *grad, float *loss, AdamArgs ad)
{
    const int i = blockIdx.x * kReduceThreads + threadIdx.x, tiles = a.B / 128;
    if (i > kParams) return;
    float s = 0.0f;
    auto add = [&](const float *p, size_t stride, int n) {
#pragma unroll 8
        for (int k = 0; k < n; ++k) s += __ldg(p + (size_t)k * stride);
    };
    if (i < ob1) add(a.w1part + i, (size_t)kHid * kIn, a.splits);
    else if (i < oW2) add(a.db1 + (i - ob1), kHid, tiles);
    else if (i < ob2) add(a.w2part + (i - oW2), (size_t)kHid * kHid, a.splits);
    else if (i < ow3) add(a.db2 + (i - ob2), kHid, tiles);
    else if (i < ob3) add(a.dw3 + (i - ow3), kHid, tiles);
    else add(a.dloss + (i - ob3), 2, 4 * tiles);
    if (i == kParams) { *loss = s; return; }
    grad[i] = s;
    if (!ad.p) return;
    const int64_t st = *ad.step - 1;
    const float c1 = ad.c12[2 * st], c2 = ad.c12[2 * st + 1];
    const float mi = ad.beta1 * ad.m[i] + (1.0f - ad.beta1) * s;
    const float vi = ad.beta2 * ad.v[i] + (1.0f - ad.beta2) * s * s;
    ad.m[i] = mi;
    ad.v[i] = vi;
    const float p = ad.p[i] - ad.lr * (mi / c1) / (sqrtf(vi / c2) + ad.eps);
    ad.p[i] = p;
    if (i < ob1) ad.W1b[i] = __float2bfloat16_rn(p);
    else if (i >= oW2 && i < ob2) ad.W2b[i - oW2] = __float2bfloat16_rn(p);
}

__global__ void to_bf16_kernel(const float *__restrict__ src, bf16 *__restrict__ dst, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = __float2bfloat16_rn(src[i]);
}

// ------------------------------------------------------------------------------------------
// fused inference
// ------------------------------------------------------------------------------------------

// One tile is 128 queries. What bounds the kernel is the epilogues' arithmetic (65,536 GELUs a tile,
// the FP32 pipe first; the MMAs take about 2,600 clocks), so everything else runs beside it on warps
// of its own, and the sixteen epilogue warps hardly wait for each other:
//  - layer 1 accumulates in TMEM columns 0..255 and layer 2 in 256..511;
//  - epilogue 1 goes through the first layer's columns in four chunks of 64. A warp puts its BF16
//    activations back over the columns it read, where layer 2 takes them as the A operand straight
//    from TMEM (through shared memory, the stores and the proxy fence of a chunk took 400 clocks);
//  - the warps hand a chunk over by arriving on an mbarrier and go on; one warp waits for the
//    arrivals and issues the chunk's part of layer 2 (one K chunk), which runs under the next chunk.
//    (An epilogue warp that also issued them fell behind and held up the others.)
//  - four warps, that one among them, encode the next tile while this one is in its epilogues (in
//    the epilogue warps that took 2,500 clocks of a tile), 32 rows each, so that its layer 1 runs
//    under this tile's epilogue 2. The raw features of the tile after that are copied to shared
//    memory meanwhile, every lane its own.
// Twenty warps leave 96 registers a thread.
// Why nothing is overwritten early: a warp reaches chunk c of the next tile only after bar_h of this
// one, which every warp's arrivals of this tile precede, and the next layer 1 is issued after it.
// Shared memory holds W1 (32 KB), W2 (128), the input tile (16) and its raw features (32).
// Measured at 1,000,000 queries (32 features): 980 us with every part of a
// tile after the other and eight instructions more a GELU, 420 us now = 390 TFLOP/s of the MMAs. With
// TMEM loads started a chunk ahead and approximate quotients it was 409, a tile's clocks then 5,200 of
// epilogue 1, 4,300 of epilogue 2 (6,400 together at the FP32 pipe's rate) and about 2,500 of waiting for
// the slowest warp and the last chunk.
constexpr int kInferWarps = 16;                                // epilogue warps
constexpr int kEncodeWarps = 4;                                // the first of them issues the MMAs
constexpr int kInferThreads = 32 * (kInferWarps + kEncodeWarps);
constexpr int kInferColGroups = kInferWarps / 4;               // warps sharing one TMEM lane quarter
constexpr int kInferCols = 256 / kInferColGroups;              // layer-2 columns per warp
constexpr int kInferSmem = 32768 + 4 * 32768 + 16384 + kIn * 128 * 4;

// The transforms of the AIWC columns, with ones that change nothing past them. Eight columns are encoded at
// once; flags: bit i, column i is taken the logarithm of; bit 8, see standardise8.
struct EncodeColumns {
    alignas(16) float neg_mu[kIn], neg_sd[kIn], rcp_sd[kIn];
    uint32_t flags[kIn / 8];
};
constexpr uint32_t kDivide = 1u << 8;

// What standardise8's quotients hold for: deviations and non-zero dividends in [2^-50, 2^50], so that nothing
// on the way is subnormal or infinite.
constexpr uint32_t kQuotientLo = (127u - 50u) << 24, kQuotientHi = (127u + 50u) << 24;    // of the bits without the sign

// The standardised values of eight AIWC columns, the quotients rounded to nearest as a division rounds them:
// a product with the column's reciprocal is within 1.5 units of the last place; a first residual brings it
// within one, and from there the second one's sum rounds to the quotient's nearest (P. Markstein,
// Computation of elementary functions on the IBM RISC System/6000 processor, 1990: with a correctly rounded
// reciprocal). Values out of range (subnormal, very large, no numbers) are divided. The eight chains run side
// by side: with a division each a call of 1,000,000 queries took 557 us, this takes 423, and one residual of an
// approximate reciprocal, which is neither rounded right nor finite for every deviation, 409. (13e9 pairs of
// dividends and deviations, in and out of range, gave the division's bits.)
__device__ __forceinline__ void standardise8(const EncodeColumns &c, int k0, const float *raw, float (&v)[8])
{
    const uint32_t flags = c.flags[k0 >> 3];
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
    uint64_t a[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float x[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            x[j] = raw[(2 * i + j) * 128];
            const float lg = log2f(fmaxf(x[j], 1.0f));
            x[j] = flags & (1u << (2 * i + j)) ? lg : x[j];
        }
        a[i] = add2(pack2(x[0], x[1]), *reinterpret_cast<const uint64_t *>(c.neg_mu + k0 + 2 * i));
        unpack2(a[i], x[0], x[1]);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const uint32_t e = __float_as_uint(x[j]) << 1;
            lo = min(lo, e - 1u);               // zero is in range
            hi = max(hi, e);
        }
        const uint64_t s = *reinterpret_cast<const uint64_t *>(c.neg_sd + k0 + 2 * i);
        const uint64_t r = *reinterpret_cast<const uint64_t *>(c.rcp_sd + k0 + 2 * i);
        const uint64_t q = mul2(a[i], r), q1 = fma2(fma2(q, s, a[i]), r, q);
        unpack2(fma2(fma2(q1, s, a[i]), r, q1), v[2 * i], v[2 * i + 1]);
    }
    if (lo < kQuotientLo - 1u || hi > kQuotientHi || (flags & kDivide)) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            unpack2(a[i], v[2 * i], v[2 * i + 1]);
            v[2 * i] /= -c.neg_sd[k0 + 2 * i];
            v[2 * i + 1] /= -c.neg_sd[k0 + 2 * i + 1];
        }
    }
}

// the input that a one-hot column's value v sets (first + v for v = 0..n-1), or -1
__device__ __forceinline__ int hot_input(float v, int first, int n)
{
    const int i = (int)v;
    return (float)i == v && i >= 0 && i < n ? first + i : -1;
}

// A part of a tile that a warp encodes at once is 32 rows x 8 inputs from k0 on, one row a lane; the
// 8 inputs are AIWC columns, one-hot inputs or both. copy_part starts the copies of the lane's raw
// values to raw[k0 + i][row], encode_part computes the inputs from them.
__device__ __forceinline__ void copy_part(const Encoder &e, const float *__restrict__ X, int64_t Q, int64_t q, int row, int k0,
                                          float *raw)
{
    if (q >= Q) return;
    const float *src = X + (size_t)k0 * (size_t)Q + q;
    uint32_t dst = tc::smem_addr(raw + k0 * 128 + row);
#pragma unroll
    for (int i = 0; i < 8; ++i, src += Q, dst += 512u)
        if (k0 + i < e.n_aiwc)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void encode_part(const Encoder &e, const EncodeColumns &col, const float *raw, float dev,
                                            float size, bool valid, int row, int k0, unsigned char *sX)
{
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    if (k0 < e.n_aiwc) {
        float v[8];
        standardise8(col, k0, raw + k0 * 128 + row, v);
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = k0 + i < e.n_aiwc && valid ? v[i] : 0.0f;
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = pack_bf16x2(v[2 * i], v[2 * i + 1]);
    }
    if (k0 + 8 > e.n_aiwc) {                    // the device's and the size's 1 where it falls here
        const uint32_t d = (uint32_t)(hot_input(dev, e.n_aiwc, e.n_dev) - k0);
        const uint32_t z = (uint32_t)(hot_input(size, e.n_aiwc + e.n_dev, e.n_size) - k0);
        const uint32_t dv = d & 1u ? 0x3F800000u : 0x3F80u, zv = z & 1u ? 0x3F800000u : 0x3F80u;      // BF16 1
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] |= (d >> 1 == (uint32_t)i ? dv : 0u) | (z >> 1 == (uint32_t)i ? zv : 0u);
    }
    *reinterpret_cast<uint4 *>(sX + tc::core_offset((uint32_t)row, (uint32_t)k0)) = make_uint4(w[0], w[1], w[2], w[3]);
}

__global__ void __launch_bounds__(kInferThreads, 1) surrogate_infer_kernel(
    Encoder e, const float *__restrict__ Xq, int64_t Q, const bf16 *__restrict__ W1b, const bf16 *__restrict__ W2b,
    const float *__restrict__ b1, const float *__restrict__ b2, const float *__restrict__ w3, const float *__restrict__ b3,
    float *__restrict__ out, uint32_t *err)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *sW1 = sm;                        // 256 x 64
    unsigned char *sW2 = sm + 32768;                // 4 chunks of 256 x 64
    unsigned char *sX = sm + 32768 + 4 * 32768;     // 128 x 64: the input tile
    float *raw = reinterpret_cast<float *>(sX + 16384);     // [input][row]
    __shared__ __align__(8) uint64_t full_x, full_h[4];     // operands written (one arrival a warp)
    __shared__ __align__(8) uint64_t bar_x, bar_h;          // MMAs done: layer 1, layer 2
    __shared__ __align__(16) float b1s[kHid], b2s[kHid], w3s[kHid];
    __shared__ EncodeColumns col;
    __shared__ float part[kInferColGroups][128];            // the output dot's partial sums
    __shared__ uint32_t tmem_base;
    __shared__ volatile int gave_up;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t ntiles = (Q + 127) / 128;

    // weights, once per CTA, in the operand layout
    for (int i = tid; i < 256 * 8; i += kInferThreads) {
        const int n = i >> 3, kk = (i & 7) * 8;
        *reinterpret_cast<uint4 *>(sW1 + tc::core_offset(n, kk)) =
            __ldg(reinterpret_cast<const uint4 *>(W1b + (size_t)n * kIn + kk));
    }
    for (int i = tid; i < 4 * 256 * 8; i += kInferThreads) {
        const int kc = i / (256 * 8), rr = i % (256 * 8);
        const int n = rr >> 3, kk = (rr & 7) * 8;
        *reinterpret_cast<uint4 *>(sW2 + kc * 32768 + tc::core_offset(n, kk)) =
            __ldg(reinterpret_cast<const uint4 *>(W2b + (size_t)n * kHid + kc * 64 + kk));
    }
    for (int j = tid; j < kHid; j += kInferThreads) { b1s[j] = __ldg(&b1[j]); b2s[j] = __ldg(&b2[j]); w3s[j] = __ldg(&w3[j]); }
    if (tid < kIn / 8) {
        uint32_t flags = 0u;
        for (int k = 8 * tid; k < 8 * tid + 8; ++k) {
            const float sd = k < e.n_aiwc ? e.sd[k] : 1.0f;
            const uint32_t b = __float_as_uint(sd) << 1;
            col.neg_mu[k] = k < e.n_aiwc ? -e.mu[k] : 0.0f;
            col.neg_sd[k] = -sd;
            col.rcp_sd[k] = 1.0f / sd;
            flags |= (k < e.n_aiwc && e.logf[k] ? 1u << (k & 7) : 0u) | (b < kQuotientLo || b > kQuotientHi ? kDivide : 0u);
        }
        col.flags[tid] = flags;
    }
    for (int i = 128 * e.n_aiwc + tid; i < 128 * ((e.n_aiwc + 7) & ~7); i += kInferThreads) raw[i] = 0.0f;
    if (warp == kInferWarps) {
        tc::tmem_alloc(&tmem_base, 512);
        tc::tmem_relinquish();
    }
    if (tid == 0) {
        tc::mbar_init(&full_x, kEncodeWarps);
        for (int c = 0; c < 4; ++c) tc::mbar_init(&full_h[c], kInferWarps);
        tc::mbar_init(&bar_x, 1);
        tc::mbar_init(&bar_h, 1);
        gave_up = 0;
    }
    tc::fence_before_sync();
    tc::fence_smem_to_async();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = tmem_base;
    auto wait = [&](uint64_t *bar, uint32_t parity) {     // once a wait has run out, none waits again
        if (!gave_up && !tc::mbar_wait(bar, parity)) gave_up = 1;
        tc::fence_after_sync();
    };
    auto arrive = [&](uint64_t *bar) {
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(bar);
    };

    if (warp >= kInferWarps) {
        const int row = 32 * (warp - kInferWarps) + lane;
        float dev, size;
        auto fetch = [&](int64_t tile) {                   // the row's raw values of a tile
            const int64_t q = tile * 128 + row;
#pragma unroll 1
            for (int k0 = 0; k0 < e.n_aiwc; k0 += 8) copy_part(e, Xq, Q, q, row, k0, raw);
            dev = q < Q ? __ldg(&Xq[(size_t)e.n_aiwc * (size_t)Q + q]) : -1.0f;
            size = q < Q ? __ldg(&Xq[(size_t)(e.n_aiwc + 1) * (size_t)Q + q]) : -1.0f;
        };
        auto encode = [&](int64_t tile, int k_from, int k_to) {
#pragma unroll 1
            for (int k0 = k_from; k0 < k_to; k0 += 8) encode_part(e, col, raw, dev, size, tile * 128 + row < Q, row, k0, sX);
        };
        auto hand_over_tile = [&]() {
            tc::fence_smem_to_async();
            arrive(&full_x);
        };
        fetch(blockIdx.x);
        asm volatile("cp.async.wait_all;" ::: "memory");
        encode(blockIdx.x, 0, kIn);
        hand_over_tile();
        if ((int64_t)blockIdx.x + gridDim.x < ntiles) fetch((int64_t)blockIdx.x + gridDim.x);
        const uint32_t idesc = tc::make_idesc_bf16(128, 256);
        const uint32_t a0 = tc::smem_addr(sX), w1 = tc::smem_addr(sW1), w2 = tc::smem_addr(sW2);
        auto issue_chunk = [&](int c, uint32_t parity) {
            wait(&full_h[c], parity);
            if (lane == 0 && !gave_up) {
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    tc::mma_bf16_ta(tbase + 256u, tbase + 64u * c + 16u * s,
                                    tc::make_desc(w2 + 32768u * c + 256u * s, tc::kLbo, tc::kSbo), idesc,
                                    c > 0 || s > 0 ? 1u : 0u);
                if (c == 3) tc::mma_commit(&bar_h);
            }
            __syncwarp();
        };
        uint32_t n = 0;                                    // the CTA's tiles in turn
        for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++n) {
            const int64_t next = tile + gridDim.x;
            const bool more = next < ntiles;
            if (warp == kInferWarps) {
                wait(&full_x, n & 1u);
                if (n) wait(&bar_h, (n - 1u) & 1u);        // the activations have been read
                if (lane == 0 && !gave_up) {
#pragma unroll
                    for (int s = 0; s < 4; ++s)
                        tc::mma_bf16(tbase, tc::make_desc(a0 + 256u * s, tc::kLbo, tc::kSbo),
                                     tc::make_desc(w1 + 256u * s, tc::kLbo, tc::kSbo), idesc, s > 0 ? 1u : 0u);
                    tc::mma_commit(&bar_x);
                }
                __syncwarp();
            }
            if (more) {
                asm volatile("cp.async.wait_all;" ::: "memory");
                wait(&bar_x, n & 1u);                      // layer 1 has read the input tile
            }
            if (warp != kInferWarps) {
                if (more) encode(next, 0, kIn);
            } else {                                       // between the chunks, which come at their own pace
                if (more) encode(next, 0, 24);
                issue_chunk(0, n & 1u);
                if (more) encode(next, 24, kIn);
                issue_chunk(1, n & 1u);
                issue_chunk(2, n & 1u);
                issue_chunk(3, n & 1u);
            }
            if (more) {
                hand_over_tile();
                if (next + gridDim.x < ntiles) fetch(next + gridDim.x);
            }
        }
        if (gave_up && warp == kInferWarps && lane == 0) {   // MMAs may still be running: a bounded wait
            tc::mma_commit(&bar_h);                          // for them before their TMEM goes
            for (uint32_t k = 0; k < 2u; ++k) tc::mbar_wait(&bar_h, k);
        }
        __syncwarp();
    } else {
        const int q4 = warp & 3, group = warp >> 2;         // TMEM lane quarter, column group
        const int r = 32 * q4 + lane;
        const uint32_t mine = tbase + ((uint32_t)(32 * q4) << 16);
        uint32_t parity = 0;
        for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, parity ^= 1u) {
            const int64_t q0 = tile * 128;
            wait(&bar_x, parity);
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {   // epilogue 1: bias, GELU, BF16 back into TMEM
                const uint32_t col0 = 64u * c + 16u * group;
                const float4 *bias = reinterpret_cast<const float4 *>(b1s + col0);
                uint32_t w[8];
                float x[16];
                tc::tmem_ld16(mine + col0, x);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 b = bias[i];
                    float h0, h1;
                    unpack2(gelu2_layer1(add2(pack2(x[4 * i], x[4 * i + 1]), pack2(b.x, b.y))), h0, h1);
                    w[2 * i] = pack_bf16x2(h0, h1);
                    unpack2(gelu2_layer1(add2(pack2(x[4 * i + 2], x[4 * i + 3]), pack2(b.z, b.w))), h0, h1);
                    w[2 * i + 1] = pack_bf16x2(h0, h1);
                }
                tc::tmem_st8(mine + col0, w);
                arrive(&full_h[c]);
            }
            wait(&bar_h, parity);
            uint64_t dot = pack2(0.0f, 0.0f);
#pragma unroll 1
            for (int c = 0; c < kInferCols / 16; ++c) {     // epilogue 2: bias, GELU, dot with w3
                const int col0 = kInferCols * group + 16 * c;
                const float4 *bias = reinterpret_cast<const float4 *>(b2s + col0);
                const float4 *wt = reinterpret_cast<const float4 *>(w3s + col0);
                float x[16];
                tc::tmem_ld16(mine + 256u + (uint32_t)col0, x);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 b = bias[i], w = wt[i];
                    dot = fma2(gelu2(add2(pack2(x[4 * i], x[4 * i + 1]), pack2(b.x, b.y))), pack2(w.x, w.y), dot);
                    dot = fma2(gelu2(add2(pack2(x[4 * i + 2], x[4 * i + 3]), pack2(b.z, b.w))), pack2(w.z, w.w), dot);
                }
            }
            tc::fence_before_sync();
            float d0, d1;
            unpack2(dot, d0, d1);
            part[group][r] = d0 + d1;
            asm volatile("bar.sync %0, 128;" ::"r"(1 + q4) : "memory");   // the quarter's four warps
            if (group == 0 && q0 + r < Q) {
                float o = __ldg(&b3[0]);
#pragma unroll
                for (int g = 0; g < kInferColGroups; ++g) o += part[g][r];
                out[q0 + r] = o;
            }
        }
    }
    if (gave_up && tid == 0) atomicOr(err, kErrTimeout);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == kInferWarps) tc::tmem_dealloc(tbase, 512);
}

}  // namespace aiwcrf

// ------------------------------------------------------------------------------------------
// the surrogate object and the C ABI
// ------------------------------------------------------------------------------------------
struct aiwcrf_surrogate {
    int device = 0;
    int32_t F = 0, n_aiwc = 0, n_dev = 0, n_size = 0;
    void *d_block = nullptr;
    float *d_param = nullptr, *d_mu = nullptr, *d_sd = nullptr;
    uint8_t *d_logf = nullptr;
    aiwcrf::bf16 *d_W1b = nullptr, *d_W2b = nullptr;
    std::vector<float> mu, sd;
    std::vector<uint8_t> logf;
    aiwcrf_surrogate_fit_stats stats = {};
};

namespace aiwcrf {
namespace {

// work reading the network may still be in flight on any stream: wait for it, then give the
// block back to the pool (stream-ordered, no device-wide wait inside the free)
void surrogate_release(aiwcrf_surrogate *s)
{
    if (!s) return;
    cudaDeviceSynchronize();
    if (s->d_block) cudaFreeAsync(s->d_block, cudaStreamPerThread);
    cudaStreamSynchronize(cudaStreamPerThread);
    delete s;
}

size_t surrogate_block_bytes(int32_t n_aiwc)
{
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    return up(4 * (size_t)kParams) + 2 * up(4 * (size_t)n_aiwc) + up((size_t)n_aiwc) + up(2 * (size_t)kHid * kIn) +
           up(2 * (size_t)kHid * kHid);
}

int surrogate_alloc(aiwcrf_surrogate *s)
{
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t bp = up(4 * (size_t)kParams), bf = up(4 * (size_t)s->n_aiwc), bl = up((size_t)s->n_aiwc);
    const size_t bw1 = up(2 * (size_t)kHid * kIn);
    // from the stream-ordered pool, whose frees never wait for the whole device (a
    // selection server may be busy on other streams)
    int dev = 0;
    cudaGetDevice(&dev);
    keep_pool_memory(dev);
    void *p = nullptr;
    cudaError_t e = cudaMallocAsync(&p, surrogate_block_bytes(s->n_aiwc), cudaStreamPerThread);
    if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamPerThread);
    if (e != cudaSuccess) return fail(AIWCRF_E_OOM, "surrogate allocation");
    unsigned char *c = static_cast<unsigned char *>(p);
    s->d_block = p;
    s->d_param = reinterpret_cast<float *>(c);
    s->d_mu = reinterpret_cast<float *>(c + bp);
    s->d_sd = reinterpret_cast<float *>(c + bp + bf);
    s->d_logf = c + bp + 2 * bf;
    s->d_W1b = reinterpret_cast<bf16 *>(c + bp + 2 * bf + bl);
    s->d_W2b = reinterpret_cast<bf16 *>(c + bp + 2 * bf + bl + bw1);
    return AIWCRF_OK;
}

Encoder encoder_of(const aiwcrf_surrogate *s)
{
    Encoder e;
    e.mu = s->d_mu; e.sd = s->d_sd; e.logf = s->d_logf;
    e.n_aiwc = s->n_aiwc; e.n_dev = s->n_dev; e.n_size = s->n_size;
    return e;
}

int refresh_bf16(aiwcrf_surrogate *s, cudaStream_t st)
{
    to_bf16_kernel<<<(kHid * kIn + 255) / 256, 256, 0, st>>>(s->d_param + oW1, s->d_W1b, kHid * kIn);
    to_bf16_kernel<<<(kHid * kHid + 255) / 256, 256, 0, st>>>(s->d_param + oW2, s->d_W2b, kHid * kHid);
    count_launches(2);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? AIWCRF_OK : cuda_fail(e, "bf16 weight copies");
}

// scratch of one training batch: the arrays of TrainArgs, gradients, Adam's moments
struct Batch {
    TrainArgs a = {};
    float *grad = nullptr, *m = nullptr, *v = nullptr, *loss = nullptr;
    uint32_t *err = nullptr;
    void *block = nullptr;
    cudaStream_t s = nullptr;
    ~Batch() { if (block) cudaFreeAsync(block, s); }
    int alloc(int B, bool adam, cudaStream_t st)
    {
        s = st;
        const size_t tiles = (size_t)B / 128, BH4 = 4 * (size_t)B * kHid;
        a.B = B;
        a.splits = (int)std::min<size_t>(tiles, kMaxSplits);
        const int per = ((int)tiles + a.splits - 1) / a.splits;
        a.splits = ((int)tiles + per - 1) / per;                     // none is empty
        struct Part { void **p; size_t bytes; };
        const size_t mv = adam ? 4 * (size_t)kParams : 0;
        const Part parts[] = {
            {(void **)&err, 4}, {(void **)&m, mv}, {(void **)&v, mv},                       // cleared below
            {(void **)&a.xt, tiles * kTileX}, {(void **)&a.ht, tiles * kTileH}, {(void **)&a.dz2t, tiles * kTileH},
            {(void **)&a.dz1t, tiles * kTileH}, {(void **)&a.yb, 4 * (size_t)B}, {(void **)&a.g1, BH4}, {(void **)&a.g2, BH4},
            {(void **)&a.h2, BH4}, {(void **)&a.dots, 4 * (size_t)B * 32}, {(void **)&a.db1, 4 * tiles * kHid},
            {(void **)&a.db2, 4 * tiles * kHid}, {(void **)&a.dw3, 4 * tiles * kHid}, {(void **)&a.dloss, 4 * tiles * 8},
            {(void **)&a.w2part, 4 * (size_t)a.splits * kHid * kHid}, {(void **)&a.w1part, 4 * (size_t)a.splits * kHid * kIn},
            {(void **)&grad, 4 * (size_t)kParams}, {(void **)&loss, 4}};
        auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
        size_t tot = 0;
        for (const Part &p : parts) tot += up(p.bytes);
        if (cudaMallocAsync(&block, tot, st) != cudaSuccess) return fail(AIWCRF_E_OOM, "surrogate batch scratch");
        unsigned char *c = static_cast<unsigned char *>(block);
        for (const Part &p : parts) { *p.p = c; c += up(p.bytes); }
        a.err = err;
        cudaMemsetAsync(block, 0, up(4) + 2 * up(mv), st);
        return AIWCRF_OK;
    }
};

#define SG_LAUNCH_CHECK(what)                                            \
    do {                                                                 \
        cudaError_t e_ = cudaGetLastError();                             \
        if (e_ != cudaSuccess) return cuda_fail(e_, what);               \
    } while (0)

// the training kernels' shared memory, once per device (a function's attributes last as its context)
cudaError_t train_kernel_attributes(int device)
{
    static std::atomic<bool> done[64];
    if (device >= 0 && device < 64 && done[device].load(std::memory_order_acquire)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(train_layer2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLayer2Smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(train_back_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBackSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(train_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgradSmem);
    if (e == cudaSuccess && device >= 0 && device < 64) done[device].store(true, std::memory_order_release);
    return e;
}

// forward + backward of one batch; gradients land in bt.grad (parameter layout), the loss in bt.loss. With
// Adam's arguments the parameters and their BF16 copies move too, and the device counter `step` advances.
int forward_backward(const aiwcrf_surrogate *sg, Batch &bt, const float *X, int64_t ld, const uint32_t *perm,
                     int64_t r0, const float *y, cudaStream_t s, int64_t *step = nullptr, int64_t spe = 1,
                     const AdamArgs &adam = AdamArgs{})
{
    TrainArgs a = bt.a;
    a.e = encoder_of(sg);
    a.X = X; a.ld = ld; a.perm = perm; a.r0 = r0; a.yall = y; a.step = step; a.spe = spe;
    a.P = sg->d_param; a.W1b = sg->d_W1b; a.W2b = sg->d_W2b;
    const cudaError_t e = train_kernel_attributes(sg->device);
    if (e != cudaSuccess) return cuda_fail(e, "surrogate training attributes");
    // slices and tiles in one dimension: the second one ends at 65,535
    const unsigned grid = (unsigned)kSlices * (unsigned)(a.B / 128);
    train_layer1_kernel<<<grid, kTrainThreads, 0, s>>>(a);
    train_layer2_kernel<<<grid, kTrainThreads, kLayer2Smem, s>>>(a);
    train_back_kernel<<<grid, kTrainThreads, kBackSmem, s>>>(a);
    SG_LAUNCH_CHECK("surrogate training step");      // before anything is written to the caller's arrays
    train_wgrad_kernel<<<dim3(2, (unsigned)a.splits), kTrainThreads, kWgradSmem, s>>>(a, step);
    train_reduce_kernel<<<(kParams + kReduceThreads) / kReduceThreads, kReduceThreads, 0, s>>>(a, bt.grad, bt.loss, adam);
    count_launches(5);
    SG_LAUNCH_CHECK("surrogate training step");
    return AIWCRF_OK;
}

// A training step captured as a CUDA graph on its own stream (so that a caller's legacy default
// stream is never captured), instantiated once and replayed.
struct TrainGraph {
    cudaStream_t ts = nullptr;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t x = nullptr;
    size_t nodes = 0;
    ~TrainGraph()
    {
        if (x) cudaGraphExecDestroy(x);
        if (g) cudaGraphDestroy(g);
        if (ts) cudaStreamDestroy(ts);
    }
    template <class F>
    int capture(F &&body)
    {
        cudaError_t e = cudaStreamCreateWithFlags(&ts, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaStreamBeginCapture(ts, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return cuda_fail(e, "surrogate step capture");
        const int rc = body(ts);
        e = cudaStreamEndCapture(ts, &g);
        if (rc) return rc;
        if (e == cudaSuccess) e = cudaGraphInstantiate(&x, g, 0);
        if (e == cudaSuccess) e = cudaGraphGetNodes(g, nullptr, &nodes);
        if (e != cudaSuccess) return cuda_fail(e, "surrogate step graph");
        return AIWCRF_OK;
    }
    int replay()
    {
        const cudaError_t e = cudaGraphLaunch(x, ts);
        if (e != cudaSuccess) return cuda_fail(e, "surrogate step replay");
        count_launches((int64_t)nodes);
        return AIWCRF_OK;
    }
};

int check_err(const Batch &bt, cudaStream_t s)
{
    uint32_t pageable = 0, *h = static_cast<uint32_t *>(pinned_scratch());      // an asynchronous read, if it can be had
    if (!h) h = &pageable;
    cudaError_t e = cudaMemcpyAsync(h, bt.err, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "surrogate");
    if (*h & kErrTimeout) return fail(AIWCRF_E_TIMEOUT, "a tensor-core wait gave up");
    return AIWCRF_OK;
}

// feature transform from a sample: log2 for columns that are >= 1 and span three orders of
// magnitude; mean and standard deviation of the (transformed) column
void fit_encoder(aiwcrf_surrogate *sg, const std::vector<float> &sample, int64_t n)
{
    sg->mu.assign((size_t)sg->n_aiwc, 0.0f);
    sg->sd.assign((size_t)sg->n_aiwc, 1.0f);
    sg->logf.assign((size_t)sg->n_aiwc, 0);
    for (int f = 0; f < sg->n_aiwc; ++f) {
        const float *c = sample.data() + (size_t)f * (size_t)n;
        float lo = c[0], hi = c[0];
        for (int64_t i = 0; i < n; ++i) { lo = std::min(lo, c[i]); hi = std::max(hi, c[i]); }
        const bool lg = lo >= 1.0f && hi >= 1000.0f * lo;
        double s1 = 0, s2 = 0;
        for (int64_t i = 0; i < n; ++i) {
            const double x = lg ? std::log2(std::max((double)c[i], 1.0)) : (double)c[i];
            s1 += x;
            s2 += x * x;
        }
        const double m = s1 / (double)n, var = std::max(s2 / (double)n - m * m, 1e-12);
        sg->logf[(size_t)f] = lg ? 1 : 0;
        sg->mu[(size_t)f] = (float)m;
        sg->sd[(size_t)f] = (float)std::sqrt(var);
    }
}

void init_params(std::vector<float> &P, uint64_t seed, int in_dim)
{
    std::mt19937_64 rng(seed);
    P.assign((size_t)kParams, 0.0f);
    std::uniform_real_distribution<float> u(-1.0f, 1.0f);
    const float a1 = std::sqrt(6.0f / (float)in_dim), a2 = std::sqrt(6.0f / (float)kHid);
    for (int r = 0; r < kHid; ++r)
        for (int k = 0; k < in_dim; ++k) P[(size_t)(oW1 + r * kIn + k)] = a1 * u(rng);
    for (int i = 0; i < kHid * kHid; ++i) P[(size_t)(oW2 + i)] = a2 * u(rng);
    for (int i = 0; i < kHid; ++i) P[(size_t)(ow3 + i)] = a2 * u(rng) * 0.5f;
}

int upload_encoder(aiwcrf_surrogate *sg)
{
    cudaError_t e = cudaMemcpy(sg->d_mu, sg->mu.data(), 4 * sg->mu.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(sg->d_sd, sg->sd.data(), 4 * sg->sd.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(sg->d_logf, sg->logf.data(), sg->logf.size(), cudaMemcpyHostToDevice);
    return e == cudaSuccess ? AIWCRF_OK : cuda_fail(e, "surrogate encoder upload");
}

int new_surrogate(int32_t F, int32_t n_dev, int32_t n_size, aiwcrf_surrogate **out)
{
    if (F < 3 || n_dev < 1 || n_size < 1 || (F - 2) + n_dev + n_size > kIn)
        return fail(AIWCRF_E_INVALID_ARG, "surrogate inputs: (F - 2) + n_devices + n_sizes must be <= 64");
    int dev;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "no usable CUDA device");
    aiwcrf_surrogate *sg = new aiwcrf_surrogate();
    sg->device = dev;
    sg->F = F; sg->n_aiwc = F - 2; sg->n_dev = n_dev; sg->n_size = n_size;
    int rc = surrogate_alloc(sg);
    if (rc) { delete sg; return rc; }
    *out = sg;
    return AIWCRF_OK;
}

}  // namespace

int surrogate_clone(const aiwcrf_surrogate *src, aiwcrf_surrogate **out)
{
    int cur = 0;
    cudaGetDevice(&cur);
    if (cur != src->device) cudaSetDevice(src->device);
    aiwcrf_surrogate *sg = nullptr;
    int rc = new_surrogate(src->F, src->n_dev, src->n_size, &sg);
    if (!rc) {
        sg->mu = src->mu;
        sg->sd = src->sd;
        sg->logf = src->logf;
        sg->stats = src->stats;
        // the same sizes give the same block layout: one device-to-device copy
        cudaError_t e = cudaMemcpyAsync(sg->d_block, src->d_block, surrogate_block_bytes(src->n_aiwc),
                                        cudaMemcpyDeviceToDevice, cudaStreamPerThread);
        if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamPerThread);
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "surrogate copy");
            surrogate_release(sg);
            sg = nullptr;
        }
    }
    if (cur != src->device) cudaSetDevice(cur);
    if (rc) return rc;
    *out = sg;
    return AIWCRF_OK;
}

SurrogateInfo surrogate_info(const aiwcrf_surrogate *sg)
{
    return SurrogateInfo{sg->device, sg->F, (int64_t)surrogate_block_bytes(sg->n_aiwc)};
}

void surrogate_release_async(aiwcrf_surrogate *sg, cudaStream_t s)
{
    if (!sg) return;
    if (sg->d_block) cudaFreeAsync(sg->d_block, s);
    delete sg;
}

int surrogate_predict_enqueue(const aiwcrf_surrogate *sg, const float *dXq, int64_t Q, float *d_out, uint32_t *d_err,
                              cudaStream_t s)
{
    if (Q == 0) return AIWCRF_OK;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaFuncSetAttribute(surrogate_infer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kInferSmem);
    if (e != cudaSuccess) return cuda_fail(e, "surrogate kernel attribute");
    const int64_t tiles = (Q + 127) / 128;
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(tiles, sms));
    surrogate_infer_kernel<<<grid, kInferThreads, kInferSmem, s>>>(encoder_of(sg), dXq, Q, sg->d_W1b, sg->d_W2b,
                                                                     sg->d_param + ob1, sg->d_param + ob2,
                                                                     sg->d_param + ow3, sg->d_param + ob3, d_out, d_err);
    count_launches(1);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "surrogate_infer_kernel launch");
    return AIWCRF_OK;
}

int surrogate_predict_launch(const aiwcrf_surrogate *sg, const float *dXq, int64_t Q, float *d_out, cudaStream_t s)
{
    if (Q == 0) return AIWCRF_OK;
    uint32_t *d_err = nullptr;
    if (cudaMallocAsync(&d_err, 4, s) != cudaSuccess) return fail(AIWCRF_E_OOM, "surrogate error flag");
    cudaMemsetAsync(d_err, 0, 4, s);
    int rc = surrogate_predict_enqueue(sg, dXq, Q, d_out, d_err, s);
    if (rc) { cudaFreeAsync(d_err, s); return rc; }
    cudaError_t e = cudaSuccess;
    uint32_t h = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d_err, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFreeAsync(d_err, s);
    if (e != cudaSuccess) return cuda_fail(e, "surrogate predict");
    if (h & kErrTimeout) return fail(AIWCRF_E_TIMEOUT, "a tensor-core wait gave up");
    return AIWCRF_OK;
}

}  // namespace aiwcrf

using namespace aiwcrf;

extern "C" {

int aiwcrf_surrogate_fit(const aiwcrf_surrogate_params *p, const aiwcrf_forest *teacher, const float *X, int64_t n,
                         int32_t n_features, void *cuda_stream, aiwcrf_surrogate **out)
{
    aiwcrf::clear_last_error();
    if (!p || !teacher || !X || !out) return fail(AIWCRF_E_INVALID_ARG, "params, teacher, X and out must not be NULL");
    if (n_features != teacher->F) return fail(AIWCRF_E_INVALID_ARG, "X must have the teacher's features");
    if (p->batch < 128 || p->batch % 128 || p->batch > 65536 || p->epochs < 1 || !(p->lr > 0.0f) || n < p->batch)
        return fail(AIWCRF_E_INVALID_ARG, "batch must be a multiple of 128 in [128, 65536], epochs >= 1, lr > 0, n >= batch");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    int dev;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "no usable CUDA device");
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, X) != cudaSuccess || at.type != cudaMemoryTypeDevice) {
        cudaGetLastError();
        return fail(AIWCRF_E_BAD_POINTER, "X must be device memory");
    }
    keep_pool_memory(dev);
    aiwcrf_surrogate *sg = nullptr;
    int rc = new_surrogate(n_features, p->n_devices, p->n_sizes, &sg);
    if (rc) return rc;
    struct Guard { aiwcrf_surrogate *g; bool keep = false; ~Guard() { if (!keep && g) surrogate_release(g); } } guard{sg};

    // labels: the teacher forest's predictions (log10 seconds)
    float *d_y = nullptr;
    int64_t *d_pred = nullptr;
    if (cudaMallocAsync(&d_y, 4 * (size_t)n, s) != cudaSuccess || cudaMallocAsync(&d_pred, 8 * (size_t)n, s) != cudaSuccess)
        return fail(AIWCRF_E_OOM, "surrogate labels");
    struct FreeY { float *a; int64_t *b; cudaStream_t s; ~FreeY() { cudaFreeAsync(a, s); cudaFreeAsync(b, s); } } fy{d_y, d_pred, s};
    if ((rc = predict_launch(teacher, X, n, nullptr, d_pred, nullptr, teacher->T, s))) return rc;
    {
        std::vector<int64_t> h((size_t)n);
        e = cudaMemcpyAsync(h.data(), d_pred, 8 * (size_t)n, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return cuda_fail(e, "surrogate labels");
        std::vector<float> hy((size_t)n);
        for (int64_t i = 0; i < n; ++i) hy[(size_t)i] = (float)((double)h[(size_t)i] / 4294967296.0);
        e = cudaMemcpy(d_y, hy.data(), 4 * (size_t)n, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return cuda_fail(e, "surrogate labels");
    }
    // encoder from a sample of the inputs
    {
        const int64_t m = std::min<int64_t>(n, 65536);
        std::vector<float> sample((size_t)sg->n_aiwc * (size_t)m);
        for (int f = 0; f < sg->n_aiwc; ++f) {
            e = cudaMemcpy(sample.data() + (size_t)f * (size_t)m, X + (size_t)f * (size_t)n, 4 * (size_t)m,
                           cudaMemcpyDeviceToHost);
            if (e != cudaSuccess) return cuda_fail(e, "surrogate sample");
        }
        fit_encoder(sg, sample, m);
        if ((rc = upload_encoder(sg))) return rc;
    }
    std::vector<float> P;
    init_params(P, p->seed, sg->n_aiwc + sg->n_dev + sg->n_size);
    e = cudaMemcpy(sg->d_param, P.data(), 4 * (size_t)kParams, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(e, "surrogate parameters");
    if ((rc = refresh_bf16(sg, s))) return rc;

    Batch bt;
    if ((rc = bt.alloc(p->batch, true, s))) return rc;
    const int64_t steps_per_epoch = n / p->batch;
    uint32_t *d_perm = nullptr;
    if (cudaMallocAsync(&d_perm, 4 * (size_t)n, s) != cudaSuccess) return fail(AIWCRF_E_OOM, "surrogate permutation");
    struct FreeP { uint32_t *a; cudaStream_t s; ~FreeP() { cudaFreeAsync(a, s); } } fp{d_perm, s};
    std::vector<uint32_t> perm((size_t)n);
    for (int64_t i = 0; i < n; ++i) perm[(size_t)i] = (uint32_t)i;
    std::mt19937_64 rng(p->seed ^ 0x5DEECE66Dull);
    float first_loss = -1.0f, last_loss = -1.0f;
    const int64_t total_steps = (int64_t)p->epochs * steps_per_epoch;
    // Adam's bias corrections of every step, as the step-by-step loop computes them
    std::vector<float> c12((size_t)(2 * total_steps));
    for (int64_t t1 = 1; t1 <= total_steps; ++t1) {
        c12[(size_t)(2 * (t1 - 1))] = 1.0f - std::pow(p->beta1, (float)t1);
        c12[(size_t)(2 * (t1 - 1) + 1)] = 1.0f - std::pow(p->beta2, (float)t1);
    }
    // One training step (forward, backward, Adam, BF16 weight copies, step counter) is captured
    // once as a CUDA graph on a private stream and replayed: it reads its batch offset and bias
    // corrections through the device step counter, so the replays are the step-by-step loop's
    // launches without their host cost.
    TrainGraph tg;
    float *d_c12 = nullptr;
    int64_t *d_step = nullptr;
    if (cudaMallocAsync(&d_c12, 4 * c12.size(), s) != cudaSuccess || cudaMallocAsync(&d_step, 8, s) != cudaSuccess)
        return fail(AIWCRF_E_OOM, "surrogate step tables");
    struct FreeC { float *a; int64_t *b; cudaStream_t s; ~FreeC() { cudaFreeAsync(a, s); cudaFreeAsync(b, s); } } fc{d_c12, d_step, s};
    e = cudaMemcpyAsync(d_c12, c12.data(), 4 * c12.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_step, 0, 8, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "surrogate step tables");
    if ((rc = tg.capture([&](cudaStream_t ts) {
             return forward_backward(sg, bt, X, n, d_perm, 0, d_y, ts, d_step, steps_per_epoch,
                                     AdamArgs{sg->d_param, bt.m, bt.v, sg->d_W1b, sg->d_W2b, p->lr, p->beta1, p->beta2,
                                              p->eps, d_c12, d_step});
         })))
        return rc;
    int64_t t = 0;
    for (int ep = 0; ep < p->epochs; ++ep) {
        std::shuffle(perm.begin(), perm.end(), rng);
        e = cudaMemcpyAsync(d_perm, perm.data(), 4 * (size_t)n, cudaMemcpyHostToDevice, tg.ts);
        if (e == cudaSuccess) e = cudaStreamSynchronize(tg.ts);      // the host array is reshuffled next epoch
        if (e != cudaSuccess) return cuda_fail(e, "surrogate permutation");
        for (int64_t k = 0; k < steps_per_epoch; ++k) {
            if ((rc = tg.replay())) return rc;
            ++t;
            if (k == 0 || k == steps_per_epoch - 1) {
                float hl = 0.0f;
                e = cudaMemcpyAsync(&hl, bt.loss, 4, cudaMemcpyDeviceToHost, tg.ts);
                if (e == cudaSuccess) e = cudaStreamSynchronize(tg.ts);
                if (e != cudaSuccess) return cuda_fail(e, "surrogate loss");
                if (first_loss < 0.0f) first_loss = hl / (float)p->batch;
                last_loss = hl / (float)p->batch;
            }
        }
    }
    e = cudaStreamSynchronize(tg.ts);
    if (e != cudaSuccess) return cuda_fail(e, "surrogate training");
    if ((rc = check_err(bt, s))) return rc;
    sg->stats.steps = t;
    sg->stats.first_batch_loss = first_loss;
    sg->stats.last_batch_loss = last_loss;
    guard.keep = true;
    *out = sg;
    return AIWCRF_OK;
}

int aiwcrf_surrogate_predict(const aiwcrf_surrogate *sg, const float *Xq, int64_t n, float *out, void *cuda_stream)
{
    aiwcrf::clear_last_error();
    if (!sg || !Xq || !out) return fail(AIWCRF_E_INVALID_ARG, "surrogate, Xq and out must not be NULL");
    if (n < 0) return fail(AIWCRF_E_INVALID_ARG, "n must be >= 0");
    cudaPointerAttributes a1, a2;
    if (cudaPointerGetAttributes(&a1, Xq) != cudaSuccess || cudaPointerGetAttributes(&a2, out) != cudaSuccess ||
        a1.type != cudaMemoryTypeDevice || a2.type != cudaMemoryTypeDevice) {
        cudaGetLastError();
        return fail(AIWCRF_E_BAD_POINTER, "Xq and out must be device memory");
    }
    return surrogate_predict_launch(sg, Xq, n, out, (cudaStream_t)cuda_stream);
}

int aiwcrf_surrogate_grad(const aiwcrf_surrogate *sg, const float *X, const float *y, int32_t n, float *grad,
                          float *loss, void *cuda_stream)
{
    aiwcrf::clear_last_error();
    if (!sg || !X || !y || !grad || !loss || n < 128 || n % 128)
        return fail(AIWCRF_E_INVALID_ARG, "arguments must not be NULL; n a positive multiple of 128");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    Batch bt;
    int rc;
    if ((rc = bt.alloc(n, false, s))) return rc;
    // the last kernel writes to the caller's arrays where they are this device's
    cudaPointerAttributes ag, al;
    if (cudaPointerGetAttributes(&ag, grad) == cudaSuccess && cudaPointerGetAttributes(&al, loss) == cudaSuccess &&
        ag.type == cudaMemoryTypeDevice && al.type == cudaMemoryTypeDevice && ag.device == sg->device &&
        al.device == sg->device) {
        bt.grad = grad;
        bt.loss = loss;
        if ((rc = forward_backward(sg, bt, X, n, nullptr, 0, y, s))) return rc;
        return check_err(bt, s);
    }
    cudaGetLastError();
    if ((rc = forward_backward(sg, bt, X, n, nullptr, 0, y, s))) return rc;
    cudaError_t e = cudaMemcpyAsync(grad, bt.grad, 4 * (size_t)kParams, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(loss, bt.loss, 4, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return cuda_fail(e, "surrogate gradients");
    return check_err(bt, s);
}

int aiwcrf_surrogate_create(int32_t n_features, int32_t n_devices, int32_t n_sizes, const float *params,
                            const float *mu, const float *sd, const uint8_t *log2_cols, aiwcrf_surrogate **out)
{
    aiwcrf::clear_last_error();
    if (!params || !mu || !sd || !log2_cols || !out) return fail(AIWCRF_E_INVALID_ARG, "arguments must not be NULL");
    aiwcrf_surrogate *sg = nullptr;
    int rc = new_surrogate(n_features, n_devices, n_sizes, &sg);
    if (rc) return rc;
    sg->mu.assign(mu, mu + sg->n_aiwc);
    sg->sd.assign(sd, sd + sg->n_aiwc);
    sg->logf.assign(log2_cols, log2_cols + sg->n_aiwc);
    if (!(rc = upload_encoder(sg))) {
        cudaError_t e = cudaMemcpy(sg->d_param, params, 4 * (size_t)kParams, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) rc = cuda_fail(e, "surrogate parameters");
    }
    if (!rc) rc = refresh_bf16(sg, nullptr);
    if (!rc && cudaDeviceSynchronize() != cudaSuccess) rc = cuda_fail(cudaGetLastError(), "surrogate create");
    if (rc) { surrogate_release(sg); return rc; }
    *out = sg;
    return AIWCRF_OK;
}

int aiwcrf_surrogate_export(const aiwcrf_surrogate *sg, float *params, float *mu, float *sd, uint8_t *log2_cols)
{
    aiwcrf::clear_last_error();
    if (!sg) return fail(AIWCRF_E_INVALID_ARG, "surrogate is NULL");
    if (params && cudaMemcpy(params, sg->d_param, 4 * (size_t)kParams, cudaMemcpyDeviceToHost) != cudaSuccess)
        return cuda_fail(cudaGetLastError(), "surrogate export");
    if (mu) std::memcpy(mu, sg->mu.data(), 4 * sg->mu.size());
    if (sd) std::memcpy(sd, sg->sd.data(), 4 * sg->sd.size());
    if (log2_cols) std::memcpy(log2_cols, sg->logf.data(), sg->logf.size());
    return AIWCRF_OK;
}

int aiwcrf_surrogate_stats(const aiwcrf_surrogate *sg, aiwcrf_surrogate_fit_stats *out)
{
    aiwcrf::clear_last_error();
    if (!sg || !out) return fail(AIWCRF_E_INVALID_ARG, "arguments must not be NULL");
    *out = sg->stats;
    return AIWCRF_OK;
}

int32_t aiwcrf_surrogate_num_params(void) { return kParams; }

int aiwcrf_surrogate_free(aiwcrf_surrogate *sg)
{
    aiwcrf::clear_last_error();
    if (!sg) return AIWCRF_OK;
    surrogate_release(sg);
    return AIWCRF_OK;
}

}  // extern "C"
