// Activation importance (Eq. 7): I[k] = sum_t X[t,k]^2, a streaming column reduction.
//
// Layout: X is [T x K] BF16 row-major.  A block covers 256 adjacent columns (each lane owns
// 8 of them = one 128-bit load per row) and a strip of rows; its 8 warps take rows
// round-robin.  The sums are kept in double: a BF16 magnitude becomes a double by two integer
// instructions (its fields moved, the exponent rebased), and one double-precision multiply-add
// squares it -- exactly -- and adds it, so a sum is off by a few 2^-53.  That is three
// instructions an element where error-free FP32 pairs took nine, and leaves the pass to the
// memory (16384 x 14336: 4.2 -> 5.8 TB/s with the launch geometry below).  A second kernel adds
// the strip partials in a fixed order and rounds once to FP32.
#include <algorithm>
#include <mutex>

#include "internal.cuh"

namespace aaac {

namespace {

constexpr int kWarps = 8;
constexpr int kUnroll = 4;
constexpr int kBlocksPerSM = 4;          // resident blocks: 64 KB of loads in flight per SM

// |a| of a BF16 value as a double (upper word; the lower is zero).  A zero or a denormal reads as some
// 2^-127 <= |a| < 2^-126, whose square is below 2^-252 and vanishes in an FP32 sum; Inf and NaN read as
// 2^128 and more, whose square is beyond an FP32 sum (see finish).
__device__ __forceinline__ double abs_lo(uint32_t w) { return __hiloint2double((int)((w & 0x7FFFu) * 8192u + 0x38000000u), 0); }
__device__ __forceinline__ double abs_hi(uint32_t w) { return __hiloint2double((int)(((w & 0x7FFF0000u) >> 3) + 0x38000000u), 0); }
__device__ __forceinline__ void add_squares(double (&s)[8], uint4 v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const double a = abs_lo(w[j]), b = abs_hi(w[j]);
        s[2 * j] = __fma_rn(a, a, s[2 * j]);
        s[2 * j + 1] = __fma_rn(b, b, s[2 * j + 1]);
    }
}

__device__ __forceinline__ void finish(float* I, int64_t k, double s, int accumulate, uint32_t* dev_status) {
    float v = (float)s;
    if (isinf(v)) v = __int_as_float(0x7FFFFFFF);          // NaN: Inf and NaN among the inputs cannot be told apart any more
    if (accumulate) v += I[k];
    I[k] = v;
    if (dev_status && !isfinite(v)) atomicOr(dev_status, AAAC_DEV_NONFINITE);
}

__global__ void __launch_bounds__(kWarps * 32, kBlocksPerSM)
act_sumsq_kernel(const uint16_t* __restrict__ X, int64_t T, int64_t K, int64_t ldx,
                 double* __restrict__ part, int rows_per_split, int strip0, float* __restrict__ I, int accumulate,
                 uint32_t* dev_status) {
    __shared__ double sm[kWarps][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t col0 = (int64_t)blockIdx.x * 256 + lane * 8;
    const bool active = col0 < K;
    const int strip = strip0 + blockIdx.y;
    const int64_t t_begin = (int64_t)strip * rows_per_split;
    const int64_t t_end = min(T, t_begin + rows_per_split);
    chain_next();
    chain_wait();
    double s8[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) s8[j] = 0.0;

    if (active) {
        const uint16_t* base = X + col0;
        int64_t t = t_begin + warp;
        for (; t + (kUnroll - 1) * kWarps < t_end; t += kUnroll * kWarps) {
            uint4 v[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u)
                v[u] = __ldcs(reinterpret_cast<const uint4*>(base + (t + u * kWarps) * ldx));
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) add_squares(s8, v[u]);
        }
        for (; t < t_end; t += kWarps) add_squares(s8, __ldcs(reinterpret_cast<const uint4*>(base + t * ldx)));
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) sm[warp][lane * 8 + j] = s8[j];
    __syncthreads();
    const int64_t col = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (col < K) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) s += sm[w][threadIdx.x];
        if (I) finish(I, col, s, accumulate, dev_status);          // the only strip
        else part[(int64_t)strip * K + col] = s;
    }
}

// A block takes 32 columns; warp w adds the strips w, w + 8, ... of its columns, and the eight partial sums
// are added in order.
__global__ void __launch_bounds__(kWarps * 32)
act_final_kernel(const double* __restrict__ part, int splits, int64_t K,
                 float* __restrict__ I, int accumulate, uint32_t* dev_status) {
    __shared__ double sm[kWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t k = (int64_t)blockIdx.x * 32 + lane;
    double s = 0.0;
    chain_next();
    chain_wait();
    if (k < K) {
#pragma unroll 4
        for (int p = warp; p < splits; p += kWarps) s += part[(int64_t)p * K + k];
    }
    sm[warp][lane] = s;
    __syncthreads();
    if (warp != 0 || k >= K) return;
#pragma unroll
    for (int w = 1; w < kWarps; ++w) s += sm[w][lane];
    finish(I, k, s, accumulate, dev_status);
}

}  // namespace

// Row strips for K input channels: one wave of resident blocks (a second, partly filled one costs more than
// shorter strips give back).
int act_splits_max(int64_t K) {
    const int64_t bx = K > 0 ? (K + 255) / 256 : 1;
    const int64_t want = (int64_t)sm_count() * kBlocksPerSM / bx;
    return (int)(want < 1 ? 1 : want > kActMaxSplits ? kActMaxSplits : want);
}

// A pass over few rows is one strip, which needs no second kernel: up to 64 rows (two loop iterations of a block) it is
// shorter than that kernel, and up to 128 where a caller waits for this result alone and nothing runs beside it
// (kActAlone; 128 x 512 3.0 -> 2.7 us, 128 x 4096 4.2 -> 2.8, but 256 x 512 3.0 -> 4.1).
ActPlan act_plan(int64_t T, int64_t K, int max_splits, int64_t one_strip_rows) {
    int64_t splits = T <= one_strip_rows ? 1 : std::min<int64_t>(max_splits, (T + kWarps - 1) / kWarps);
    ActPlan p;
    p.rows = ((T + splits - 1) / splits + kWarps - 1) / kWarps * kWarps;
    p.strips = (int)((T + p.rows - 1) / p.rows);
    return p;
}

cudaError_t launch_act_strips(const uint16_t* X, int64_t T, int64_t K, int64_t ldx, const ActPlan& plan, int first, int count,
                              float* I, int accumulate, uint32_t* dev_status, double* part, cudaStream_t st) {
    note_launch();
    return launch_chained(act_sumsq_kernel, dim3((unsigned)((K + 255) / 256), (unsigned)count), kWarps * 32, 0, st, X, T, K, ldx, part,
                          (int)plan.rows, first, plan.strips == 1 ? I : nullptr, accumulate, dev_status);
}

cudaError_t launch_act_finish(int64_t K, const ActPlan& plan, float* I, int accumulate, uint32_t* dev_status, const double* part,
                              cudaStream_t st) {
    if (plan.strips == 1) return cudaSuccess;              // the strip kernel has finished the sums itself
    note_launch();
    return launch_chained(act_final_kernel, (unsigned)((K + 31) / 32), kWarps * 32, 0, st, part, plan.strips, K, I, accumulate, dev_status);
}

namespace {
// both launches; `part` holds [max_splits][K] doubles.  Every partial that the second kernel reads is written
// by the first: nothing has to be cleared.
cudaError_t run_act_stats(const uint16_t* X, int64_t T, int64_t K, int64_t ldx, float* I, int accumulate, uint32_t* dev_status,
                          double* part, int max_splits, int64_t one_strip_rows, cudaStream_t st) {
    const ActPlan plan = act_plan(T, K, max_splits, one_strip_rows);
    const cudaError_t e = launch_act_strips(X, T, K, ldx, plan, 0, plan.strips, I, accumulate, dev_status, part, st);
    return e != cudaSuccess ? e : launch_act_finish(K, plan, I, accumulate, dev_status, part, st);
}
}  // namespace

cudaError_t launch_act_stats(const uint16_t* X, int64_t T, int64_t K, int64_t ldx, float* I, int accumulate,
                             uint32_t* dev_status, const Workspace& ws, int64_t one_strip_rows, cudaStream_t st) {
    return run_act_stats(X, T, K, ldx, I, accumulate, dev_status, ws.act_part, act_splits_max(K), one_strip_rows, st);
}

}  // namespace aaac

// ---------------------------------------------------------------------------------------------
// aaac_act_stats_noalloc: the same reduction for callers that cannot hand over scratch memory.
//
// The strip partials live in a fixed array in the library's own device image instead of a
// caller workspace, so the call needs no buffer besides X and I.  The array exists once per
// GPU that loads the library and is shared by every call on that GPU.
// ---------------------------------------------------------------------------------------------
namespace aaac {
namespace {

constexpr int kNoAllocMaxK = 32768;       // widest layer input the built-in scratch covers
constexpr int kNoAllocSplits = 32;        // row strips (8 MiB of scratch in total)

static __device__ __align__(256) double g_noalloc_part[(size_t)kNoAllocSplits * kNoAllocMaxK];

std::mutex g_noalloc_mu;
double* g_noalloc_ptr[64] = {nullptr};   // device address of the array, per device ordinal

// Host code cannot use the array's name as a pointer: the name only identifies the symbol.
// Its device address is looked up once per device, with that device current.
cudaError_t noalloc_scratch(double** out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        double* p = nullptr;
        e = cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_noalloc_part);
        if (e != cudaSuccess) return e;
        if (!p) return cudaErrorInvalidSymbol;
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    return cudaSuccess;
}

}  // namespace
}  // namespace aaac

extern "C" int aaac_act_stats_noalloc(const void* X, int64_t T, int64_t K, int64_t ldx, float* I, int accumulate,
                                      uint32_t* dev_status, void* stream) {
    using namespace aaac;
    if (!X || !I) return AAAC_ERR_NULL;
    if (T < 1 || K < 1 || K % 8 || ldx < K || ldx % 8) return AAAC_ERR_SHAPE;
    if (K > kNoAllocMaxK) return AAAC_ERR_TOO_LARGE;
    if ((reinterpret_cast<uintptr_t>(X) % 16) || (reinterpret_cast<uintptr_t>(I) % 4)) return AAAC_ERR_ALIGN;
    double* part = nullptr;
    if (noalloc_scratch(&part) != cudaSuccess) return AAAC_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int splits = std::min(act_splits_max(K), kNoAllocSplits);
    if (run_act_stats(static_cast<const uint16_t*>(X), T, K, ldx, I, accumulate, dev_status, part, splits, kActAlone, st) != cudaSuccess) return AAAC_ERR_CUDA;
    return AAAC_OK;
}
