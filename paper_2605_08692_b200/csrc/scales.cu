// Per-group positive scales (Algorithm 1, line 1).
//
//   INT4  (g = 128): s = bf16_rne(absmax / 7), 1 for an all-zero group, never below 2^-126.
//                    Also writes r = fl32(1/s) per group for the fit rounds.
//   NVFP4 (g = 16) : s_t = layer absmax / 2688 (a first pass over W), then per group
//                    q = E4M3_rne(absmax / (6 s_t)) kept inside 0x01..0x7E; in the lowest
//                    subnormal step the code is raised so that |w / s| <= 7.5.
// Both rules keep every normalised weight strictly inside (-8, 8).
//
// One warp handles 256 adjacent weights (one 128-bit load per lane); the group
// maximum is a shuffle reduction over the 16 (INT4) or 2 (NVFP4) lanes of the group.
#include "internal.cuh"

namespace aaac {

namespace {

__device__ __forceinline__ uint32_t absmax16(uint4 v) {
    // max over the eight BF16 magnitudes (bit patterns of non-negative floats order like ints)
    uint32_t m = 0;
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        m = max(m, w[j] & 0x7FFFu);
        m = max(m, (w[j] >> 16) & 0x7FFFu);
    }
    return m;
}

// Layer absmax, eight pieces in flight per thread.
constexpr int kAbsLoads = 8;
template <bool DENSE>
__global__ void __launch_bounds__(256)
absmax_kernel(const uint16_t* __restrict__ W, unsigned n, unsigned per_row, int64_t ldw, Ctrl* ctrl, uint32_t* dev_status) {
    chain_next();
    chain_wait();
    const int lane = threadIdx.x & 31;
    const unsigned step = gridDim.x * 256u;
    uint32_t m = 0;
    for (unsigned i = blockIdx.x * 256u + threadIdx.x; i < n; i += step * kAbsLoads) {
        uint4 v[kAbsLoads];
#pragma unroll
        for (int u = 0; u < kAbsLoads; ++u) v[u] = load_piece<DENSE>(W, min(i + u * step, n - 1u), per_row, ldw);
#pragma unroll
        for (int u = 0; u < kAbsLoads; ++u) m = max(m, absmax16(v[u]));
    }
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if (lane == 0 && m) {
        atomicMax(&ctrl->absmax_bits, m << 16);
        if (m >= 0x7F80u) {
            atomicOr(&ctrl->nonfinite, 1u);
            if (dev_status) atomicOr(dev_status, AAAC_DEV_NONFINITE);
        }
    }
}

// The two scale rules, with the division replaced by a multiplication by the reciprocal wherever that cannot
// change the result: the product is within three units in the last place of the quotient, so the rounding
// that follows (to BF16, to E4M3) gives the same unless the product lies that close to a half-way point.
// Those few, and small quotients, take the division (it cost four instructions per weight of the pass).
__device__ __forceinline__ uint32_t int4_scale_bits(float a) {
    if (a == 0.f) return 0x3F80u;
    float y = __fmul_rn(a, 1.f / 7.f);
    if ((((__float_as_uint(y) + 0x8004u) & 0xFFFFu) <= 8u) || !(y >= 0x1p-100f)) y = __fdiv_rn(a, 7.f);
    float s = __uint_as_float(f32_to_bf16_rne(y) << 16);
    if (s < 0x1p-126f) s = 0x1p-126f;
    return __float_as_uint(s) >> 16;
}
__device__ __forceinline__ uint32_t nvfp4_scale_code(float a, float d6, float inv6) {
    const float y = __fmul_rn(a, inv6);
    const uint32_t u = __float_as_uint(y);
    if (y >= 0.0157f && y < 447.f && ((u + 0x80004u) & 0xFFFFFu) > 8u)            // normal codes: 3 mantissa bits
        return ((u + 0x7FFFFu + ((u >> 20) & 1u)) >> 20) - 960u;
    const float x = __fdiv_rn(a, d6);
    uint32_t q = e4m3_encode(x);
    if (q <= 1u) q = (x > 1.25f * 0x1p-9f) ? 2u : 1u;
    return q;
}

template <int MODE, bool DENSE>
__global__ void __launch_bounds__(256)
scales_kernel(const uint16_t* __restrict__ W, unsigned n, unsigned per_row, int64_t ldw, void* __restrict__ scales,
              float* __restrict__ rinv, float* __restrict__ tensor_scale, Ctrl* ctrl, uint32_t* dev_status) {
    constexpr int G = MODE == AAAC_INT4 ? 128 : 16;
    constexpr int LPG = G / 8;                         // lanes per group
    chain_next();
    chain_wait();
    const int lane = threadIdx.x & 31;
    const unsigned step = gridDim.x * blockDim.x;

    float s_t = 1.f, d6 = 6.f, inv6 = 1.f;
    if (MODE == AAAC_NVFP4) {
        const float A = __uint_as_float(ctrl->absmax_bits);
        s_t = (A == 0.f) ? 1.f : __fdiv_rn(A, 2688.f);
        if (s_t < 0x1p-96f) s_t = 0x1p-96f;
        d6 = __fmul_rn(6.f, s_t);
        inv6 = __frcp_rn(d6);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctrl->s_t = s_t;
        if (tensor_scale) tensor_scale[0] = s_t;
    }
    bool bad = false;
    // four pieces in flight per thread; whole warps go round the loop (a group is 2 or 16 lanes, and n a
    // multiple of that)
    for (unsigned i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); i0 < n; i0 += 4 * step) {
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned i = i0 + u * step + lane;
            v[u] = i < n ? load_piece<DENSE>(W, i, per_row, ldw) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned i = i0 + u * step + lane;
            uint32_t m = absmax16(v[u]);
#pragma unroll
            for (int o = LPG / 2; o; o >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
            if (i < n && (lane % LPG) == 0) {
                const float a = __uint_as_float(m << 16);
                bad |= (m >= 0x7F80u);
                const unsigned gi = i / LPG;
                if (MODE == AAAC_INT4) {
                    const uint32_t b = int4_scale_bits(a);
                    reinterpret_cast<uint16_t*>(scales)[gi] = (uint16_t)b;
                    rinv[gi] = __frcp_rn(__uint_as_float(b << 16));
                } else {
                    reinterpret_cast<uint8_t*>(scales)[gi] = (uint8_t)nvfp4_scale_code(a, d6, inv6);
                }
            }
        }
    }
    if (bad) {
        atomicOr(&ctrl->nonfinite, 1u);
        if (dev_status) atomicOr(dev_status, AAAC_DEV_NONFINITE);
    }
}

// The same pass that also counts the quantile start's histogram (Eq. 9-10 need order statistics of all
// w~ = fl32(w * fl32(1/s)); their first step is a 16384-bin histogram): every lane of a group holds the
// group's maximum after the butterfly, forms the scale and its reciprocal itself -- with exactly the
// expressions the later passes use -- and bins its eight normalised weights into the block's
// shared-memory histogram, which is merged into the global one at the end.
constexpr int kHistBlocksPerSM = 2;
template <int MODE, bool DENSE>
__global__ void __launch_bounds__(512, kHistBlocksPerSM)
scales_hist_kernel(const uint16_t* __restrict__ W, unsigned n, unsigned per_row, int64_t ldw, void* __restrict__ scales,
                   float* __restrict__ rinv, float* __restrict__ tensor_scale, Ctrl* ctrl, uint32_t* dev_status,
                   uint32_t* __restrict__ hist) {
    constexpr int G = MODE == AAAC_INT4 ? 128 : 16;
    constexpr int LPG = G / 8;                         // lanes per group
    extern __shared__ uint32_t sm[];                   // kQBins counters
    chain_next();
    for (int i = threadIdx.x; i < kQBins; i += blockDim.x) sm[i] = 0;
    chain_wait();
    const int lane = threadIdx.x & 31;
    const unsigned step = gridDim.x * blockDim.x;

    float s_t = 1.f, d6 = 6.f, inv6 = 1.f;
    if (MODE == AAAC_NVFP4) {
        const float A = __uint_as_float(ctrl->absmax_bits);
        s_t = (A == 0.f) ? 1.f : __fdiv_rn(A, 2688.f);
        if (s_t < 0x1p-96f) s_t = 0x1p-96f;
        d6 = __fmul_rn(6.f, s_t);
        inv6 = __frcp_rn(d6);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctrl->s_t = s_t;
        if (tensor_scale) tensor_scale[0] = s_t;
    }
    __shared__ float rl[128];                          // fl32(1 / s) per E4M3 code, or per mantissa of a BF16 scale (bf16_rcp)
    if (threadIdx.x < 128)
        rl[threadIdx.x] = MODE == AAAC_NVFP4 ? __frcp_rn(__fmul_rn(e4m3_value(threadIdx.x), s_t)) : bf16_rcp_entry(threadIdx.x);
    __syncthreads();
    bool bad = false;
    for (unsigned i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); i0 < n; i0 += 4 * step) {
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned i = i0 + u * step + lane;
            v[u] = i < n ? load_piece<DENSE>(W, i, per_row, ldw) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned i = i0 + u * step + lane;
            uint32_t m = absmax16(v[u]);
#pragma unroll
            for (int o = LPG / 2; o; o >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
            if (i >= n) continue;
            const float a = __uint_as_float(m << 16);
            bad |= (m >= 0x7F80u);
            float r;                                   // fl32(1 / s), as the later passes form it
            if (MODE == AAAC_INT4) {
                const uint32_t b = int4_scale_bits(a);
                r = bf16_rcp(rl, b);
                if ((lane % LPG) == 0) {
                    reinterpret_cast<uint16_t*>(scales)[i / LPG] = (uint16_t)b;
                    rinv[i / LPG] = r;
                }
            } else {
                const uint32_t q = nvfp4_scale_code(a, d6, inv6);
                r = rl[q];
                if ((lane % LPG) == 0) reinterpret_cast<uint8_t*>(scales)[i / LPG] = (uint8_t)q;
            }
            uint32_t bin[8];
            qbins(v[u], r, bin);
#pragma unroll
            for (int j = 0; j < 8; ++j) atomicAdd(&sm[bin[j]], 1u);
        }
    }
    if (bad) {
        atomicOr(&ctrl->nonfinite, 1u);
        if (dev_status) atomicOr(dev_status, AAAC_DEV_NONFINITE);
    }
    __syncthreads();
    // every block starts elsewhere, so that they do not meet on the same counters
    const unsigned first = threadIdx.x + blockIdx.x * blockDim.x;
    for (unsigned k = 0; k < kQBins; k += blockDim.x) {
        const unsigned i = (first + k) % kQBins;
        if (sm[i]) atomicAdd(&hist[i], sm[i]);
    }
}

}  // namespace

cudaError_t launch_scales(const uint16_t* W, int64_t N, int64_t K, int64_t ldw, int mode, void* scales,
                          float* tensor_scale, uint32_t* dev_status, const Workspace& ws, cudaStream_t st, bool with_hist) {
    const int blocks = sm_count() * 8;
    const bool dense = ldw == K;
    const unsigned n = (unsigned)(N * (K / 8)), per_row = (unsigned)(K / 8);       // (layers are below 2^32 elements)
    cudaError_t e = cudaSuccess;
    if (mode == AAAC_NVFP4) {
        note_launch();
        if ((e = launch_chained(dense ? absmax_kernel<true> : absmax_kernel<false>, blocks, 256, 0, st, W, n, per_row, ldw, ws.ctrl, dev_status)) != cudaSuccess) return e;
    }
    note_launch();
    float* const rinv = mode == AAAC_NVFP4 ? nullptr : ws.rinv;
    if (!with_hist) {
        auto kern = mode == AAAC_NVFP4 ? (dense ? scales_kernel<AAAC_NVFP4, true> : scales_kernel<AAAC_NVFP4, false>)
                                       : (dense ? scales_kernel<AAAC_INT4, true> : scales_kernel<AAAC_INT4, false>);
        return launch_chained(kern, blocks, 256, 0, st, W, n, per_row, ldw, scales, rinv, tensor_scale, ws.ctrl, dev_status);
    }
    static std::atomic<size_t> ready[4][kMaxDevices];
    const size_t smem = kQBins * sizeof(uint32_t);
    auto kern = mode == AAAC_NVFP4 ? (dense ? scales_hist_kernel<AAAC_NVFP4, true> : scales_hist_kernel<AAAC_NVFP4, false>)
                                   : (dense ? scales_hist_kernel<AAAC_INT4, true> : scales_hist_kernel<AAAC_INT4, false>);
    if ((e = allow_smem(kern, smem, ready[2 * (mode == AAAC_NVFP4) + dense])) != cudaSuccess) return e;
    return launch_chained(kern, sm_count() * kHistBlocksPerSM, 512, smem, st, W, n, per_row, ldw, scales, rinv, tensor_scale, ws.ctrl, dev_status, ws.qhist);
}

}  // namespace aaac
