// Dequantisation (Eq. 5): w^ = T_sigma[c] * s, with sigma the sign bit of the stored scale (or,
// when the selection group is 16 inside a scale group of 128, the group's bit of the separate
// selection bytes) and s the scale's magnitude (times the tensor scale for NVFP4).  A pure stream: 0.5 byte of codes and a
// scale per group in, 2 bytes out per weight.  A thread expands one 32-bit word of codes (8 weights)
// into one 128-bit store, so a warp's loads and stores are contiguous.
//
// Codes, scales and selection bytes are dense, so the position of a word in the whole layer gives
// its group and selection byte by a shift; only an output with gaps between its rows needs the
// row.  Four words per thread and step are in flight, those of the next step loaded before this
// step's are expanded.  The tables stand in shared memory once per lane (a lookup by 32 different
// codes then costs one bank cycle instead of about three, and eight of them a word were what the
// kernel waited for).  14336 x 4096 NVFP4: 35.1 -> 28.6 us
// (4.3 -> 5.3 TB/s); 4096 x 4096 INT4 14.6 -> 9.7 us.
#include "internal.cuh"

namespace aaac {

namespace {

constexpr int kDqThreads = 256;
constexpr int kDqWords = 4;              // words of codes per thread and step
constexpr int kDqBlocksPerSM = 6;

template <int MODE, bool SEP, bool GAPS>
__global__ void __launch_bounds__(kDqThreads, kDqBlocksPerSM)
dequant_kernel(const uint32_t* __restrict__ codes, const void* __restrict__ scales,
               const uint8_t* __restrict__ sigma_bits, const float* __restrict__ tensor_scale, const uint16_t* __restrict__ Tb,
               int64_t words, unsigned per_row, uint16_t* __restrict__ What, int64_t ldo) {
    constexpr int kGroupShift = MODE == AAAC_INT4 ? 4 : 1;          // words of a scale group, as a shift
    __shared__ float T[2 * kM][32];
    __shared__ float slut[128];
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t step = (int64_t)gridDim.x * (kDqThreads * kDqWords);
    int64_t w0 = (int64_t)blockIdx.x * (kDqThreads * kDqWords) + tid;
    uint32_t word[kDqWords], sb[kDqWords], sg[kDqWords];
    auto fetch = [&](int64_t at) {
#pragma unroll
        for (int u = 0; u < kDqWords; ++u) {
            const int64_t w = at + u * kDqThreads;
            if (w < words) {
                word[u] = __ldcs(codes + w);
                sb[u] = MODE == AAAC_INT4 ? (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(scales) + (w >> kGroupShift))
                                          : (uint32_t)__ldg(reinterpret_cast<const uint8_t*>(scales) + (w >> kGroupShift));
                if (SEP) sg[u] = __ldg(sigma_bits + (w >> 4));
            }
        }
    };
    chain_next();
    chain_wait();
    fetch(w0);
    for (int i = tid; i < 2 * kM * 32; i += kDqThreads) T[i >> 5][i & 31] = __uint_as_float((uint32_t)Tb[i >> 5] << 16);
    if (MODE == AAAC_NVFP4 && tid < 128) slut[tid] = __fmul_rn(e4m3_value(tid), tensor_scale[0]);
    __syncthreads();
    while (w0 < words) {
        uint32_t cw[kDqWords], cb[kDqWords], cg[kDqWords];
#pragma unroll
        for (int u = 0; u < kDqWords; ++u) { cw[u] = word[u]; cb[u] = sb[u]; if (SEP) cg[u] = sg[u]; }
        fetch(w0 + step);
#pragma unroll
        for (int u = 0; u < kDqWords; ++u) {
            const int64_t w = w0 + u * kDqThreads;
            if (w >= words) break;
            uint32_t sigma;
            float s;
            if (MODE == AAAC_INT4) {
                sigma = cb[u] >> 15;
                s = __uint_as_float((cb[u] & 0x7FFFu) << 16);
            } else {
                sigma = cb[u] >> 7;
                s = slut[cb[u] & 0x7Fu];
            }
            if (SEP) sigma = (cg[u] >> ((w >> 1) & 7)) & 1u;
            const float* Ts = &T[sigma * kM][lane];
            uint32_t o[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                // two products rounded to BF16 (nearest even) and packed by one conversion instruction
                const float lo = __fmul_rn(Ts[((cw[u] >> (8 * j)) & 15u) * 32], s);
                const float hi = __fmul_rn(Ts[((cw[u] >> (8 * j + 4)) & 15u) * 32], s);
                asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(o[j]) : "f"(hi), "f"(lo));
            }
            int64_t at = w * 8;
            if (GAPS) {
                // (with selection bytes, a 32-bit division where it will do: 14336 x 4096 38.5 -> 37.9 us; without, that is 1 % slower)
                const int64_t row = SEP && words <= 0xFFFFFFFFll ? (int64_t)((uint32_t)w / per_row) : w / per_row;
                at = row * ldo + (w - row * per_row) * 8;
            }
            __stcs(reinterpret_cast<uint4*>(What + at), make_uint4(o[0], o[1], o[2], o[3]));
        }
        w0 += step;
    }
}

template <int MODE, bool SEP>
cudaError_t launch_dequant_variant(const uint8_t* codes, const void* scales, const uint8_t* sigma_bits, const float* tensor_scale,
                                   const uint16_t* Tb, int64_t N, int64_t K, uint16_t* What, int64_t ldo, cudaStream_t st) {
    const int64_t words = N * (K / 8);
    int64_t blocks = (words + kDqThreads * kDqWords - 1) / (kDqThreads * kDqWords);
    const int64_t cap = (int64_t)sm_count() * kDqBlocksPerSM;
    if (blocks > cap) blocks = cap;
    note_launch();
    auto kern = ldo == K ? dequant_kernel<MODE, SEP, false> : dequant_kernel<MODE, SEP, true>;
    return launch_chained(kern, (unsigned)blocks, kDqThreads, 0, st, reinterpret_cast<const uint32_t*>(codes), scales, sigma_bits,
                          tensor_scale, Tb, words, (unsigned)(K / 8), What, ldo);
}

}  // namespace

cudaError_t launch_dequant(const uint8_t* codes, const void* scales, const uint8_t* sigma_bits,
                           const float* tensor_scale, const uint16_t* Tb, int64_t N, int64_t K, int mode,
                           uint16_t* What, int64_t ldo, cudaStream_t st) {
    if (mode == AAAC_INT4 && sigma_bits)
        return launch_dequant_variant<AAAC_INT4, true>(codes, scales, sigma_bits, tensor_scale, Tb, N, K, What, ldo, st);
    if (mode == AAAC_INT4)
        return launch_dequant_variant<AAAC_INT4, false>(codes, scales, nullptr, tensor_scale, Tb, N, K, What, ldo, st);
    return launch_dequant_variant<AAAC_NVFP4, false>(codes, scales, nullptr, tensor_scale, Tb, N, K, What, ldo, st);
}

}  // namespace aaac
