// Shared device helpers and launcher declarations of the AAAC sm_100a library.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/aaac.h"

namespace aaac {

constexpr int kM = 16;            // entries per table
constexpr int kNBP = 30;          // merged breakpoints: 15 midpoints of T0 + 15 of T1
constexpr int kNJ = 31;           // merged intervals
constexpr int kPartStride = 2;    // doubles per block partial of the pack pass
constexpr int kMaxBlocks = 2048;  // upper bound on its grid
constexpr int kQBins = 16384;     // first-level histogram bins of the quantile selection
constexpr int kQReq = 64;         // order statistics requested (2 per table entry)
constexpr int kActMaxSplits = 128;  // row strips of the activation statistics

// ---- control block at the start of the workspace (device memory) ----
// It, the fit's sum buffers and the start's histogram follow one another in the workspace, so that one
// memset brings them to zero at the start of a fit.
struct Ctrl {
    double T[2 * kM];               // current tables (double between rounds)
    float reach;                    // INIT_USER: (how far from an entry a weight can be / 16) squared, 1 or more
    float s_t;                      // NVFP4 tensor scale
    uint32_t absmax_bits;           // layer max |w| as float bits (atomicMax on non-negative floats)
    uint32_t nonfinite;             // set if a non-finite weight was seen
    // the incremental rounds: the tables and centre constants of the pass they start from, its sums, and where they end
    double keep_T[2 * kM], keep_sx[2 * kM], keep_sw[2 * kM];
    double keep_q;                  // that pass's objective
    float keep_c[2 * kM];
    uint32_t keep_ok;               // its tables were in order
    uint32_t next_round, passes;    // the first pass of the fit not done; passes made so far (the sum buffers rotate per pass)
    uint32_t first_incremental, end_incremental;    // passes first .. end - 1 of the fit were incremental
    uint32_t abort;                 // set when a block's wait for the totals of a pass ran out
    // quantile selection
    double frac[2 * kM];            // interpolation fraction per table entry
    float rank_val[kQReq];          // selected order statistics
    uint32_t req_slot[kQReq];       // slot of each request
    unsigned long long req_local[kQReq];   // rank inside the slot's list
    uint32_t nslots;
    unsigned long long slot_off[kQReq + 1];
    uint32_t slot_fill[kQReq];
    uint32_t slot_over[kQReq];      // the slot's candidates did not fit the list: only their smallest and largest key are kept
    uint32_t slot_kmin[kQReq], slot_kmax[kQReq];
    uint32_t scratch_short;         // an order statistic could not be found within the scratch given
    // pack results, and the counter of finished blocks that the selection and pack kernels use (zero between them)
    double pack_err[2];
    unsigned long long pack_stats[4];
    uint32_t done;
};

constexpr int kFitAccWords = 3 * (2 * kM + 1) * 16;     // the fit rounds' sum buffers (see fit.cu)

struct Workspace {
    Ctrl* ctrl;
    unsigned long long* acc; // [kFitAccWords]
    uint32_t* qhist;         // [kQBins]
    double* part;            // [kMaxBlocks][kPartStride]: the pack pass's block partials
    float* rinv;             // [N*K/g]  INT4 reciprocal scales (one element in NVFP4 mode)
    float* I;                // [K] importance computed from X
    double* act_part;        // row strip partials of the activation statistics
    uint8_t* qslot_of_bin;   // [kQBins]
    uint32_t* qlist;         // [qcap] candidates of the quantile selection; afterwards the fit's selection bits [N][ceil(K/256)]
    size_t qcap;             // entries of qlist
    size_t bytes;
    size_t zero_bytes(bool with_hist) const {
        return (size_t)(reinterpret_cast<char*>(qhist) - reinterpret_cast<char*>(ctrl)) + (with_hist ? sizeof(uint32_t) * kQBins : 0);
    }
};

// ---- formats ----
__device__ __forceinline__ float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xFFFF0000u); }

__device__ __forceinline__ uint32_t f32_to_bf16_rne(float f) {
    uint32_t u = __float_as_uint(f);
    u += 0x7FFFu + ((u >> 16) & 1u);
    return u >> 16;
}

// E4M3 (no infinities, 0x7F = NaN): value of a code with the sign bit already removed
__device__ __forceinline__ float e4m3_value(uint32_t c) {
    uint32_t e = (c >> 3) & 15u, m = c & 7u;
    return e ? __uint_as_float(((e + 120u) << 23) | (m << 20)) : (float)m * 0.001953125f;
}

// nearest-even E4M3 code of a finite x >= 0, saturating at 448 (0x7E)
__device__ __forceinline__ uint32_t e4m3_encode(float x) {
    if (!(x < 448.f)) return 0x7Eu;
    if (x < 0.015625f) return (uint32_t)__float2int_rn(x * 512.f);   // subnormal step 2^-9; 8 -> 2^-6
    uint32_t u = __float_as_uint(x);
    u += 0x7FFFFu + ((u >> 20) & 1u);
    u = (u >> 20) - 960u;                                            // rebias 127 -> 7
    return u > 0x7Eu ? 0x7Eu : u;
}

// Packed pairs of FP32 values in one 64-bit register and the two-wide FP32 instructions of
// sm_100 on them (each half is rounded exactly like the scalar instruction).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ float lo2(uint64_t v) { float lo, hi; unpack2(v, lo, hi); return lo; }
__device__ __forceinline__ float hi2(uint64_t v) { float lo, hi; unpack2(v, lo, hi); return hi; }
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t fma2_rd(uint64_t a, uint64_t b, uint64_t c) {      // rounded down
    uint64_t r;
    asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// The bins floor(1024 w~ + 8192) of the quantile start's histogram for a lane's eight normalised weights
// w~ = fl32(w r): one multiply-add rounded down onto 1.5 * 2^23 (where floats are spaced by 1) leaves the integer
// in the low mantissa bits.  Two weights per instruction.  |w~| < 8 by the scale rules; in a group that holds a NaN
// it may be anything, and the mask keeps it inside the table.  The pass that counts the bins and the one that
// collects their weights both take them from here: a weight that they placed differently would have no room in its list.
__device__ __forceinline__ void qbins(const uint4& v, float r, uint32_t (&bin)[8]) {
    constexpr float kAdd = 8192.f + 12582912.f;
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    const uint64_t rr = pack2(r, r);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint64_t t = fma2_rd(mul2(pack2(bf16_lo(w[j]), bf16_hi(w[j])), rr), pack2(1024.f, 1024.f), pack2(kAdd, kAdd));
        bin[2 * j] = __float_as_uint(lo2(t)) & (uint32_t)(kQBins - 1);
        bin[2 * j + 1] = __float_as_uint(hi2(t)) & (uint32_t)(kQBins - 1);
    }
}

// fl32(1 / s) of a positive BF16 scale, from fl32(1 / (1 + m / 128)) per mantissa m: a power of two more does
// not change the rounding (scales are 2^-126 or more; that of a group with an infinite weight is infinite, and 0 here).
__device__ __forceinline__ float bf16_rcp(const float* lut, uint32_t b) {
    return __fmul_rn(lut[b & 0x7Fu], __uint_as_float((uint32_t)max(254 - (int)((b >> 7) & 0xFFu), 0) << 23));
}
__device__ __forceinline__ float bf16_rcp_entry(uint32_t m) { return __frcp_rn(1.f + (float)m * 0.0078125f); }

// The passes before the fit take a layer as a list of 16-byte pieces (8 weights), piece i of a row-major
// layer in group i / (g / 8): without gaps between the rows (DENSE) neither rows nor columns need to be
// known, which is half of such a pass's instructions; with gaps the row is found by a division.
template <bool DENSE>
__device__ __forceinline__ uint4 load_piece(const uint16_t* __restrict__ W, unsigned i, unsigned per_row, int64_t ldw) {
    if (DENSE) return __ldg(reinterpret_cast<const uint4*>(W) + i);
    const unsigned row = i / per_row;
    return __ldg(reinterpret_cast<const uint4*>(W + row * ldw + (i - row * per_row) * 8u));
}

// largest float <= d
__device__ __forceinline__ float f32_round_down(double d) { return __double2float_rd(d); }

// ---- launchers (each enqueues on `st` and returns the launch status) ----
cudaError_t launch_act_stats(const uint16_t* X, int64_t T, int64_t K, int64_t ldx, float* I, int accumulate,
                             uint32_t* dev_status, const Workspace& ws, int64_t one_strip_rows, cudaStream_t st);
// the same in pieces: strips [first, first + count) of the plan, then the sum over the strips
struct ActPlan { int64_t rows; int strips; };
constexpr int64_t kActAlone = 128, kActBeside = 64;    // rows that make one strip (see act_stats.cu)
ActPlan act_plan(int64_t T, int64_t K, int max_splits, int64_t one_strip_rows);
cudaError_t launch_act_strips(const uint16_t* X, int64_t T, int64_t K, int64_t ldx, const ActPlan& plan, int first, int count,
                              float* I, int accumulate, uint32_t* dev_status, double* part, cudaStream_t st);
cudaError_t launch_act_finish(int64_t K, const ActPlan& plan, float* I, int accumulate, uint32_t* dev_status, const double* part,
                              cudaStream_t st);
// with_hist: the scales pass also counts the 16384-bin histogram of the normalised weights (the quantile
// start's first pass over W) into ws.qhist, which is zero before
cudaError_t launch_scales(const uint16_t* W, int64_t N, int64_t K, int64_t ldw, int mode, void* scales,
                          float* tensor_scale, uint32_t* dev_status, const Workspace& ws, cudaStream_t st, bool with_hist = false);
cudaError_t launch_init(const uint16_t* W, int64_t N, int64_t K, int64_t ldw, int mode, int init,
                        const void* scales, const float* T01_user, uint32_t* dev_status, const Workspace& ws, cudaStream_t st);
int act_splits_max(int64_t K);    // most row strips launch_act_stats uses for K input channels (sizes its partials)
// the rounds of several layers of one mode, up to eight in a launch
struct FitLayerArgs {
    const uint16_t* W;
    int64_t N, K, ldw;
    const void* scales;
    const float* I;
    double* err_trace;
    float* T01_out;          // where the fitted tables go as FP32 (written by the last launch), or null
    Workspace ws;
    const float* reach = nullptr;   // Ctrl::reach where the start tables are the caller's, else null
    bool twin_entries = false;      // a start table holds one value twice (the NVFP4 grid: 0)
};
cudaError_t launch_fit_rounds_batch(const FitLayerArgs* layers, int n, int mode, int sel_group, int n_outer, int n_inner,
                                    uint32_t* dev_status, cudaStream_t st);
cudaError_t launch_export_tables(float* T01, const Workspace& ws, cudaStream_t st);
// row0, row1: only these rows (row0 a multiple of 64; the launches of a layer in order, the last one, with row1 = N,
// hands the results out); the default is all of them.
// sigma_bits: null when the selection group is the scale group (sigma in the scale's sign bit)
cudaError_t launch_pack(const uint16_t* W, int64_t N, int64_t K, int64_t ldw, int mode, int sel_group, const float* I,
                        const float* T01_f32, uint16_t* T01_bf16, void* scales, const float* tensor_scale,
                        uint8_t* codes, uint8_t* sigma_bits, double* err_out, unsigned long long* stats,
                        const Workspace& ws, cudaStream_t st, int64_t row0 = 0, int64_t row1 = -1);
cudaError_t launch_dequant(const uint8_t* codes, const void* scales, const uint8_t* sigma_bits,
                           const float* tensor_scale, const uint16_t* Tb, int64_t N, int64_t K, int mode,
                           uint16_t* What, int64_t ldo, cudaStream_t st);

cudaError_t launch_prescale(const uint16_t* W, int64_t N, int64_t K, int64_t ldw, const float* a, uint16_t* Wout,
                            int64_t ldo, const float* I, float* Iout, uint32_t* dev_status, cudaStream_t st);

// Kernels of a call follow one another with a programmatic dependency: the next one's blocks are put on the
// SMs as the previous one's leave them and wait inside (chain_wait, before the kernel's first access to
// global memory), so that launching them is not added to the chain.  A kernel that waits for the previous
// grid's end has waited for everything before it too.
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// the next kernel of the chain may take its place on the SMs from here on
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Raises a kernel's dynamic shared memory limit, once per device.
constexpr int kMaxDevices = 64;
template <typename K>
cudaError_t allow_smem(K kern, size_t bytes, std::atomic<size_t> (&done)[kMaxDevices]) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < kMaxDevices && done[dev].load(std::memory_order_relaxed) >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && dev >= 0 && dev < kMaxDevices) done[dev].store(bytes, std::memory_order_relaxed);
    return e;
}

// the row ranges in which the host-buffer call packs a layer, so that the codes of one travel while the next is packed
constexpr int kPackRanges = 4;
inline int64_t pack_range_rows(int64_t N) { return ((N + kPackRanges - 1) / kPackRanges + 63) / 64 * 64; }

int sm_count();
void note_launch(int n = 1);      // counts kernel launches (aaac_launch_count)
void set_fit_wait(int extra_arrivals, unsigned spin_limit);   // knobs of the fit rounds' bounded wait (aaac_debug_fit_wait)

}  // namespace aaac
