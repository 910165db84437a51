// The fit rounds (Algorithm 1 lines 6-16).  With n_inner = 1 a round is the assignment step
// (Eq. 8) and the activation-weighted centroid update (Eq. 11) in a single pass over W, and all
// rounds of a layer run in ONE persistent kernel (one block per SM, cooperative launch): after
// its pass every block adds its sums, as fixed-point integers of two 47-bit limbs, into 65 global
// accumulators; every 64-bit accumulator word also counts, in its upper bits, the blocks that have
// added to it, so a block knows that a total is complete by reading the total itself -- no separate
// barrier, no fence between the sums and an arrival counter -- and every block ends up with the
// same new tables without a relaunch (integer addition does not depend on the order in which the
// blocks arrive, so the result is bitwise reproducible).  The wait for the totals is bounded: if
// it runs out, the kernel sets AAAC_DEV_TIMEOUT in the device status word and returns.
// What a round costs besides its pass (block sums, exchange, new tables) is latency: about 8.5k
// cycles, kept short by leaving the small steps to one warp that needs no block barrier, by
// lookups and conversions chosen for it (see below), and by having the first rows of the next pass
// in flight, and the bins being cleared, meanwhile.  A pass of a 512 x 512 layer took 11.4 us with 19k cycles of it and whole
// items, 5.2 us now; 4096 x 4096, 27.4 -> 23.3 us.
// (NVFP4 layers of enough units and rounds leave most of their rounds to the incremental ones of fit_delta.cuh, and run as
// four launches: see can_increment.)
// With n_inner > 1 the assignment pass (which is also the first inner iteration) stores the
// selection bits, one word per row and 256-column slab, and the remaining n_inner - 1 inner
// iterations are passes of a second instance of the kernel that reads those bits instead of
// forming the two errors; both instances share everything else.  The tables are put in
// ascending order after every pass: in one dimension a centroid update keeps an ascending table
// ascending (ties aside), and the cells depend on the entries' values only, so this equals
// sorting after the last inner iteration.
//
// Per weight the kernel needs (a) the interval J of the merged breakpoint list of both tables
// that holds w~ = fl32(w * r) (Eq. 2) -- J fixes the nearest entry of T0 and of T1 (Eq. 4) --
// (b) its two weighted squared errors, and (c) one accumulation into the centroid sums of cell
// (sigma, J).
//
// (a) Interval.  NB uniform bins on (-8, 8) (512 of width 1/32): with s = NB / 16 the mantissa of
//     fl32(s x + NB / 2 + 1.5 * 2^(23-k)) holds (s x + NB / 2) * 2^k rounded to an integer; masked,
//     it is the byte offset bin * 2^k of the bin's table entry (2^k = bytes per bin over all
//     copies), bin = floor of s x + NB / 2 after rounding to a multiple of 2^-k.
//     A table gives per bin either {P, Q} of (b) itself, where no breakpoint lies in the bin (four
//     fifths of the weights), or {thr, address}: thr is the one breakpoint inside, and the address
//     names {P, Q} of the interval below it, the row after it that of the interval above.  Only the
//     lanes with such a bin look up a second time, and a shared-memory load of a few lanes costs one
//     cycle where a full 8-byte one costs two (9.8 -> 8.9 wavefronts per 32 weights; the shared-memory
//     pipe was 93 % busy during a pass).
//     Breakpoints are the rounded-down FP32 midpoints, for which x > thr <=> x > midpoint, so the
//     interval is exact.  A bin that holds two or more breakpoints names a poisoned row (J = 31)
//     whose entries are NaN: the group falls through to the exact path below, which searches J
//     directly.  (Fitted tables keep their merged breakpoints apart -- the two codebooks
//     specialise -- so such bins are rare outside degenerate starts.)
// (b) Selection.  {P, Q} are the FP32 roundings of the nearest entries of T0
//     and T1 on interval J, moved by at most 8 units in the last place so that the low 4 mantissa
//     bits equal the entry's index (so the
//     same 8 bytes also say which cell the weight falls into).  u_r = x - T_r,
//     E_r = sum_k I_k u_r^2 (Eq. 8), summed per lane and over the lanes of the group by shuffles;
//     sigma = [E1 < E0].
//     Rounding: the constants differ from the entries by at most eta = 17 * 2^-24 max|T|, so
//     |E_r - E_r,exact| <= 2^-24 * 16 E_r + 2 eta sum I |u_r| and
//     sum I |u_r| <= sqrt(sum I * E_r).  Groups with
//     |E0 - E1| <= 2^-24 (16 (E0 + E1) + 2.83 * 17 max|T| sqrt(sum I (E0 + E1))) (and NaN) are
//     re-evaluated in double with the exact entries, so sigma is the double-precision decision
//     (the kernel tests against the slightly larger bound that sqrt(a b) <= a / 16 + 4 b gives,
//     which needs one multiply-add per group).  The errors are summed by pairs of columns
//     (mul / fma.f32x2).
// (c) Centroid sums, centred.  Lane-private shared-memory bins [sigma][entry] hold
//     (sum I (x - c), sum I) with c the constant of (b) for the entry the weight is assigned to,
//     so the new entry is c + sum I (x - c) / sum I.  The residual sums are small and of mixed
//     sign, which keeps the FP32 accumulation error some 20 times below that of sum I x.  Within
//     a block: no atomics, fixed order.  Across blocks: integer atomics (see above).  After the
//     barrier the centroids are formed (entries of empty cells keep their value) and
//     sorted; block 0 stores the Eq. 8 objective of the round (sum over groups of the smaller
//     error) and, after the last round, the tables.
//
// Tables in shared memory are replicated against bank conflicts: the per-bin table and the
// {P, Q} table 16 times (lane l uses copy l mod 16, so the 16 lanes that share a wavefront of an
// 8-byte load never collide; an address in a bin's entry names the same copy), the bins once per lane.
//
// Thread mapping.  A block of 16 warps works on items of 64 rows (32 or 16 in layers that have too
// few items for the blocks) x 256 columns, dealt to
// blocks as contiguous ranges (slab-major), so every sum has a fixed order and results are
// bitwise reproducible.  A warp takes 4 rows; each lane 8 adjacent columns (one 128-bit load
// per row), so its eight importances stay in registers.  A group is 2 lanes (g = 16) or 16
// lanes (g = 128).  A row's registers are refilled from the next item right after the row is unpacked.
#include <algorithm>

#include "lookup.cuh"

namespace aaac {

namespace {

struct FitParams {
    const uint16_t* W;
    int64_t N, K, ldw;
    const uint8_t* scales;        // NVFP4 scale bytes
    const float* rinv;            // INT4 reciprocal scales
    const float* I;
    const float* reach;           // what the caller's start tables add to the bound of the sums (a factor), or null
    Ctrl* ctrl;
    unsigned long long* acc;      // [3][kAccBuffer] words: fixed-point sums over the blocks, one buffer per pass in rotation
    double* err_trace;            // [n_rounds] or null
    float* T01_out;               // [2][16] or null: the tables after the launch's last pass, as FP32
    uint32_t* dev_status;         // or null
    uint32_t* sigw;               // [N][slabs]: selection bits of a row's 256-column slab, bit = lane (n_inner > 1)
    int n_rounds;                 // passes over W in this launch (incremental rounds, kRest: of the fit so far, with this launch's)
    int trace_base;               // err_trace index of this launch's first assignment pass
    unsigned bar_base;            // passes of the layer's earlier launches (the sum buffers rotate per pass)
    unsigned arrivals;            // blocks whose sums a total must hold before it is read (the grid size)
    unsigned spin_limit;          // polls of a total before the wait is given up
    int rows;                     // rows per warp of an item: 4, or 2 or 1 for layers that have too few items of 4
    int items, per_block, nrb;    // items of 16 * rows rows x 256 columns, items per block, row blocks per slab
    int tail_item0, tail_quarters;   // items from tail_item0 on are dealt out a quarter (one row per warp) per block
    uint32_t* kept;               // [N][K / 16], the same memory (kKeep and the incremental rounds): per 16 adjacent weights, bit 2 j the low bit
                                  // of the index of weight j's entry in the table its group has chosen, bit 1 that choice
    int n_inner;                  // incremental rounds: passes per round
    int n_total;                  // kInnerRest: passes of the whole fit
    bool from_kept;               // kInnerRest: the selection stands in the kept words, and the round that they belong to is finished
};

constexpr uint32_t kLut1At = 65536;                    // shared address of the bin table (see fit_rounds_body)
constexpr int kFitWarps = 16;
constexpr int kMaxFitBlocks = 255;                    // grid limit: the limbs' sums have 8 bits of room, the arrivals are counted in the 9 above
constexpr int kLimbs = 2;                             // a sum is a fixed-point number of two 47-bit limbs
constexpr int kLimbBits = 47;
constexpr double kLimb = (double)(1ll << kLimbBits);
constexpr int kSumBits = 2 * kLimbBits - 1;           // a block's sum as an integer is below 2^kSumBits in magnitude
constexpr unsigned kDefaultSpinLimit = 1u << 23;      // polls of several hundred ns each: seconds
// An accumulator buffer: per cell the limbs of the residual sum and of the weight sum, 32 bytes next to one
// another (four lanes add them with one request, a reader takes them with two loads), cells 128 bytes apart
// so that the blocks' atomics on different cells do not queue behind one another; then the objective's.
constexpr int kAccStride = 16;
constexpr int kAccBuffer = (kCells + 1) * kAccStride;  // 64-bit words of one pass's buffer
constexpr int kCountShift = 55;                       // an accumulator word: limb sum below, arrivals above
constexpr unsigned long long kLimbMask = (1ull << kCountShift) - 1ull;
constexpr unsigned long long kOneArrival = 1ull << kCountShift;
constexpr long long kTopBias = 1ll << (kLimbBits - 1);   // added to the (signed) top limb so that every block adds a non-negative number

__device__ __forceinline__ void ld_relaxed_2xu64(const unsigned long long* p, unsigned long long& a, unsigned long long& b) {
    asm volatile("ld.relaxed.gpu.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ unsigned ld_relaxed_u32(const unsigned* p) {
    unsigned v;
    asm volatile("ld.relaxed.gpu.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// process-wide knobs of the wait (aaac_debug_fit_wait): extra arrivals a total must show before it is
// taken (0 in normal use; 1 makes every wait run out) and the poll limit
int g_extra_arrivals = 0;
unsigned g_spin_limit = kDefaultSpinLimit;

// Near-tie groups are not decided inside the row pipeline: their lanes send the row's centred
// terms to a spare bin slot that nobody reads, the group goes on a short per-warp list, and
// resolve_deferred (after the pass's items, or when the list fills up) decides it in double and
// adds its weights to the bins.  That keeps the hot loop free of the slow path, whose latency every
// pass would otherwise pay on the warp that drew the most near-ties.
constexpr int kDeferCap = 96;                         // list entries per warp: {row, first column of the group}
constexpr int kBinSlots = kCells + 1;                 // [sigma][entry] and the spare slot
constexpr int kSpareSlot = kCells;

__device__ __forceinline__ void sts_u2(uint32_t addr, uint32_t a, uint32_t b) {
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" :: "r"(addr), "r"(a), "r"(b) : "memory");
}

// A launch runs passes of one kind.  kRounds: assignment passes, each also the (only) inner
// iteration of its round -- the n_inner = 1 procedure, all rounds of a layer in one launch.
// kAssignKeep: the same pass, which also stores the selection bits.  kInner: further inner
// iterations with the stored selection.  With n_inner > 1 a round is one kAssignKeep launch of a
// single pass followed by one kInner launch of n_inner - 1 passes.
// kKeep: one assignment pass with exact weight sums (collect_counts) that also stores, per 16 columns of a row, the low
// bits of the entries' indices and the selection; the passes after it are those of fit_delta.cuh.  (A launch of its own:
// with the first rounds in it, their bin updates paid for the choice of what to add, 14 us a pass of 16432 x 8192.)
// kRest: assignment passes again, as many as those have left: the last of the fit, whose sums are made anew for the
// tables that are handed out, and mostly no other.  With n_inner > 1 kInnerRest finishes the
// round in which they ended, with the selection that they kept, and one kAssignRest and one kInnerRest launch per further
// round make it, unless it is done.
enum PassKind { kRounds = 0, kAssignKeep = 1, kInner = 2, kKeep = 3, kRest = 4, kAssignRest = 5, kInnerRest = 6 };

__device__ __forceinline__ void add_term(uint32_t addr, float v) {
    float a;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(a) : "r"(addr) : "memory");
    asm volatile("st.shared.f32 [%0], %1;" :: "r"(addr), "f"(a + v) : "memory");
}
__device__ __forceinline__ void count_weight(uint32_t addr, uint32_t one) {
    asm volatile("red.shared.add.u32 [%0], %1;" :: "r"(addr), "r"(one) : "memory");
}

// Decides the listed selection groups in double (Eq. 8: each lane adds its weights' terms in index
// order, the lanes of the group are combined pairwise; a tie goes to table 0) and adds every weight
// to the calling lane's bins under the chosen table, with the arithmetic of the row pipeline
// (centred term I (x - c), c the chosen entry's centre constant).  Every lane of the warp calls;
// returns the sum of the groups' smaller errors in lane 0 (0 elsewhere).
struct DeferArgs {                // what the routine needs of the layer (passed by value: the kernel's
    const uint16_t* W;            // parameters themselves stay where they are)
    int64_t K, ldw;
    const uint8_t* scales;
    const float* rinv;
    const float* I;
    uint32_t* sigw;
    uint32_t* kept;
};
template <int MODE, int SEL, int KIND>
__device__ __noinline__ double resolve_deferred(const FitTables* S, const DeferArgs p, uint32_t list_addr, int count,
                                                uint32_t bins_lane, int lane) {
    constexpr int G = MODE == AAAC_INT4 ? 128 : 16;      // scale group
    constexpr int WPL = SEL >= 32 ? SEL / 32 : 1;        // weights per lane
    constexpr int ACTIVE = SEL / WPL;                    // lanes that hold weights of the group (32 or 16)
    constexpr int LPG = SEL / 8;                         // lanes of the group in the row pipeline
    const int K = (int)p.K, Gr = K / G, slabs = (K + 255) >> 8;
    double esum = 0.0;
    for (int e = 0; e < count; ++e) {
        uint32_t urow, ucol;
        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(urow), "=r"(ucol) : "r"(list_addr + (uint32_t)e * 8u));
        const int row = (int)urow, cg = (int)ucol;
        float xs[WPL], Is[WPL];
        int Js[WPL];
        double e0 = 0.0, e1 = 0.0;
        if (lane < ACTIVE) {
#pragma unroll
            for (int t = 0; t < WPL; ++t) {
                const int col = cg + lane * WPL + t;
                const uint32_t wb = p.W[(size_t)row * (size_t)p.ldw + col];
                const size_t gi = (size_t)row * (size_t)Gr + (uint32_t)col / G;
                const float rinv = MODE == AAAC_NVFP4 ? S->rlut[p.scales[gi] & 0x7Fu] : __ldg(p.rinv + gi);
                const float x = __fmul_rn(__uint_as_float(wb << 16), rinv);
                const float iv = __ldg(p.I + col);
                int J = 0;
#pragma unroll
                for (int step = 16; step; step >>= 1)      // number of breakpoints below x (sorted list)
                    if (J + step <= kNBP && S->bp[J + step - 1] < x) J += step;
                const double2 pq = S->PQ[J];
                const double xd = (double)x, id = (double)iv;
                const double d0 = __dsub_rn(xd, pq.x), d1 = __dsub_rn(xd, pq.y);
                e0 = __dadd_rn(e0, __dmul_rn(id, __dmul_rn(d0, d0)));
                e1 = __dadd_rn(e1, __dmul_rn(id, __dmul_rn(d1, d1)));
                xs[t] = x; Is[t] = iv; Js[t] = J;
            }
        }
#pragma unroll
        for (int o = ACTIVE / 2; o; o >>= 1) {
            e0 = __dadd_rn(e0, __shfl_xor_sync(0xFFFFFFFFu, e0, o));
            e1 = __dadd_rn(e1, __shfl_xor_sync(0xFFFFFFFFu, e1, o));
        }
        e0 = __shfl_sync(0xFFFFFFFFu, e0, 0);
        e1 = __shfl_sync(0xFFFFFFFFu, e1, 0);
        const bool sg = e1 < e0;
        uint32_t parity = 0;
        if (lane < ACTIVE) {
#pragma unroll
            for (int t = 0; t < WPL; ++t) {
                const float2 c2 = S->pq32[Js[t]];
                const float c = sg ? c2.y : c2.x;
                const uint32_t a = bins_lane + ((sg ? (uint32_t)kM : 0u) + (__float_as_uint(c) & kIdxMask)) * kSlotBytes;
                const float term = __fmul_rn(Is[t], __fsub_rn(xs[t], c));
                if (KIND == kKeep) {
                    // (the count belongs to the lane that has the column in the row pipeline)
                    static_assert(KIND != kKeep || WPL == 1, "a weight per lane");
                    const uint32_t col = (uint32_t)(cg + lane) & 255u;
                    add_term(a, term);
                    count_weight(a + ((col >> 3) - (uint32_t)lane) * 8u + 4u, 1u << (4 * (col & 7u)));
                } else {
                    float2 b = lds_bin(a);
                    b.x += term;
                    b.y += Is[t];
                    sts_bin(a, b);
                }
                if (KIND == kKeep) parity = __float_as_uint(c) & 1u;
            }
        }
        if (KIND == kKeep) {
            // the group's lanes put their bits together
            parity <<= 2 * (lane & 15);
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) parity |= __shfl_xor_sync(0xFFFFFFFFu, parity, o);
            if (lane == 0) p.kept[(size_t)row * (size_t)(K / 16) + (uint32_t)(cg / 16)] = parity | (sg ? 2u : 0u);
        }
        if (lane == 0) {
            esum += sg ? e1 : e0;
            if (KIND == kAssignKeep || KIND == kAssignRest) {
                // the stored selection bits of the row's slab: bit = lane of the row pipeline
                const uint32_t first = ((uint32_t)cg & 255u) >> 3;
                const uint32_t mask = (LPG >= 32 ? 0xFFFFFFFFu : ((1u << LPG) - 1u)) << first;
                uint32_t* wp = p.sigw + (size_t)row * (size_t)slabs + (cg >> 8);
                const uint32_t old = *wp;
                *wp = sg ? (old | mask) : (old & ~mask);
            }
        }
    }
    return esum;
}

// Integers of up to 51 bits travel to and from doubles by an addition (the 64-bit conversion instructions
// run at a small fraction of the double-precision rate).
constexpr double kIntMagic = 0x1.8p52;

struct FitShared {
    FitTables t;
    double wsum[kFitWarps][2 * kCells + 2];   // the warps' sums of a pass: residuals, weights, objective
    double fix_scale, fix_unscale;   // fixed-point scale of the sums over the blocks and its inverse
    int failed;
};

// Double value of FP32 bits times 2^-896: the float's fields moved into a double's (zeros and denormals
// included: their double is a denormal of the same scale, and double-precision hardware handles those at
// full speed).  Three integer instructions instead of the slow conversion; the caller multiplies its sum
// by 2^896.
__device__ __forceinline__ double scaled_double(float f) {
    const int u = __float_as_int(f);
    return __hiloint2double((u >> 3) & (int)0x8FFFFFFFu, u << 29);
}

// The two error sums of a group of LPG lanes, the same in each of them.  With 16 lanes the first step leaves one of
// the sums to either half (lane bit 3), so that a sum costs one exchange a step from then on: 5 exchanges and 4
// additions instead of 8 and 8 (an exchange takes a cycle of the shared-memory pipe; 14336 x 4096 INT4 74.3 -> 73.8
// us a round.  In the pack pass, which has that pipe to spare, the longer chain took 1 % more).
template <int LPG>
__device__ __forceinline__ void group_sums(float& e0, float& e1, int lane) {
    constexpr unsigned kAll = 0xFFFFFFFFu;
    if constexpr (LPG == 16) {
        const bool upper = (lane & 8) != 0;
        float v = (upper ? e1 : e0) + __shfl_xor_sync(kAll, upper ? e0 : e1, 8);
#pragma unroll
        for (int s = 4; s; s >>= 1) v += __shfl_xor_sync(kAll, v, s);
        const float other = __shfl_xor_sync(kAll, v, 8);
        e0 = upper ? other : v;
        e1 = upper ? v : other;
    } else {
#pragma unroll
        for (int s = LPG / 2; s; s >>= 1) {
            e0 += __shfl_xor_sync(kAll, e0, s);
            e1 += __shfl_xor_sync(kAll, e1, s);
        }
    }
}

// The weight sums of the pass that the incremental rounds start from.  They carry a cell's sum of I from round to round,
// and an error of it counts times the way its entry has gone since, where one of any other pass counts times the entry's
// movement in that pass.  FP32 sums in a lane's bins are not good enough for that: a lane's eight importances are the same
// in every row, so are their rounding errors (those of a massive channel's neighbours above all), and no number of rows
// averages them out: -1e-8 of the sum in every cell.  In this pass a bin's second word therefore counts the weights of the
// lane's eight columns, four bits each.  After every 12 rows, and before the slab changes, the block adds its warps'
// counts and multiplies them by the importances in double: warp w takes the cells 2 w and 2 w + 1, and their residuals
// too.  The bins are zero again behind it.  Every thread calls.
// Tables of one pass against 64-bit sums, 2-norm, 35520 x 1024 Student-t weights, pass 25: 3.4e-9 -> 1.7e-10 (a full
// pass: 1.2e-10); bins emptied into doubles after every item instead: 2.4e-10 to 5.6e-10.
constexpr int kCountedItems = 3;                      // items of four rows: 12 rows, a count has room for 15
static_assert(kCountedItems * kRowsPerWarp < 16, "four bits a count");
struct CountedSums { double x[2], y[2]; };            // a lane's part of two cells' sums, 2^-896 times
__device__ __noinline__ void collect_counts(CountedSums* const sums, const uint32_t low_at, const uint32_t high_at, const int n_low,
                                            const uint32_t warp_bytes, const float4 I0, const float4 I1, const int warp, const int lane) {
    const float I[8] = {I0.x, I0.y, I0.z, I0.w, I1.x, I1.y, I1.z, I1.w};
    __syncthreads();
    const uint32_t at = (uint32_t)(2 * warp) * kSlotBytes + (uint32_t)lane * 8u;
    double x[2] = {0.0, 0.0}, y[2] = {0.0, 0.0};
    uint32_t even[2] = {0u, 0u}, odd[2] = {0u, 0u};   // counts over the warps, a byte each (16 times 12 at most)
#pragma unroll 4
    for (int w = 0; w < kFitWarps; ++w) {
        const uint32_t a = at + (w < n_low ? low_at + (uint32_t)w * warp_bytes : high_at + (uint32_t)(w - n_low) * warp_bytes);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float2 b = lds_bin(a + c * kSlotBytes);
            sts_bin(a + c * kSlotBytes, make_float2(0.f, 0.f));
            x[c] += scaled_double(b.x);
            const uint32_t n = __float_as_uint(b.y);
            even[c] += n & 0x0F0F0F0Fu;
            odd[c] += (n >> 4) & 0x0F0F0F0Fu;
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const double Id = scaled_double(I[j]);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const uint32_t n = (((j & 1) ? odd[c] : even[c]) >> (8 * (j >> 1))) & 255u;
            // (n as a double: 2^52 + n has it in its low bits; no 0 * Inf in cells without the column)
            if (n) y[c] = __fma_rn(Id, __hiloint2double(0x43300000, (int)n) - 0x1p52, y[c]);
        }
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        sums->x[c] += x[c];
        sums->y[c] += y[c];
    }
    __syncthreads();
}

// SEL is the selection group size S (Sec. 3.1): the weights that share one codebook choice; the
// scale group g is fixed by the format.
// The passes of one layer, run by the nblk blocks bid = 0 .. nblk - 1 (a whole grid, or the part
// of a grid that a batch of layers gives to this layer).
template <int MODE, int SEL, int KIND>
__device__ __forceinline__ void fit_rounds_body(const FitParams& p, const unsigned bid, const unsigned nblk) {
    constexpr int NW = kFitWarps, NB = kNBins, REP = kRep;
    constexpr unsigned kAll = 0xFFFFFFFFu;
    constexpr int G = MODE == AAAC_INT4 ? 128 : 16;      // scale group
    constexpr int LPG = SEL / 8;                         // lanes per selection group
    constexpr int R = kRowsPerWarp;
    const int rows = p.rows;                             // rows per warp of an item (R or fewer)
    constexpr int NT = NW * 32;
    constexpr int kBinBytes = kBinSlots * kSlotBytes;        // per warp
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ FitShared sh;
    FitTables& S = sh.t;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr bool REST = KIND == kRest || KIND == kAssignRest || KIND == kInnerRest;
    const int passed = REST ? (int)p.ctrl->next_round : 0;
    int n_rounds = p.n_rounds, trace_base = p.trace_base;
    if (KIND == kRest) {
        n_rounds -= passed;
        trace_base += passed;
    }
    if (KIND == kAssignRest && passed != p.trace_base * p.n_inner) return;
    if (KIND == kInnerRest) {
        if (p.from_kept) n_rounds = passed < p.n_total && passed % p.n_inner ? p.n_inner - passed % p.n_inner : 0;
        else if (passed != p.trace_base * p.n_inner + 1) return;
    }
    if (REST && n_rounds <= 0) return;
    const unsigned bar_base = REST ? p.ctrl->passes : p.bar_base;

    // 32-bit shared addresses.  The bin table sits at a shared address that is a multiple of its own
    // span (64 KB), so that a lookup's address -- bin bits, the lane's copy and the table base -- is one
    // three-input logic instruction; the bins of the first warps fill the space below it, the other
    // warps' bins, the {P, Q} table and the near-tie lists follow it.  Slot offsets carry the address of
    // this lane's column of the {P, Q} table, so a lookup there needs no further arithmetic.
    static_assert(kLut1Bytes == (int)kLut1At, "the bin table spans exactly the alignment of its address");
    const uint32_t dyn_at = (uint32_t)__cvta_generic_to_shared(dyn);
    const uint32_t sm_base = (dyn_at + 255u) & ~255u;        // (a bin slot is 256 bytes: its lanes' offsets can be formed by xor)
    uint32_t dyn_size;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn_size));
    const uint32_t gap = kLut1At - sm_base;                                            // bytes of the dynamic region below the table
    const int n_low = min(NW, (int)(gap / (uint32_t)kBinBytes));                       // warps whose bins lie below the table
    const uint32_t hi_base = kLut1At + kLut1Bytes;
    const uint32_t lut2_addr = hi_base + (uint32_t)(NW - n_low) * kBinBytes;           // the {P, Q} table
    const uint32_t lists_at = lut2_addr + kLut2Bytes;
    if (sm_base > kLut1At || lists_at + NW * (kDeferCap * 8) > dyn_at + dyn_size) {
        // the layout does not fit the shared memory this launch was given (the same for every block, so
        // all of them leave before any of them waits): reported like a wait that ran out -- no valid result
        if (bid == 0 && threadIdx.x == 0 && p.dev_status) atomicOr(p.dev_status, AAAC_DEV_TIMEOUT);
        return;
    }
    const uint32_t lut1_or = kLut1At | ((lane & (REP - 1)) * 8);                        // table base | this lane's copy of a bin's entry; | bin * REP * 8
    const uint32_t bins_warp = warp < n_low ? sm_base + warp * kBinBytes : hi_base + (uint32_t)(warp - n_low) * kBinBytes;
    const uint32_t bins_lane = bins_warp + lane * 8;                                   // + cell * 256
    const uint32_t spare_lane = bins_lane + kSpareSlot * kSlotBytes;                   // sink of the near-tie groups' rows
    const uint32_t list_addr = lists_at + warp * (kDeferCap * 8);

    // 32-bit index arithmetic throughout (N, K < 2^31); only the final element offsets are 64-bit
    const int N = (int)p.N, K = (int)p.K;
    const int Gr = K / G;
    const int slabs = (K + 255) >> 8;
    // A block takes a contiguous range of whole items; what does not divide evenly (the items from
    // tail_item0 on) is dealt out one quarter item -- one row per warp -- per block, so that the
    // busiest block has at most a quarter item more than the others.
    const int it0 = (int)bid * p.per_block;
    const int it1 = min(p.tail_item0, it0 + p.per_block);
    const bool has_tail = (int)bid < p.tail_quarters;
    const int tail_item = p.tail_item0 + ((int)bid >> 2), tail_u = (int)bid & 3;
    static_assert(R == 4, "a tail quarter is one of the four rows of a warp");

    // Row registers of the item being processed; a row's registers are refilled with the same row
    // of the next item as soon as the row has been unpacked, so the load has about an item's time
    // to arrive and no second buffer is needed.  After the last item of a pass the next is the first
    // one again: its rows, and the importances as long as the slab stays the same, are there when the
    // next pass starts (a layer of one item per block waits for no load at all).
    uint4 v[R];
    uint32_t sc[R];           // NVFP4: scale byte; INT4: bits of the reciprocal scale
    uint32_t sgw[R];          // inner iteration: the row's stored selection bits
    constexpr bool INNER = KIND == kInner || KIND == kInnerRest;
    constexpr bool keep_sigma = KIND == kAssignKeep || KIND == kAssignRest;
    // (the selection's words per row, and a lane's bit: see FitParams)
    const bool from_kept = KIND == kInnerRest && p.from_kept;
    const uint32_t* const sel = from_kept ? p.kept : p.sigw;
    const unsigned sel_row = from_kept ? (unsigned)K / 16u : (unsigned)slabs;
    const int sel_bit = from_kept ? 1 : lane;
    // Offsets of the item being loaded (element offsets fit 32 bits: the entry points refuse layers of 2^32
    // elements and more).  Nothing guards the loads: rows past the item's last read that one again, lanes past
    // K the row's last columns (their importances are zero).
    unsigned nwo = 0u, ngo = 0u, nso = 0u;
    int nlast = 0;
    auto aim = [&](int slab, int rb) {
        const int row = min((rb * NW + warp) * rows, N - 1);
        const unsigned col = (unsigned)min(slab * 256 + lane * 8, K - 8);
        nwo = (unsigned)row * (unsigned)p.ldw + col;
        ngo = (unsigned)row * (unsigned)Gr + col / G;
        if (INNER) nso = (unsigned)row * sel_row + (from_kept ? col / 16u : (unsigned)slab);
        nlast = min(N - row, rows) - 1;
    };
    // (volatile: the compiler would move these loads down to where the row is worked on, to save registers)
    auto load_row = [&](int u) {
        const unsigned m = (unsigned)min(u, nlast);
        asm volatile("ld.global.cs.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[u].x), "=r"(v[u].y), "=r"(v[u].z), "=r"(v[u].w)
                     : "l"(p.W + (nwo + m * (unsigned)p.ldw)));
        if (MODE == AAAC_NVFP4) asm volatile("ld.global.u8 %0, [%1];" : "=r"(sc[u]) : "l"(p.scales + (ngo + m * (unsigned)Gr)));   // masked at use
        else asm volatile("ld.global.u32 %0, [%1];" : "=r"(sc[u]) : "l"(p.rinv + (ngo + m * (unsigned)Gr)));
        if (INNER) asm volatile("ld.global.u32 %0, [%1];" : "=r"(sgw[u]) : "l"(sel + (nso + m * sel_row)));
    };
    int cur_slab = -1;
    uint64_t II[4];           // importances of the lane's eight columns, in pairs
    float isum_raw = 0.f;     // sum of I over the lane's group (rounded up a little)
    bool col_ok = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) II[j] = 0ull;
    auto Ic = [&](int j) { return (j & 1) ? hi2(II[j >> 1]) : lo2(II[j >> 1]); };

    // (slab, row block) of the current item and of the one being loaded
    const int n_main = max(it1 - it0, 0), n_items = n_main + (has_tail ? 1 : 0);
    const int first = n_main > 0 ? it0 : tail_item;
    const int first_slab = first / p.nrb, first_rb = first - first_slab * p.nrb;
    int slab = first_slab, rb = first_rb;
    int nslab = slab, nrb = rb;
    if (n_items > 0) {
        aim(slab, rb);
#pragma unroll
        for (int u = 0; u < R; ++u) load_row(u);
    }

    if (MODE == AAAC_NVFP4 && tid >= 64 && tid < 192) {
        const int c = tid - 64;
        const float sv = __fmul_rn(e4m3_value((uint32_t)c), p.ctrl->s_t);
        S.rlut[c] = c ? __frcp_rn(sv) : 0.f;
    }

    // Fixed-point scale of the sums over the blocks.  The sums of a cell, and a sixteenth of the objective, are
    // below B = 16 N sum_k I_k (|w~ - c| < 16, or more with tables of the caller's outside (-8, 8): then B is larger
    // by that, squared), so with 2^e > B the value v 2^(93 - e) fits the limbs.  What is dropped lies 2^-93 below
    // B: also a cell whose only weight has 10^-20 of the importances' sum moves its entry.  Integer addition is
    // order-independent, so the totals do not depend on the order in which the blocks arrive.
    {
        float sum = 0.f;
        for (int k = tid; k < K; k += NT) sum = __fadd_ru(sum, fabsf(__ldg(p.I + k)));
#pragma unroll
        for (int o = 16; o; o >>= 1) sum = __fadd_ru(sum, __shfl_xor_sync(kAll, sum, o));
        if (p.reach) sum = __fmul_ru(sum, *p.reach);
        if (lane == 0) sh.wsum[warp][0] = (double)sum;
        __syncthreads();
        if (warp == 0) {
            double B = sh.wsum[lane & 15][0];
#pragma unroll
            for (int o = 8; o; o >>= 1) B += __shfl_xor_sync(kAll, B, o);
            B *= 257.0 / 16.0 * (double)N;
            if (lane == 0) {
                const int e = B > 0.0 && B < 1e300 ? ilogb(B) + 1 : 0;
                sh.fix_scale = scalbn(1.0, kSumBits - e);
                sh.fix_unscale = scalbn(1.0, e - kSumBits);
                sh.failed = 0;
            }
            derive_tables(S, lane, p.ctrl->T[lane]);
        }
    }
    for (int b = 0; b < kBinSlots; ++b) sts_bin(bins_lane + b * kSlotBytes, make_float2(0.f, 0.f));
    __syncthreads();
    write_tables<NT, true>(S, S.pq32, tid, kLut1At, lut2_addr);
    __syncthreads();

    // bin arithmetic: the masked mantissa of fl32(kBinsPerUnit x + kMagic) is bin * (REP * 8)
    constexpr float kBinsPerUnit = (float)(NB / 16);
    constexpr float kMagic = (float)(NB / 2) + 1.5f * (float)(1 << 23) / (float)(REP * 8);
    constexpr uint32_t kBinMask = (uint32_t)(NB - 1) * (REP * 8);

  for (int round = 0; round < n_rounds; ++round) {
    const unsigned pass_no = bar_base + (unsigned)round;
    // block 0 clears the buffer of the next pass: it was the buffer of two passes ago, and every block
    // finished reading it before it added to the previous pass's buffer, whose totals block 0 has seen
    static_assert(NT >= 256 + kCells * 4 + kLimbs, "threads 256.. of block 0 clear the next buffer");
    if (bid == 0 && tid >= 256 && tid < 256 + kCells * 4 + kLimbs) {
        const int w = tid - 256;
        p.acc[(size_t)((pass_no + 1u) % 3u) * kAccBuffer + (size_t)(w >> 2) * kAccStride + (w & 3)] = 0ull;
        __threadfence();
    }
    // near-tie bound: sqrt(a b) <= (kappa a + b / kappa) / 2, so the bound of the header comment is at
    // most g1 * (E0 + E1) + g2 * sum I, with kappa = 1/8 (about the usual |w~ - entry|)
    const float g1 = 0x1p-24f * __fmaf_ru(S.tmax283, 4.f, 16.f), g2 = 0x1p-24f * __fmul_ru(S.tmax283, 0.0625f);
    double Eacc = 0.0;

    CountedSums collected{};
    int counted = 0;          // items since the last collect_counts
    int ndefer = 0;           // groups on the warp's list (the same in every lane)
    float isum = __fmul_ru(isum_raw, g2);
    for (int i = 0; i < n_items; ++i) {
        slab = nslab;
        rb = nrb;
        if (i + 1 < n_main) {
            if (++nrb == p.nrb) { nrb = 0; ++nslab; }
        } else {                                           // the tail item comes next (if any)
            nslab = tail_item / p.nrb;
            nrb = tail_item - nslab * p.nrb;
        }
        // (the loads of the next item's rows stand in the row pipeline without a branch around them: with
        // one, the compiler kept them from moving, 835 -> 799 Gweights/s)
        if (i + 1 >= n_items) { nslab = first_slab; nrb = first_rb; }
        aim(nslab, nrb);
        const bool whole = i < n_main;                     // else: row tail_u of every warp only

        if (slab != cur_slab) {
            cur_slab = slab;
            const int col0 = slab * 256 + lane * 8;
            col_ok = col0 < K;
            isum_raw = 0.f;
            float Iv[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) Iv[j] = 0.f;
            if (col_ok) {
                const float4 a = __ldg(reinterpret_cast<const float4*>(p.I + col0));
                const float4 b = __ldg(reinterpret_cast<const float4*>(p.I + col0 + 4));
                Iv[0] = a.x; Iv[1] = a.y; Iv[2] = a.z; Iv[3] = a.w;
                Iv[4] = b.x; Iv[5] = b.y; Iv[6] = b.z; Iv[7] = b.w;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) isum_raw += Iv[j];
#pragma unroll
            for (int j = 0; j < 4; ++j) II[j] = pack2(Iv[2 * j], Iv[2 * j + 1]);
#pragma unroll
            for (int o = LPG / 2; o; o >>= 1) isum_raw += __shfl_xor_sync(0xFFFFFFFFu, isum_raw, o);
            isum_raw *= 1.0001f;
            isum = __fmul_ru(isum_raw, g2);
        }
        const int row0 = (rb * NW + warp) * rows;
        const int nrows = min(rows, N - row0);                // rows of this warp inside the layer (may be <= 0)

        // The rows of the item go through three stages, written out in the order in which the
        // shared-memory operations are to be issued, so that the read-modify-write chain on the
        // bins of one row runs while the table lookups of the next row are in flight:
        //   L1(u): w~ and the loads of {J_low, thr};   L2(u): slot and the loads of {P, Q};
        //   M(u):  errors, sigma, the centred terms and bin addresses;   B(u): bins += terms.
        float eitem = 0.f;                                 // objective of this item's groups led by this lane
        float x[8];                                        // w~ of the row in L1..M
        uint64_t pq[8];                                    // the bins' entries, then {P, Q}
        float mt[2][8];                                    // chosen centred term I (x - c) of the rows in B / M
        uint32_t ba[2][8];                                 // its bin address
        bool sg_row = false;                               // inner iteration: this lane's stored selection bit
        auto L1 = [&](int u) {
            if (INNER) sg_row = (sgw[u] >> sel_bit) & 1u;
            const float rinv = MODE == AAAC_NVFP4 ? S.rlut[sc[u] & 0x7Fu] : __uint_as_float(sc[u]);
            const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
            const uint64_t rr = pack2(rinv, rinv);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint64_t xx = mul2(pack2(bf16_lo(w[j]), bf16_hi(w[j])), rr);
                const uint64_t bb = fma2(xx, pack2(kBinsPerUnit, kBinsPerUnit), pack2(kMagic, kMagic));
                unpack2(xx, x[2 * j], x[2 * j + 1]);
                // (bin bits | lane's copy | table base) is one three-input logic instruction: no add per weight
                pq[2 * j] = lds_table_b64((__float_as_uint(lo2(bb)) & kBinMask) | lut1_or);
                pq[2 * j + 1] = lds_table_b64((__float_as_uint(hi2(bb)) & kBinMask) | lut1_or);
            }
        };
        // same, then refill the row's registers from the next item
        auto L1n = [&](int u) {
            L1(u);
            load_row(u);
        };
        auto L2 = [&]() {
#pragma unroll
            for (int j = 0; j < 8; ++j) second_lookup(pq[j], x[j]);
        };
        auto M = [&](int row, float (&mt_o)[8], uint32_t (&ba_o)[8]) {
            if constexpr (INNER) {
                // selection frozen: the centred term under the stored table only.  A poisoned
                // slot shows as NaN; those lanes search their intervals directly.
                const bool sg = sg_row;
                float c[8], chk = 0.f;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    c[j] = sg ? hi2(pq[j]) : lo2(pq[j]);
                    mt_o[j] = __fmul_rn(Ic(j), __fsub_rn(x[j], c[j]));
                    chk += mt_o[j];
                }
                const bool bad = !(chk == chk);
                if (__any_sync(0xFFFFFFFFu, bad)) {
                    Row8 r;
#pragma unroll
                    for (int j = 0; j < 8; ++j) { r.x[j] = x[j]; r.I[j] = Ic(j); r.hint[j] = kNoHint; }
                    const Exact8 ex = exact_groups<LPG>(&S, r, (int)bad);
                    if (bad) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float2 e = lds_table_f2(pq_entry_addr(lut2_addr, ex.J[j], lane));
                            c[j] = sg ? e.y : e.x;
                            mt_o[j] = __fmul_rn(Ic(j), __fsub_rn(x[j], c[j]));
                        }
                    }
                }
                const uint32_t base = bins_lane + (sg ? kM * kSlotBytes : 0);
#pragma unroll
                for (int j = 0; j < 8; ++j) ba_o[j] = base + (__float_as_uint(c[j]) & kIdxMask) * kSlotBytes;
                return;
            }
            // (pairs of columns rather than pairs of tables: eight registers of importances instead of sixteen)
            uint64_t m0[4], m1[4];                         // I (x - P), I (x - Q)
            uint64_t s0 = 0ull, s1 = 0ull;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint64_t u0 = pack2(__fsub_rn(x[2 * j], lo2(pq[2 * j])), __fsub_rn(x[2 * j + 1], lo2(pq[2 * j + 1])));
                const uint64_t u1 = pack2(__fsub_rn(x[2 * j], hi2(pq[2 * j])), __fsub_rn(x[2 * j + 1], hi2(pq[2 * j + 1])));
                m0[j] = mul2(II[j], u0);
                m1[j] = mul2(II[j], u1);
                s0 = fma2(m0[j], u0, s0);
                s1 = fma2(m1[j], u1, s1);
            }
            float e0 = lo2(s0) + hi2(s0), e1 = lo2(s1) + hi2(s1);
            group_sums<LPG>(e0, e1, lane);
            const float es = e0 + e1;
            const float tau = __fmaf_ru(es, g1, isum);
            // lanes past K carry I = 0 and the row's last weights; they need the exact path only if their slot is
            // poisoned (NaN), so that no NaN reaches a bin
            const bool near = !(fabsf(e1 - e0) > tau) && (col_ok || !(es == es));
            const bool sg = e1 < e0;
            float emin = sg ? e1 : e0;
            uint32_t base = bins_lane + (sg ? kM * kSlotBytes : 0), idx_mask = kIdxMask;
            if (__any_sync(0xFFFFFFFFu, near)) {
                // near-ties and poisoned slots (rare): the group goes on the warp's list, to be decided
                // in double by resolve_deferred; its lanes send this row's terms to the spare slot
                const bool lead = near && col_ok && (lane % LPG) == 0;
                const unsigned lm = __ballot_sync(0xFFFFFFFFu, lead);
                if (lead) sts_u2(list_addr + (uint32_t)(ndefer + __popc(lm & ((1u << lane) - 1u))) * 8u, (uint32_t)row,
                                 (uint32_t)(slab * 256 + lane * 8));
                ndefer += __popc(lm);
                if (near) { emin = 0.f; base = spare_lane; idx_mask = 0u; }
            }
            if (col_ok && (lane % LPG) == 0) eitem += emin;
            if (keep_sigma) {
                const unsigned bits = __ballot_sync(0xFFFFFFFFu, sg);        // (the bits of listed groups are set when they are decided)
                if (lane == 0) p.sigw[(size_t)row * (size_t)slabs + slab] = bits;
            }
            if (KIND == kKeep) {
                // (the two lanes of 16 columns write a half each; the selection stands in the lower one)
                uint32_t bits = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) bits = __funnelshift_r(bits, __float_as_uint(sg ? hi2(pq[j]) : lo2(pq[j])), 2);
                bits = ((bits >> 16) & 0x5555u) | (sg && !(lane & 1) ? 2u : 0u);
                if (col_ok) reinterpret_cast<uint16_t*>(p.kept)[(unsigned)row * (unsigned)(K / 8) + (unsigned)(slab * 32 + lane)] = (uint16_t)bits;
            }
            // cell = entry index (low bits of the centre constant) under the chosen table
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float a0 = (j & 1) ? hi2(m0[j >> 1]) : lo2(m0[j >> 1]), a1 = (j & 1) ? hi2(m1[j >> 1]) : lo2(m1[j >> 1]);
                mt_o[j] = sg ? a1 : a0;
                ba_o[j] = base + (__float_as_uint(sg ? hi2(pq[j]) : lo2(pq[j])) & idx_mask) * kSlotBytes;
            }
        };
        auto B = [&](const float (&mt_i)[8], const uint32_t (&ba_i)[8], int j0, int j1) {
#pragma unroll
            for (int j = j0; j < j1; ++j) {
                float2 a = lds_bin(ba_i[j]);
                a.x += mt_i[j];
                if (KIND == kKeep) a.y = __uint_as_float(__float_as_uint(a.y) + (1u << (4 * j)));
                else a.y += Ic(j);
                sts_bin(ba_i[j], a);
            }
        };

        if (nrows == R && whole) {
            // full item: L1(0) L2(0) M(0) | L1(1) B(0)[0..1] L2(1) B(0)[2..7] M(1) | ... | B(R-1)
            // (where the second lookups cut into the previous row's bin updates was chosen by measurement: 2 + 6)
            L1n(0);
            L2();
            M(row0, mt[0], ba[0]);
#pragma unroll
            for (int u = 1; u < R; ++u) {
                const int prev = (u - 1) & 1, cur = u & 1;
                L1n(u);
                B(mt[prev], ba[prev], 0, 2);
                L2();
                B(mt[prev], ba[prev], 2, 8);
                M(row0 + u, mt[cur], ba[cur]);
            }
            B(mt[(R - 1) & 1], ba[(R - 1) & 1], 0, 8);
        } else if (nrows == 2 && rows == 2) {
            L1n(0);
            L2();
            M(row0, mt[0], ba[0]);
            L1n(1);
            B(mt[0], ba[0], 0, 2);
            L2();
            B(mt[0], ba[0], 2, 8);
            M(row0 + 1, mt[1], ba[1]);
            B(mt[1], ba[1], 0, 8);
        } else {
            // ragged last row block of the layer, quarter items, items of one row: row by row, then refill all rows
            uint4 vr[R];
            uint32_t sr[R], gr[R];
#pragma unroll
            for (int t = 0; t < R; ++t) { vr[t] = v[t]; sr[t] = sc[t]; gr[t] = INNER ? sgw[t] : 0u; }
            const int ulo = whole ? 0 : tail_u, uhi = whole ? nrows : min(nrows, tail_u + 1);
            for (int u = ulo; u < uhi; ++u) {
                // (u is uniform over the warp; the stages read row 0 of v[] and sc[])
#pragma unroll
                for (int t = 0; t < R; ++t)
                    if (u == t) { v[0] = vr[t]; sc[0] = sr[t]; if (INNER) sgw[0] = gr[t]; }
                L1(0);
                L2();
                M(row0 + u, mt[0], ba[0]);
                B(mt[0], ba[0], 0, 8);
            }
#pragma unroll
            for (int t = 0; t < R; ++t) load_row(t);
        }
        Eacc += (double)eitem;
        const bool collect = KIND == kKeep && (++counted == kCountedItems || i + 1 == n_items || nslab != slab);
        if (!INNER && (ndefer > kDeferCap - R * (32 / LPG) || (collect && ndefer > 0))) {    // the next item could overflow the list, or the counts
            __syncwarp();
            Eacc += resolve_deferred<MODE, SEL, KIND>(&S, DeferArgs{p.W, p.K, p.ldw, p.scales, p.rinv, p.I, p.sigw, p.kept}, list_addr, ndefer, bins_lane, lane);
            ndefer = 0;
        }
        if (collect) {
            collect_counts(&collected, sm_base, hi_base, n_low, kBinBytes, make_float4(Ic(0), Ic(1), Ic(2), Ic(3)),
                           make_float4(Ic(4), Ic(5), Ic(6), Ic(7)), warp, lane);
            counted = 0;
        }
    }
    if (!INNER && ndefer > 0) {
        __syncwarp();
        Eacc += resolve_deferred<MODE, SEL, KIND>(&S, DeferArgs{p.W, p.K, p.ldw, p.scales, p.rinv, p.I, p.sigw, p.kept}, list_addr, ndefer, bins_lane, lane);
    }

    // ---- the warp's sums: lane c adds the 32 lane-private values of cell c (in an order of its own that
    //      avoids bank conflicts, and a fixed one).  In double, 32 FP32 values are added without rounding
    //      unless they are more than 2^24 apart ----
    const bool trace = KIND == kKeep || (!INNER && p.err_trace != nullptr);
    __syncwarp();
    if (KIND != kKeep) {
        const uint32_t cell_addr = bins_warp + lane * (kSlotBytes + 8);
        double dx[4] = {0.0, 0.0, 0.0, 0.0}, dy[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
        for (uint32_t i = 0; i < 256; i += 32) {
#pragma unroll
            for (uint32_t t = 0; t < 4; ++t) {
                const float2 a = lds_bin(cell_addr ^ (i + t * 8));
                dx[t] += scaled_double(a.x);
                dy[t] += scaled_double(a.y);
            }
        }
        sh.wsum[warp][lane] = ((dx[0] + dx[1]) + (dx[2] + dx[3])) * 0x1p896;
        sh.wsum[warp][kCells + lane] = ((dy[0] + dy[1]) + (dy[2] + dy[3])) * 0x1p896;
    } else {
        // the block's sums of two cells, which the others' rows add nothing to
        sh.wsum[warp][lane] = sh.wsum[warp][kCells + lane] = 0.0;
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            double x = collected.x[c], y = collected.y[c];
#pragma unroll
            for (int s = 16; s; s >>= 1) {
                x += __shfl_xor_sync(kAll, x, s);
                y += __shfl_xor_sync(kAll, y, s);
            }
            if (lane == 0) {
                sh.wsum[warp][2 * warp + c] = x * 0x1p896;
                sh.wsum[warp][kCells + 2 * warp + c] = y * 0x1p896;
            }
        }
    }
    if (trace) {
#pragma unroll
        for (int s = 16; s; s >>= 1) Eacc += __shfl_xor_sync(kAll, Eacc, s);
        if (lane == 0) sh.wsum[warp][2 * kCells] = Eacc;
    }
    __syncthreads();                                       // every warp is done with the lookup tables, its sums are there
    unsigned long long* const acc = p.acc + (size_t)(pass_no % 3u) * kAccBuffer;
    // ---- the block's sums: half-warp h of warp v adds cell 2 v + h, a lane per warp, pairwise ----
    static_assert(NW == 16 && 2 * NW == kCells, "a half-warp per cell, a lane per warp");
    {
        const int sum_warp = lane & 15, sum_cell = 2 * warp + (lane >> 4);
        double dxs = sh.wsum[sum_warp][sum_cell], dys = sh.wsum[sum_warp][kCells + sum_cell];
        double de = 0.0;
        const bool do_e = trace && warp == NW - 1;
        if (do_e) de = sh.wsum[sum_warp][2 * kCells];
#pragma unroll
        for (int s = 8; s; s >>= 1) {
            dxs += __shfl_xor_sync(kAll, dxs, s);
            dys += __shfl_xor_sync(kAll, dys, s);
            if (do_e) de += __shfl_xor_sync(kAll, de, s);
        }
        // The sums go into the pass's buffer as two 47-bit limbs, each with one arrival in the word's upper
        // bits: lanes 0-1 of the half-warp add the residual sum's limbs, 2-3 those of the weight sum, 4-5 of
        // the last warp's first half those of the objective.
        // A sum outside the limbs' range -- it cannot be right: an infinite or NaN weight or importance, reported by the
        // passes that read them -- counts as none, so that it does not spill into the arrivals.
        const int which = sum_warp >> 1;
        double sd = (which == 0 ? dxs : which == 1 ? dys : de * 0.0625) * sh.fix_scale;
        if (!(fabs(sd) < 0x1p93)) sd = 0.0;
        const double topm = __dadd_rd(sd * (1.0 / kLimb), kIntMagic);         // floor, as the low bits of a double near 1.5 2^52
        const long long top = __double_as_longlong(topm) - __double_as_longlong(kIntMagic);          // in [-2^46, 2^46)
        const double lowm = __dadd_rd(__fma_rn(-(topm - kIntMagic), kLimb, sd), kIntMagic);
        const long long low = __double_as_longlong(lowm) - __double_as_longlong(kIntMagic);          // in [0, 2^47]
        const unsigned long long add = (unsigned long long)((sum_warp & 1) ? top + kTopBias : low) + kOneArrival;
        if (which < 2) atomicAdd(acc + sum_cell * kAccStride + sum_warp, add);
        else if (do_e && lane < 6 && which == 2) atomicAdd(acc + kCells * kAccStride + (lane - 4), add);
    }
    // ---- meanwhile the bins start the next pass at zero: behind the sums, which the other blocks wait for
    //      (warp 1 clears those of warp 0, which waits) ----
    if (warp) {
#pragma unroll 8
        for (int b = 0; b < kCells; ++b) sts_bin(bins_lane + b * kSlotBytes, make_float2(0.f, 0.f));
        if (warp == 1) {
#pragma unroll 8
            for (int b = 0; b < kCells; ++b) sts_bin((n_low > 0 ? sm_base : hi_base) + lane * 8 + b * kSlotBytes, make_float2(0.f, 0.f));
        }
    }
    // ---- one warp waits until every block's sums are in and derives the new tables; lane c takes cell c ----
    if (warp == 0) {
        const unsigned long long want = (unsigned long long)p.arrivals;
        const bool my_e = trace && bid == 0 && lane == 0;
        bool ok = true;
        unsigned long long x[2], y[2], e[2] = {0, 0};
        for (unsigned spins = 0;; ++spins) {
            ld_relaxed_2xu64(acc + lane * kAccStride, x[0], x[1]);
            ld_relaxed_2xu64(acc + lane * kAccStride + 2, y[0], y[1]);
            if (my_e) ld_relaxed_2xu64(acc + kCells * kAccStride, e[0], e[1]);
            bool in = true;
#pragma unroll
            for (int l = 0; l < kLimbs; ++l)
                in = in && (x[l] >> kCountShift) >= want && (y[l] >> kCountShift) >= want && (!my_e || (e[l] >> kCountShift) >= want);
            if (__all_sync(kAll, in)) break;
            if (__any_sync(kAll, spins >= p.spin_limit || ((spins & 15u) == 15u && ld_relaxed_u32(&p.ctrl->abort)))) { ok = false; break; }
        }
        if (!ok) {
            if (lane == 0) sh.failed = 1;
        } else {
            auto total = [&](const unsigned long long (&w)[2]) {
                const unsigned long long sum = w[0] & kLimbMask;         // (its upper bits belong to the top limb)
                const long long low = (long long)(sum & ((1ull << kLimbBits) - 1ull));
                const long long top = (long long)(w[1] & kLimbMask) + (long long)(sum >> kLimbBits) - (long long)nblk * kTopBias;
                const double t = __longlong_as_double(top + __double_as_longlong(kIntMagic)) - kIntMagic;
                const double l = __longlong_as_double(low + __double_as_longlong(kIntMagic)) - kIntMagic;
                return __fma_rn(t, kLimb, l) * sh.fix_unscale;
            };
            // Eq. 11; cells of duplicate entries are empty: they keep their value
            const double sx = total(x), wt = total(y);
            double T = wt > 0.0 ? (double)S.centre[lane] + __ddiv_rn(sx, wt) : S.Td[lane];
            // the trace holds the Eq. 8 objective of each assignment step
            double err = 0.0, about = 0.0;
            if (KIND == kRest && trace) {
                // (the errors were formed about the constants, up to 8 units in the last place from the entries: sum I (x - T)^2 is
                // sum I (x - c)^2 less this.  Behind incremental rounds, whose objective has no such error: 1e-7 of it -> 1e-9)
                const double d = S.Td[lane] - (double)S.centre[lane];
                about = d * (2.0 * sx - d * wt);
#pragma unroll
                for (int s = 16; s; s >>= 1) about += __shfl_xor_sync(kAll, about, s);
            }
            if (my_e) {
                err = 16.0 * total(e);
                if (about < 0.5 * err) err -= about;
                if (KIND != kKeep || p.err_trace) p.err_trace[trace_base + round] = err;
            }
            const double Tp = __shfl_up_sync(kAll, T, 1);
            const double before = KIND == kKeep ? S.Td[lane] : 0.0;
            const bool unsorted = __any_sync(kAll, (lane & 15) != 0 && Tp > T);
            if (unsorted) {
                // ascending order within the table by rank (ties by index)
                int rank = 0;
#pragma unroll 1
                for (int i = 0; i < kM; ++i) {
                    const double o = __shfl_sync(kAll, T, (lane & 16) + i);
                    rank += (o < T) || (o == T && i < (lane & 15));
                }
                S.Td[(lane & 16) + rank] = T;
                __syncwarp();
                T = S.Td[lane];
                __syncwarp();
            }
            if (KIND == kKeep && bid == 0) {
                // what the incremental rounds start from
                Ctrl& c = *p.ctrl;
                c.keep_T[lane] = before;
                c.keep_c[lane] = S.centre[lane];
                c.keep_sx[lane] = sx;
                c.keep_sw[lane] = wt;
                if (lane == 0) {
                    c.keep_q = err;
                    c.keep_ok = !unsorted;
                    c.next_round = (uint32_t)(trace_base + round + 1);
                    c.passes = pass_no + 1u;
                }
            }
            derive_tables(S, lane, T);
        }
    }
    __syncthreads();
    if (sh.failed) {
        // a wait ran out (here or in another block): tell the others, report, leave
        if (tid == 0) {
            atomicExch(&p.ctrl->abort, 1u);
            if (p.dev_status) atomicOr(p.dev_status, AAAC_DEV_TIMEOUT);
        }
        return;
    }
    if (round + 1 < n_rounds) {
        write_tables<NT, true>(S, S.pq32, tid, kLut1At, lut2_addr);
        __syncthreads();
    }
  }
    if (bid == 0 && tid < 2 * kM) {
        p.ctrl->T[tid] = S.Td[tid];
        if (p.T01_out) p.T01_out[tid] = (float)S.Td[tid];
        if (REST && tid == 0) {
            p.ctrl->next_round = (uint32_t)(passed + n_rounds);
            p.ctrl->passes = bar_base + (unsigned)n_rounds;
        }
    }
}

// Several layers in one launch (the paper processes layers independently, Sec. 3.3): the grid is
// cut into consecutive ranges of blocks, one per layer, and every range runs that layer's rounds
// by itself -- its blocks wait only for each other, on the layer's own accumulators -- so the
// per-round fixed cost (sums across blocks, new tables, table building) is paid once for the
// whole batch instead of once per layer, and small layers no longer leave most of the GPU idle.
constexpr int kMaxBatch = 8;
struct FitBatch {
    FitParams L[kMaxBatch];
    unsigned first[kMaxBatch + 1];    // first block of every layer; first[n..] = grid size
};

#include "fit_delta.cuh"

template <int MODE, int SEL, int KIND>
__global__ void __launch_bounds__(kFitWarps * 32, 1) fit_kernel(const __grid_constant__ FitBatch b) {
    // a single layer: its parameters at fixed places (1-3 % faster than picked by index, which for several
    // layers is as fast as a copy of the body per layer)
    if (b.first[1] == gridDim.x) { fit_rounds_body<MODE, SEL, KIND>(b.L[0], blockIdx.x, gridDim.x); return; }
    int l = 0;
    while (l + 1 < kMaxBatch && blockIdx.x >= b.first[l + 1]) ++l;
    fit_rounds_body<MODE, SEL, KIND>(b.L[l], blockIdx.x - b.first[l], b.first[l + 1] - b.first[l]);
}

__global__ void export_tables_kernel(const Ctrl* ctrl, float* T01) {
    if (threadIdx.x < 2 * kM) T01[threadIdx.x] = (float)ctrl->T[threadIdx.x];
}

// The fit kernels place their tables at fixed shared addresses and take all the shared memory a block
// may have beyond their static part (one block per SM either way); the kernel checks that its layout fits.
template <void (*kern)(FitBatch)>
cudaError_t launch_variant(FitBatch& b, unsigned grid, cudaStream_t st) {
    static std::atomic<size_t> ready[kMaxDevices];          // dynamic shared memory, once it is set up on a device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    size_t smem = ready[dev].load(std::memory_order_relaxed);
    if (smem == 0) {
        cudaFuncAttributes a;
        int optin = 0;
        if ((e = cudaFuncGetAttributes(&a, reinterpret_cast<const void*>(kern))) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
        if ((size_t)optin <= a.sharedSizeBytes) return cudaErrorInvalidValue;
        smem = (size_t)optin - a.sharedSizeBytes;
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
        ready[dev].store(smem, std::memory_order_relaxed);
    }
    void* args[] = {&b};
    note_launch();
    // cooperative: the blocks of a layer wait for each other, so all of them must be resident
    return cudaLaunchCooperativeKernel(reinterpret_cast<void*>(kern), dim3(grid), dim3(kFitWarps * 32), args, smem, st);
}

template <int KIND>
cudaError_t launch_kind(FitBatch& b, unsigned grid, int mode, int sel_group, cudaStream_t st) {
    if (mode == AAAC_INT4 && sel_group == 16) return launch_variant<fit_kernel<AAAC_INT4, 16, KIND>>(b, grid, st);
    if (mode == AAAC_INT4) return launch_variant<fit_kernel<AAAC_INT4, 128, KIND>>(b, grid, st);
    return launch_variant<fit_kernel<AAAC_NVFP4, 16, KIND>>(b, grid, st);
}


// n_inner > 1: per round an assignment pass and the further inner iterations
template <typename Assign, typename Inner>
cudaError_t launch_inner(FitBatch& b, int m, int first, int n_outer, int n_inner, Assign assign, Inner inner) {
    cudaError_t e = cudaSuccess;
    for (int outer = first; outer < n_outer && e == cudaSuccess; ++outer) {
        for (int l = 0; l < m; ++l) { b.L[l].n_rounds = 1; b.L[l].trace_base = outer; }
        e = assign();
        for (int l = 0; l < m; ++l) { b.L[l].bar_base += 1u; b.L[l].n_rounds = n_inner - 1; }
        if (e == cudaSuccess) e = inner();
        for (int l = 0; l < m; ++l) b.L[l].bar_base += (unsigned)(n_inner - 1);
    }
    return e;
}

}  // namespace

// Deals a layer's items to `blocks` blocks: whole items in contiguous ranges plus, where that is
// shorter for the busiest block, a tail dealt out one row per warp (a quarter item) per block.
// Returns the number of blocks actually used.
static int64_t plan_layer(FitParams& p, int64_t N, int64_t K, int64_t blocks) {
    const int64_t slabs = (K + 255) / 256, g = blocks < kMaxFitBlocks ? blocks : kMaxFitBlocks;
    p.rows = kRowsPerWarp;
    p.nrb = (int)((N + kRowsPerWarp * kFitWarps - 1) / (kRowsPerWarp * kFitWarps));
    const int64_t items = slabs * p.nrb;
    p.per_block = (int)((items + g - 1) / g);
    p.tail_item0 = (int)items;
    p.tail_quarters = 0;
    int64_t grid = 0, cost = 10 * kRowsPerWarp * (int64_t)p.per_block;
    {
        // an even number of whole items per block plus a quarter-item tail, where that is shorter for
        // the busiest block (a tail row costs more than a quarter of a pipelined item: count it double)
        const int64_t whole = items / g, rest = items - whole * g;
        if (whole >= 4 && rest > 0 && 4 * rest <= g && 2 * whole + 1 < 2 * p.per_block) {
            p.per_block = (int)whole;
            p.tail_item0 = (int)(whole * g);
            p.tail_quarters = (int)(4 * rest);
            grid = g;
        }
    }
    // Layers with few items per block: items of two rows or one row per warp, where that is shorter for the
    // busiest block (a row of such an item counts for 1.2 and 1.6 rows of the four-row pipeline).  512 x 512:
    // 16 blocks of one item, 8.5 us a pass -> 64 blocks of one row per warp, 6.9; 1531 x 2064: two items of
    // four rows -> three of two, 11.4 -> 10.6 us.
    for (int rows = 2; rows >= 1; --rows) {
        const int64_t nrb = (N + rows * kFitWarps - 1) / (rows * kFitWarps), it = slabs * nrb, per = (it + g - 1) / g;
        const int64_t c = per * (rows == 2 ? 24 : 16);
        if (c < cost && p.tail_quarters == 0) {
            cost = c;
            p.rows = rows;
            p.nrb = (int)nrb;
            p.per_block = (int)per;
            p.tail_item0 = (int)it;
        }
    }
    p.items = (int)(slabs * p.nrb);
    if (p.tail_quarters == 0) grid = (p.items + p.per_block - 1) / p.per_block;
    p.arrivals = (unsigned)grid + (unsigned)g_extra_arrivals;
    return grid;
}

static bool fill_params(FitParams& p, const FitLayerArgs& a, int n_outer, uint32_t* dev_status) {
    p = FitParams{};
    p.W = a.W; p.N = a.N; p.K = a.K; p.ldw = a.ldw;
    p.scales = static_cast<const uint8_t*>(a.scales); p.rinv = a.ws.rinv; p.I = a.I; p.reach = a.reach;
    p.ctrl = a.ws.ctrl; p.acc = a.ws.acc; p.err_trace = a.err_trace; p.T01_out = a.T01_out; p.dev_status = dev_status;
    p.n_rounds = n_outer; p.trace_base = 0; p.bar_base = 0u;
    p.spin_limit = g_spin_limit;
    p.kept = a.ws.qlist;
    p.sigw = a.ws.qlist;            // the quantile selection's list is free once the start tables exist
    const int64_t slabs = (a.K + 255) / 256;
    const int64_t nrb = (a.N + kFitWarps - 1) / kFitWarps;
    return !(a.N > 0x7FFFFFFF || a.K > 0x7FFFFFFF || slabs * nrb > 0x7FFFFFFF);
}

// Incremental rounds (fit_delta.cuh) pay where few weights move and the passes are long.  4096 x 14336, us a pass, all
// weights added against those that move: NVFP4 70 against 93 in the second round, 70 in the third to sixth, 56 from the
// tenth on; INT4, whose tables move more, 74 against 112 and 95.  Three launches, the counts of the keeping pass and what
// is left on the warps' lists cost 60 to 100 us, and the early rounds gain nothing.  How many weights move is not known here: the
// more even the importances, the more (and with heavier tails more from quantiles, fewer from the grid).  Time of all full rounds /
// time so, the lowest and highest of normal and Student-t weights from the quantile and the grid start (units are 16 x 512 weights a block):
//   units x rounds             12 x 30    20 x 21    20 x 30    28 x 19    48 x 16    48 x 20    48 x 30    98 x 10    98 x 14    98 x 20    98 x 30
//   massive channels          .96- .98   .97-1.03  1.00-1.08  1.00-1.04   .99-1.02  1.01-1.04  1.05-1.09   .95- .98   .99-1.03  1.02-1.07  1.07-1.12
//   log-normal, deviation 1.2 .91- .95   .91- .95   .95-1.00   .93- .97   .92- .96   .93- .98   .98-1.03   .91- .95   .93- .98   .95-1.01   .99-1.06
//   equal                     .90- .94   .86- .94   .94- .98   .92- .96   .90- .95   .91- .97   .96-1.02   .87- .93   .92- .96   .94- .99   .98-1.04
// Activations have massive channels, so the first row counts double against the second: the line is about 20 x 26, 28 x 23, 48 x 19, 98 x 16.
// Further inner iterations have no flips and gain from the first pass on, the assignments between them lose.  Mean of normal and Student-t
// weights from the quantile start, massive channels / log-normal:
//   3 x 10   6 units 1.08 / 1.03, 9 1.08 / 1.02        2 x 10   7 units 1.03 / .99, 16 1.09 / 1.04        1 x 10   13 units .99 / .98, 16 1.01 / .99, 20 1.03 / 1.02
//   3 x 7    9 units 1.04 / .98                        2 x 7   13 units 1.01 / .97                        1 x 8   48 units 1.01 / 1.01, 98 1.02 / 1.01
//   3 x 6   13 units 1.05 / 1.00, 28 1.12 / 1.05       2 x 6   16 units 1.00 / .97, 20 1.02 / .99, 48 1.04 / .99
//   3 x 5   16 units 1.04 / .98, 20 1.05 / 1.00        2 x 5   20 units  .99 / .96                        2 x 4   12 to 98 units .92-.96 / .91-.94
// Roughly the units times these iterations tell.
// They start from the first pass's tables, though, and do not begin where these hold one value twice, as the NVFP4 grid
// does (tried and made again, 4096 x 4096 took 778 us for 743, and 312 for 274 in one round of 10).
// A piece is read with one 32-byte load; its number must be divisible by more than one piece per row (row_of).
constexpr int kFullRounds = 3;                        // the last of them the keeping one
static bool can_increment(const FitLayerArgs& a, int64_t blocks, int n_outer, int n_inner) {
    const int64_t slabs = (a.K + kDeltaCols - 1) / kDeltaCols, units = slabs * ((a.N + kFitWarps - 1) / kFitWarps);
    const int64_t frozen = (int64_t)n_outer * (n_inner - 1);      // further inner iterations
    const bool pays = n_inner == 1 ? units >= 20 * blocks && (n_outer - 13) * units >= 260 * blocks
                                   : n_inner >= 5 && frozen >= 9 && frozen * units >= 165 * blocks;
    return pays && !(n_inner > 1 && a.twin_entries) && a.ws.qcap >= (size_t)a.N * (size_t)a.K / 16 && a.K >= 64 && reinterpret_cast<uintptr_t>(a.W) % 32 == 0 &&
           a.ldw % 16 == 0 && 8 * a.K >= 7 * kDeltaCols * slabs;
}

cudaError_t launch_fit_rounds_batch(const FitLayerArgs* layers, int n, int mode, int sel_group, int n_outer, int n_inner,
                                    uint32_t* dev_status, cudaStream_t st) {
    if (n_outer <= 0 || n <= 0) return cudaSuccess;
    if (n_inner < 1 || (int64_t)n_outer * n_inner > 0x7FFFFFFF) return cudaErrorInvalidValue;
    static_assert(kFitAccWords == 3 * kAccBuffer, "the workspace holds three sum buffers");
    const int sms = sm_count();
    for (int at = 0; at < n;) {
        const int m = std::min({n - at, kMaxBatch, sms});
        FitBatch b{};
        int64_t items[kMaxBatch], share[kMaxBatch];
        constexpr int kRowsPerItem = kRowsPerWarp * kFitWarps;
        for (int l = 0; l < m; ++l) {
            const FitLayerArgs& a = layers[at + l];
            if (!fill_params(b.L[l], a, n_outer, dev_status)) return cudaErrorInvalidValue;
            items[l] = ((a.K + 255) / 256) * ((a.N + kRowsPerItem - 1) / kRowsPerItem);
            share[l] = 1;
        }
        // one block per layer, then every further block to the layer whose busiest block has the most items
        for (int left = sms - m; left > 0; --left) {
            int best = -1;
            int64_t load = 0;
            for (int l = 0; l < m; ++l) {
                const int64_t per = (items[l] + share[l] - 1) / share[l];
                if (share[l] < kRowsPerWarp * items[l] && share[l] < kMaxFitBlocks && per > load) { load = per; best = l; }
            }
            if (best < 0) break;
            ++share[best];
        }
        unsigned grid = 0;
        for (int l = 0; l < m; ++l) {
            const FitLayerArgs& a = layers[at + l];
            b.first[l] = grid;
            grid += (unsigned)plan_layer(b.L[l], a.N, a.K, share[l]);
        }
        for (int l = m; l <= kMaxBatch; ++l) b.first[l] = grid;
        const int full = n_inner == 1 ? kFullRounds : 1;
        bool incremental = mode == AAAC_NVFP4 && n_outer * n_inner > full + 1;
        for (int l = 0; l < m; ++l) incremental = incremental && can_increment(layers[at + l], b.first[l + 1] - b.first[l], n_outer, n_inner);
        cudaError_t e = cudaSuccess;
        if (incremental) {
            // the first rounds (the first pass), the last of which stores what the incremental ones need; these; and the
            // last pass, or whatever they leave undone.  (16432 x 8192: the keeping pass takes 41 us more than a full one, 18 of them
            // the counts, the rest its launch; 4096 x 14336: 33 and 19.)
            if (n_inner == 1) {
                for (int l = 0; l < m; ++l) b.L[l].n_rounds = full - 1;
                e = launch_kind<kRounds>(b, grid, mode, sel_group, st);
            }
            for (int l = 0; l < m; ++l) { b.L[l].n_rounds = 1; b.L[l].trace_base = full - 1; b.L[l].bar_base = (unsigned)(full - 1); }
            if (e == cudaSuccess) e = launch_variant<fit_kernel<AAAC_NVFP4, 16, kKeep>>(b, grid, st);
            for (int l = 0; l < m; ++l) b.L[l].trace_base = 0;
            for (int l = 0; l < m; ++l) { b.L[l].n_rounds = n_outer * n_inner - 1; b.L[l].n_inner = n_inner; }
            if (e == cudaSuccess) e = launch_variant<delta_kernel>(b, grid, st);
            for (int l = 0; l < m; ++l) b.L[l].n_rounds = n_outer * n_inner;
            if (e == cudaSuccess && n_inner == 1) e = launch_variant<fit_kernel<AAAC_NVFP4, 16, kRest>>(b, grid, st);
            if (e == cudaSuccess && n_inner > 1) {
                auto inner_rest = [&] { return launch_variant<fit_kernel<AAAC_NVFP4, 16, kInnerRest>>(b, grid, st); };
                for (int l = 0; l < m; ++l) { b.L[l].n_total = n_outer * n_inner; b.L[l].from_kept = true; }
                e = inner_rest();
                for (int l = 0; l < m; ++l) b.L[l].from_kept = false;
                if (e == cudaSuccess)
                    e = launch_inner(b, m, 1, n_outer, n_inner, [&] { return launch_variant<fit_kernel<AAAC_NVFP4, 16, kAssignRest>>(b, grid, st); },
                                     inner_rest);
            }
        } else if (n_inner == 1) {
            e = launch_kind<kRounds>(b, grid, mode, sel_group, st);
        } else {
            e = launch_inner(b, m, 0, n_outer, n_inner, [&] { return launch_kind<kAssignKeep>(b, grid, mode, sel_group, st); },
                             [&] { return launch_kind<kInner>(b, grid, mode, sel_group, st); });
        }
        if (e != cudaSuccess) return e;
        at += m;
    }
    return cudaSuccess;
}

void set_fit_wait(int extra_arrivals, unsigned spin_limit) {
    g_extra_arrivals = extra_arrivals > 0 ? extra_arrivals : 0;
    g_spin_limit = spin_limit ? spin_limit : kDefaultSpinLimit;
}

cudaError_t launch_export_tables(float* T01, const Workspace& ws, cudaStream_t st) {
    export_tables_kernel<<<1, 32, 0, st>>>(ws.ctrl, T01);
    note_launch();
    return cudaGetLastError();
}

}  // namespace aaac
