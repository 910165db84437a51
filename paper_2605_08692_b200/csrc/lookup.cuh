// Lookup machinery shared by the fit rounds (fit.cu) and the pack pass (pack.cu): the tables that
// turn a normalised weight into its interval of the merged breakpoint list and into the nearest
// entries of T0 and T1, their construction, and the double-precision fallback.  See the header
// comment of fit.cu for the method.
#pragma once
#include "internal.cuh"

namespace aaac {

constexpr int kRowsPerWarp = 4;
constexpr int kNBins = 512;                        // uniform bins of the per-bin table on (-8, 8): width 1/32
constexpr int kRep = 16;                           // copies of the per-bin table: one per lane of a half-warp, so an 8-byte lookup has no bank conflicts
constexpr int kJSlots = 32;                        // 31 intervals + the poisoned slot
constexpr int kSlotBytes = 32 * 8;                 // bytes of a lane-private bin slot (one 8-byte entry per lane)
// The {P, Q} table: one row per interval J, 16 columns of 8 bytes, so that a bin's table entry can
// name the row of its lower interval and a weight above the bin's breakpoint takes the next row.  Lane l
// uses column l mod 16: an 8-byte load is served a half-warp at a time, so lanes l and l + 16 never meet.
constexpr int kPqRow = 128;
constexpr int kPqCols = 16;
constexpr int kPoison = kNJ * kPqRow;              // byte offset of the poisoned row (NaN)
constexpr int kLut1Bytes = kNBins * kRep * 8;
constexpr int kLut2Bytes = kJSlots * kPqRow;
constexpr int kCells = 2 * kM;                     // bins per lane: [sigma][entry]
constexpr uint32_t kNoHint = 0xFFu;                // in the place of an interval: search for it
constexpr uint32_t kIdxMask = 15u;                 // low mantissa bits of a centre constant = entry index

// Shared-memory accesses of the hot loop with explicit 32-bit addresses.  All are volatile asm,
// which keeps them in the order in which the loop writes them (table lookups of one row issued
// ahead of the read-modify-write chain of the previous one).
__device__ __forceinline__ float2 lds_table_f2(uint32_t addr) {
    float2 r;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "r"(addr));
    return r;
}
// Two forms of a bin's entry.  The pack pass, which is bound by its instructions: {address of the lower
// interval's {P, Q}, breakpoint}, and every weight looks {P, Q} up, a row further if it lies above the
// breakpoint (one compare, one predicated add).
__device__ __forceinline__ uint32_t above_addr(uint32_t a, float x, uint32_t thr_bits) {
    asm("{\n\t.reg .pred p;\n\tsetp.gt.f32 p, %1, %2;\n\t@p add.u32 %0, %0, 128;\n\t}"
        : "+r"(a) : "f"(x), "f"(__uint_as_float(thr_bits)));
    return a;
}
__device__ __forceinline__ uint2 lds_table_u2(uint32_t addr) {
    uint2 r;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "r"(addr));
    return r;
}

// The fit rounds, bound by shared memory: {P, Q} itself where no breakpoint lies in the bin (four fifths of the weights), else
// {breakpoint, address of the lower interval's {P, Q}}: an address is below kAddrLimit, which no centre
// constant is as an integer.  Such a weight looks {P, Q} up, in the next row if it lies above the
// breakpoint; the other lanes take no part, and a load of a few lanes costs half of a full one.
__device__ __forceinline__ void second_lookup(uint64_t& pq, float x) {
    asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b32 a;\n\t.reg .f32 b;\n\t"
                 "mov.b64 {b, a}, %0;\n\t"
                 "setp.lt.u32 p, a, 262144;\n\t"
                 "setp.gt.and.f32 q, %1, b, p;\n\t"
                 "@q add.u32 a, a, 128;\n\t"
                 "mov.b64 %0, {b, a};\n\t"
                 "@p ld.shared.b64 %0, [a];\n\t}"
                 : "+l"(pq) : "f"(x));
}
__device__ __forceinline__ uint64_t lds_table_b64(uint32_t addr) {
    uint64_t r;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(r) : "r"(addr));
    return r;
}

__device__ __forceinline__ float2 lds_bin(uint32_t addr) {
    float2 r;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "r"(addr) : "memory");
    return r;
}
__device__ __forceinline__ void sts_bin(uint32_t addr, float2 v) {
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" :: "r"(addr), "f"(v.x), "f"(v.y) : "memory");
}

struct FitTables {
    double Td[2 * kM];            // the tables
    double2 PQ[kJSlots];          // nearest entries of T0 / T1 on interval J, as double
    float bp[32];                 // sorted breakpoints, bp[30] = bp[31] = +inf
    float2 pq32[kJSlots];         // {P, Q} of every interval
    float tmp_b[32];              // breakpoints by table
    float centre[2 * kM];         // centre constant of every entry (index in the low 4 mantissa bits)
    float rlut[128];              // NVFP4: fl32(1 / s_eff) per E4M3 code
    uint8_t src[32];              // table a breakpoint comes from
    uint8_t exact[32];            // the breakpoint is the exact midpoint of two different entries
    float tmax283;                // 2.83 * 17 * max |entry|, rounded up
    int no_dup;                   // no table holds two equal entries: the interval of a weight is then the sum of its two entry indices
};

// number of breakpoints below x (sorted list): the interval of x
__device__ __forceinline__ int find_interval(const float* bp, float x) {
    int J = 0;
#pragma unroll
    for (int step = 16; step; step >>= 1)
        if (J + step <= kNBP && bp[J + step - 1] < x) J += step;
    return J;
}

// Everything that follows from the tables and is small: the merged breakpoints, the nearest entries of
// every interval, the centre constants, the near-tie bound.  One warp, lane t with entry t in T, and no
// block barrier: there are only 32 values of each, and what it costs is latency (0.4 us; the version that
// used the block's threads and four barriers took 1.8 us of every round).
__device__ __forceinline__ void derive_tables(FitTables& S, const int lane, const double T) {
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int r = lane >> 4, i = lane & 15;
    S.Td[lane] = T;
    const double Tn = __shfl_down_sync(kAll, T, 1), Tp = __shfl_up_sync(kAll, T, 1);
    const unsigned dup = __ballot_sync(kAll, i > 0 && Tp == T);          // equal to its predecessor
    const bool sorted = !__any_sync(kAll, i > 0 && !(Tp <= T));
    const double mid = (T + Tn) * 0.5;
    const float b = i < 15 ? f32_round_down(mid) : __int_as_float(0x7F800000);
    // place in the merged list (equal breakpoints: table 0 first, then by index), found by binary search in
    // the other table's list; tables given by the caller may be out of order: count
    S.tmp_b[lane] = b;
    __syncwarp();
    const float* other = S.tmp_b + (r ? 0 : 16);
    int rank = 0;
    if (sorted) {
#pragma unroll
        for (int step = 8; step; step >>= 1) {
            const float ob = other[rank + step - 1];
            if (r ? ob <= b : ob < b) rank += step;                      // (15 entries: index 14 at most)
        }
        rank += i;
    } else {
#pragma unroll 1
        for (int j = 0; j < 15; ++j) {
            const float ob = other[j], own = S.tmp_b[(lane & 16) + j];
            rank += (r ? ob <= b : ob < b) + ((own < b) || (own == b && j < i));
        }
    }
    if (i == 15) rank = 30 + r;
    S.bp[rank] = b;
    S.src[rank] = (uint8_t)(i == 15 ? 0 : r);
    S.exact[rank] = (uint8_t)(i < 15 && (double)b == mid && T != Tn);
    // lowest index of the entries equal to entry k of table t
    auto canonical = [&](int t, int k) { return 31 - __clz(~(t ? dup >> 16 : dup & 0xFFFFu) & ((2u << k) - 1u)); };
    // centre constant: the float nearest to the FP32 rounding of the entry whose low 4 mantissa bits are
    // the entry's canonical index (at most 8 units in the last place away)
    // (and is never below 2^-100 in magnitude, so that as an integer it cannot be taken for an address)
    const uint32_t bits = __float_as_uint((float)T);
    const int ci = canonical(r, i), tt = max((int)(bits & 0x7FFFFFFFu), 0x0D800010) + 8 - ci;
    S.centre[lane] = __uint_as_float((bits & 0x80000000u) | (uint32_t)((tt & ~15) + ci));
    __syncwarp();
    // entries of T0 / T1 whose upper midpoint lies below interval `lane`
    const unsigned from1 = __ballot_sync(kAll, S.src[lane] == 1);
    int i1 = min(__popc(from1 & ((1u << lane) - 1u)), 15), i0 = max(0, min(lane - i1, 15));
    i0 = canonical(0, i0);
    i1 = canonical(1, i1);
    const float nan = __int_as_float(0x7FC00000);
    S.PQ[lane] = lane < kNJ ? make_double2(S.Td[i0], S.Td[kM + i1]) : make_double2(0.0, 0.0);
    S.pq32[lane] = lane < kNJ ? make_float2(S.centre[i0], S.centre[kM + i1]) : make_float2(nan, nan);
    const uint32_t tm = __reduce_max_sync(kAll, __float_as_uint(fmaxf(__double2float_ru(fabs(T)), 0x1p-70f)));
    if (lane == 0) {
        S.tmax283 = __fmul_ru(__uint_as_float(tm), 2.83f * 17.f);
        S.no_dup = dup == 0u;
    }
}

// The two lookup tables, written by the whole block (no barrier inside).  Bin b of width 1/32 holds the x
// with 32 x + 256 in [b - h, b + 1 - h], h = half of the rounding step 1 / 128 of the bin arithmetic.  The
// breakpoints are sorted, so those inside a bin are the first ones not below its lower edge.  A thread
// writes the 16 copies of its bin, two per store, in an order rotated by its lane, so that the eight
// lanes that a 16-byte store is served for meet in no bank.
// rows: the constants of every interval; low, where given: the interval of every bin's lower edge (kNoHint if poisoned).  DIRECT: the fit rounds' form of the bins' entries.
template <int NT, bool DIRECT>
__device__ __forceinline__ void write_tables(const FitTables& S, const float2* rows, const int tid, const uint32_t lut1_addr, const uint32_t lut2_addr,
                                             uint8_t* low = nullptr) {
    static_assert(kNBins % NT == 0, "whole bins per thread");
    constexpr float h = 0.5f / (float)(kRep * 8);
    constexpr float kHalf = (float)(kNBins / 2), kWidth = 16.f / (float)kNBins;
#pragma unroll
    for (int b = tid; b < kNBins; b += NT) {
        const float lo = ((float)b - kHalf - h) * kWidth, hi = ((float)b - (kHalf - 1.f) - h) * kWidth;
        const int below = find_interval(S.bp, lo);
        const float v0 = S.bp[below], v1 = S.bp[below + 1];     // bp[30], bp[31] = +inf
        const bool poison = v1 <= hi;                            // two breakpoints or more
        if (low) low[b] = (uint8_t)(poison ? kNoHint : (uint32_t)below);
        uint32_t e0, e1, c1 = 0;                                // c1: what an address grows by from copy to copy
        if (!DIRECT) {
            e0 = lut2_addr + (poison ? (uint32_t)kPoison : (uint32_t)(below * kPqRow));
            e1 = !poison && v0 <= hi ? __float_as_uint(v0) : 0x7F800000u;
        } else if (!poison && !(v0 <= hi)) {
            const float2 v = rows[below];
            e0 = __float_as_uint(v.x);
            e1 = __float_as_uint(v.y);
        } else {
            e0 = poison ? 0x7F800000u : __float_as_uint(v0);
            e1 = lut2_addr + (poison ? (uint32_t)kPoison : (uint32_t)(below * kPqRow));
            c1 = 8u;
        }
        const uint32_t at = lut1_addr + (uint32_t)b * (kRep * 8);
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const uint32_t c = (uint32_t)((s + tid) & 7) * 16u;
            if (DIRECT) {
                const uint32_t f = e1 + (c1 ? c : 0u);
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %1, %3};" :: "r"(at + c), "r"(e0), "r"(f), "r"(f + c1) : "memory");
            } else {
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %2};" :: "r"(at + c), "r"(e0 + c), "r"(e1), "r"(e0 + c + 8u) : "memory");
            }
        }
    }
    static_assert(kLut2Bytes / 16 <= NT, "one store per thread");
    if (tid < kLut2Bytes / 16) {
        const float2 v = rows[tid >> 3];
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %1, %2};" :: "r"(lut2_addr + (uint32_t)tid * 16u), "f"(v.x), "f"(v.y) : "memory");
    }
}

// address of column (lane mod 16) of interval J's entry in the {P, Q} table that starts at lut2_addr
__device__ __forceinline__ uint32_t pq_entry_addr(uint32_t lut2_addr, int J, int lane) {
    return lut2_addr + (uint32_t)(J * kPqRow) + (uint32_t)(lane & (kPqCols - 1)) * 8u;
}

// hint[j] < kNJ names the interval of weight j where the caller knows it, else the interval is searched
struct Row8 { float x[8]; float I[8]; uint32_t hint[8]; };

// The interval of a weight from the constants {P, Q} the fast path has looked up: with no equal
// entries inside a table, entry index = number of that table's breakpoints below the weight, and
// the interval of the merged list is the sum of the two.  (A poisoned slot reads as NaN: no hint.)
__device__ __forceinline__ uint32_t interval_hint(const FitTables& S, float P, float Q) {
    return (S.no_dup && P == P) ? (__float_as_uint(P) & kIdxMask) + (__float_as_uint(Q) & kIdxMask) : kNoHint;
}
struct Exact8 { int J[8]; double emin; int sigma; int tie; };

// Double-precision decision (Eq. 8 as a plain double-precision loop states it, lanes of a group
// combined by a shuffle tree) for the groups whose lanes pass need != 0; every lane of the warp
// calls.  The interval of every weight is found by binary search of the breakpoint list.
template <int LPG>
__device__ __noinline__ Exact8 exact_groups(const FitTables* S, Row8 r, int need) {
    Exact8 out;
    double e0 = 0.0, e1 = 0.0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        int J = 0;
        if (need) {
            if (r.hint[j] < (uint32_t)kNJ) {
                J = (int)r.hint[j];
            } else {
#pragma unroll
                for (int step = 16; step; step >>= 1)      // number of breakpoints below x (sorted list)
                    if (J + step <= kNBP && S->bp[J + step - 1] < r.x[j]) J += step;
            }
            const double2 pq = S->PQ[J];
            const double xd = (double)r.x[j], id = (double)r.I[j];
            const double d0 = __dsub_rn(xd, pq.x), d1 = __dsub_rn(xd, pq.y);
            e0 = __dadd_rn(e0, __dmul_rn(id, __dmul_rn(d0, d0)));
            e1 = __dadd_rn(e1, __dmul_rn(id, __dmul_rn(d1, d1)));
        }
        out.J[j] = J;
    }
#pragma unroll
    for (int s = LPG / 2; s; s >>= 1) {
        e0 = __dadd_rn(e0, __shfl_xor_sync(0xFFFFFFFFu, e0, s));
        e1 = __dadd_rn(e1, __shfl_xor_sync(0xFFFFFFFFu, e1, s));
    }
    out.sigma = e1 < e0;
    out.tie = e0 == e1;
    out.emin = out.sigma ? e1 : e0;
    return out;
}

}  // namespace aaac
