// The incremental rounds (included by fit.cu, inside its namespaces).
//
// From one round to the next most weights stay in their cell (NVFP4, quantile start: 4-10 % of the weights move in the
// second round, 1-3 % from the tenth on; INT4: 8-11 %, then 5 %).  A pass of fit_rounds_body nevertheless adds every
// weight to its cell, and that read-modify-write is half of its shared-memory traffic and a third of its instructions.  Here
// the sums of the cells are carried from round to round, and a pass takes the weights that move out of their old
// cell and adds them to their new one.  The assignment itself is made for every weight in every round, exactly as there.
//
// Assignment.  A lane holds 16 adjacent weights of a row (a whole selection group: no exchange between lanes, and
// what a row costs besides its weights is paid once per 16).  Only the difference of the two errors decides, and
// (x - P)^2 - (x - Q)^2 = x A + B with A = 2 (Q - P), B = P^2 - Q^2 constant on an interval, so the tables hold
// {A, B} and a weight costs one multiply-add and half of a two-wide one where the two errors cost six instructions.
// The low two bits of A are the low bits of the two entries' indices; a funnel shift per weight collects them.
// Rounding: A is within 2.5 units in the last place of its value, B within half a one, x A + B is rounded once, and the sum takes
// 12 additions at most, so |D - D_exact| <= 2^-24 sum I (5 |x A| + |B| + 14 |x A + B|), which is at most `margin` times sum I,
// margin being the maximum over the intervals.  Groups inside that (1e-4 of them) are decided in double.
//
// Moves.  Kept per 16 weights is one word: bit 2 j the low bit of the index of weight j's entry in the table its group has chosen, bit 1 that
// choice.  That is enough to see every move as long as no weight can pass a whole cell in one round, that is as long
// as every breakpoint stays between its old neighbours; the warp that derives the tables checks it, and that no two
// entries of a table are equal.  The old cell of a weight whose bit has changed is then the neighbour on the side
// of the old breakpoint that the weight lies on.  Pieces whose bits differ go on one list of the warp, pieces whose selection
// differs, or is to be decided in double, on another; apply_moves and apply_flips work them off 32 at a time, a piece per
// lane, and change the lane's bins.
//
// Accuracy.  The sums start from a full pass (kKeep), centred on that pass's constants c, and stay centred on them:
// sum I (x - c) and sum I.  T = c + sum I (x - c) / sum I, so an error of sum I counts times T - c, which is the way the
// entry has gone since that pass (0.2 to 0.6 at the end, where a full pass has the 0.01 of a round): the sums of I start
// exact (collect_counts).  A weight leaves a cell with the very term it came with, rounding included, so what is left is one
// FP32 rounding per weight of a cell, as in a full pass, of terms that are larger by |x - c| over |x - T|, and the
// roundings of the few that meet in a bin within a pass.  Tables of one pass against 64-bit sums, 2-norm, mean over 24
// fits of four sizes: 1.2e-10, a full pass 1.0e-10.  The last pass of a fit is a full one, so the tables that are handed
// out have a full pass's error.  A cell that has lost three quarters
// of the most weight it has had (the roundings of all that passed through its bins would weigh four times as much in what
// is left), or gains weight from nothing, ends the incremental rounds before its sum is used.  So do a table out of order, equal entries and a breakpoint
// that passes a neighbour; the rounds that are left are then made by fit_rounds_body.
//
// Objective of a round (Eq. 8), from the same sums: with q = sum I (x - c)^2 carried along like them and d = T - c,
// sum I (x - T)^2 = q - sum over the cells (2 d sum I (x - c) - d^2 sum I).  Where that falls below a sixteenth of the
// largest q there has been, the incremental rounds end, whether a trace is wanted or not, and the round is made in full:
// the difference would have lost four bits, and the terms of the cells' sums are then larger than a full pass's by more
// than four.  (From the third round's constants it is 0.24 to 0.95 of q over 30 rounds, from the first pass's 0.15 to 0.4;
// start tables far from the weights come to 0.01.)
//
// Inner iterations (n_inner > 1).  All passes of the fit but the first and the last run here; in a further inner iteration the kept
// selection stands, and only moves within a table occur.
//
// What bounds it.  A pass over 4096 x 14336 takes 42 us where nothing moves (full rounds: 70), 19 instructions a weight at 72 %
// of the issue slots, the shared-memory pipe 75-80 % busy; with 9-10 % of the pieces moving, as in late rounds, 55-57 us, 11
// SM cycles for each of them: an address per lane, so a wavefront per lane and load, and eight for a weight's two bins.
// Measured against it: list work inside the row loop (its registers spill, 103 us), by all warps at a time between barriers
// (66 us: nothing runs beside it), two, four and eight weights of a flip side by side in half-warps (57, 57, 63 us), the full rounds' form of
// the table (a second lookup for some weights only: 57.8 against 56.5 us), importances from shared memory (56.8 against 55.0 us: less room for the lists).
//
// Work.  A unit is 16 rows (one per warp) x 512 columns; every block takes a contiguous range of the layer's units
// (slab by slab), all of them within one unit of the same length.

// What a pass ends with, as in fit_rounds_body, which spells it out: with these functions in their place its INT4 rounds took
// 1.5 % more.

// ---- a block's sums: half-warp h of warp v adds cell 2 v + h, a lane per warp, pairwise.  wsum: one row of `stride`
//      doubles per warp (residuals, weights, objective) ----
__device__ __forceinline__ void put_block_sums(const double* wsum, const int stride, unsigned long long* acc, const double fix_scale,
                                               const int warp, const int lane) {
    constexpr unsigned kAll = 0xFFFFFFFFu;
    static_assert(kFitWarps == 16 && 2 * kFitWarps == kCells, "a half-warp per cell, a lane per warp");
    const int sum_warp = lane & 15, sum_cell = 2 * warp + (lane >> 4);
    const double* row = wsum + sum_warp * stride;
    double dxs = row[sum_cell], dys = row[kCells + sum_cell];
    double de = 0.0;
    const bool do_e = warp == kFitWarps - 1;
    if (do_e) de = row[2 * kCells];
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
    double sd = (which == 0 ? dxs : which == 1 ? dys : de * 0.0625) * fix_scale;
    if (!(fabs(sd) < 0x1p93)) sd = 0.0;
    const double topm = __dadd_rd(sd * (1.0 / kLimb), kIntMagic);         // floor, as the low bits of a double near 1.5 2^52
    const long long top = __double_as_longlong(topm) - __double_as_longlong(kIntMagic);          // in [-2^46, 2^46)
    const double lowm = __dadd_rd(__fma_rn(-(topm - kIntMagic), kLimb, sd), kIntMagic);
    const long long low = __double_as_longlong(lowm) - __double_as_longlong(kIntMagic);          // in [0, 2^47]
    const unsigned long long add = (unsigned long long)((sum_warp & 1) ? top + kTopBias : low) + kOneArrival;
    if (which < 2) atomicAdd(acc + sum_cell * kAccStride + sum_warp, add);
    else if (do_e && lane < 6 && which == 2) atomicAdd(acc + kCells * kAccStride + (lane - 4), add);
}

// The totals of a pass, lane c those of cell c, lane 0 that of the objective too, as one warp waits for them.  False: the
// wait ran out, here or in another block.
struct Totals { unsigned long long x[2], y[2], e[2]; };
__device__ __forceinline__ bool await_totals(Totals& t, const unsigned long long* acc, const FitParams& p, const int lane) {
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const bool my_e = lane == 0;
    const unsigned long long want = (unsigned long long)p.arrivals;
    t.e[0] = t.e[1] = 0;
    for (unsigned spins = 0;; ++spins) {
        ld_relaxed_2xu64(acc + lane * kAccStride, t.x[0], t.x[1]);
        ld_relaxed_2xu64(acc + lane * kAccStride + 2, t.y[0], t.y[1]);
        if (my_e) ld_relaxed_2xu64(acc + kCells * kAccStride, t.e[0], t.e[1]);
        bool in = true;
#pragma unroll
        for (int l = 0; l < kLimbs; ++l)
            in = in && (t.x[l] >> kCountShift) >= want && (t.y[l] >> kCountShift) >= want && (!my_e || (t.e[l] >> kCountShift) >= want);
        if (__all_sync(kAll, in)) return true;
        if (__any_sync(kAll, spins >= p.spin_limit || ((spins & 15u) == 15u && ld_relaxed_u32(&p.ctrl->abort)))) return false;
    }
}

__device__ __forceinline__ double total_of(const unsigned long long (&w)[2], const unsigned nblk, const double fix_unscale) {
    const unsigned long long sum = w[0] & kLimbMask;         // (its upper bits belong to the top limb)
    const long long low = (long long)(sum & ((1ull << kLimbBits) - 1ull));
    const long long top = (long long)(w[1] & kLimbMask) + (long long)(sum >> kLimbBits) - (long long)nblk * kTopBias;
    const double t = __longlong_as_double(top + __double_as_longlong(kIntMagic)) - kIntMagic;
    const double l = __longlong_as_double(low + __double_as_longlong(kIntMagic)) - kIntMagic;
    return __fma_rn(t, kLimb, l) * fix_unscale;
}

// One warp, lane t with entry t: the entries of either table in ascending order (ties by index); true if any moved.
__device__ __forceinline__ bool sort_tables(FitTables& S, double& T, const int lane) {
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const double Tp = __shfl_up_sync(kAll, T, 1);
    if (!__any_sync(kAll, (lane & 15) != 0 && Tp > T)) return false;
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
    return true;
}

// Fixed-point scale of the sums over the blocks.  The sums of a cell, and a sixteenth of the objective, are
// below B = 16 N sum_k I_k (|w~ - c| < 16, or more with tables of the caller's outside (-8, 8): then B is larger
// by that, squared), so with 2^e > B the value v 2^(93 - e) fits the limbs.  What is dropped lies 2^-93 below
// B: also a cell whose only weight has 10^-20 of the importances' sum moves its entry.  Integer addition is
// order-independent, so the totals do not depend on the order in which the blocks arrive.
// Every thread calls; part: a double per warp, `stride` apart.  Warp 0 returns {scale, its inverse} in every lane.
__device__ __forceinline__ double2 fixed_point_scale(const FitParams& p, double* part, const int stride, const int tid) {
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int lane = tid & 31, warp = tid >> 5, K = (int)p.K;
    float sum = 0.f;
    for (int k = tid; k < K; k += kFitWarps * 32) sum = __fadd_ru(sum, fabsf(__ldg(p.I + k)));
#pragma unroll
    for (int o = 16; o; o >>= 1) sum = __fadd_ru(sum, __shfl_xor_sync(kAll, sum, o));
    if (p.reach) sum = __fmul_ru(sum, *p.reach);
    if (lane == 0) part[warp * stride] = (double)sum;
    __syncthreads();
    double2 r = make_double2(1.0, 1.0);
    if (warp == 0) {
        double B = part[(lane & 15) * stride];
#pragma unroll
        for (int o = 8; o; o >>= 1) B += __shfl_xor_sync(kAll, B, o);
        B *= 257.0 / 16.0 * (double)(int)p.N;
        const int e = B > 0.0 && B < 1e300 ? ilogb(B) + 1 : 0;
        r = make_double2(scalbn(1.0, kSumBits - e), scalbn(1.0, e - kSumBits));
    }
    return r;
}

// The 32 lane-private values of every cell of a warp's bins, added in double: lane c returns cell c's (in an order of
// its own that avoids bank conflicts, and a fixed one).  In double, 32 FP32 values are added without rounding
// unless they are more than 2^24 apart.
__device__ __forceinline__ double2 warp_sums(const uint32_t bins_warp, const int lane) {
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
    return make_double2(((dx[0] + dx[1]) + (dx[2] + dx[3])) * 0x1p896, ((dy[0] + dy[1]) + (dy[2] + dy[3])) * 0x1p896);
}

constexpr int kDeltaCols = 512;                       // columns of a slab
// A warp's list: moves from the front, flips from the back.  Behind a pass its place holds the warp's sums (66
// doubles); the 16 bytes spread the warps over the banks.
constexpr int kDeltaCap = 110;
constexpr int kLeastFlips = 20;                       // flips that are worked off before the end of a pass
constexpr int kDeltaScales = kDeltaCap * 8;           // the entries' reciprocal scales, behind the entries
constexpr int kDeltaWeights = kDeltaCap * 12;         // the moving weights being worked off (63 at most), two bytes each
constexpr int kDeltaList = kDeltaWeights + 192 + 16;
static_assert(192 >= 2 * 63, "room for the moving weights");
static_assert(kDeltaList % 8 == 0, "the sums are doubles");
constexpr int kDeltaBins = kCells * kSlotBytes;       // a warp's bins (no spare slot)
// a flip's entry is {piece | flags, old word}, a move's {piece, changed bits | selection in bit 1}; a piece's number is
// below 2^28 (a layer has less than 2^32 elements)
constexpr uint32_t kPieceMask = (1u << 28) - 1u, kSelected = 1u << 28, kUndecided = 1u << 29;

struct DeltaShared {
    FitTables t;
    double sx[kCells], sw[kCells], sw_most[kCells];   // the cells' sums, and the largest weight sums that they have had
    double q, q_most;
    double fix_scale, fix_unscale;
    float2 ab[kJSlots];                           // {A, B} of every interval
    uint2 row[kJSlots];                           // {its upper breakpoint, the entries' indices in T0, T1 on it and on the next (four bits each)}
    float c[kCells];                              // the constants the sums are centred on
    float mid_old[kCells];                        // breakpoints of the tables of the pass before, by table (those of this pass: t.tmp_b)
    float margin;
    int failed, stop;
    uint8_t low[kNBins];                          // interval of every bin's lower edge
};

// no weight's entry index changes by more than one between tables with the breakpoints a and b (by table, lane's own at [lane])
__device__ __forceinline__ bool interlaced(const float* a, const float* b, const int lane) {
    const bool ok = (lane & 15) == 15 || (a[lane + 1] >= b[lane] && b[lane + 1] >= a[lane]);
    return __all_sync(0xFFFFFFFFu, ok);
}

// {A, B} of the intervals and the margin, behind derive_tables; one warp, lane J with interval J
__device__ __forceinline__ void derive_differences(DeltaShared& sh, const int lane) {
    const FitTables& S = sh.t;
    const double2 pq = S.PQ[lane];
    const float2 e = S.pq32[lane];
    const double A = 2.0 * (pq.y - pq.x), B = (pq.x - pq.y) * (pq.x + pq.y);
    const uint32_t low = (__float_as_uint(e.x) & 1u) | ((__float_as_uint(e.y) & 1u) << 1);
    const uint32_t a = __float_as_uint((float)A);
    // the nearest float with these low bits
    const float fa = __uint_as_float((a & 0x80000000u) | (((max(a & 0x7FFFFFFFu, 4u) + 2u - low) & ~3u) + low));
    const float fb = (float)B;
    const bool real = lane < kNJ;
    const float nan = __int_as_float(0x7FC00000);
    sh.ab[lane] = real ? make_float2(fa, fb) : make_float2(nan, nan);
    const float lo = lane == 0 ? -8.f : S.bp[max(lane, 1) - 1], hi = lane < kNBP ? S.bp[lane] : 8.f;
    float m = real ? 5.f * fmaxf(fabsf(lo), fabsf(hi)) * fabsf(fa) + fabsf(fb) +
                         14.f * fmaxf(fabsf(fmaf(lo, fa, fb)), fabsf(fmaf(hi, fa, fb)))
                   : 0.f;
#pragma unroll
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    const uint32_t idx = (__float_as_uint(e.x) & kIdxMask) | ((__float_as_uint(e.y) & kIdxMask) << 4);
    sh.row[lane] = make_uint2(__float_as_uint(S.bp[lane]), idx | (__shfl_down_sync(0xFFFFFFFFu, idx, 1) << 8));
    if (lane == 0) sh.margin = m * (0x1p-24f * 1.01f);
}

// the entries nearest to x: index in T0, index in T1 << 4
__device__ __forceinline__ uint32_t entries_of(const DeltaShared* sh, float x) {
    constexpr float kMagic = (float)(kNBins / 2) + 1.5f * (float)(1 << 23) / (float)(kRep * 8);
    const uint32_t bin = (__float_as_uint(__fmaf_rn(x, (float)(kNBins / 16), kMagic)) / (kRep * 8)) & (uint32_t)(kNBins - 1);
    const uint32_t J = sh->low[bin];
    if (J == kNoHint) return sh->row[find_interval(sh->t.bp, x)].y;
    const uint2 r = sh->row[J];
    return x > __uint_as_float(r.x) ? r.y >> 8 : r.y;
}

// the quotient of a piece's number and the pieces per row: m = floor(2^32 / K16)
__device__ __forceinline__ unsigned row_of(unsigned at, unsigned K16, unsigned m) {
    const unsigned q = __umulhi(at, m);                   // (at < 2^28: the row or one less)
    return q + (at - q * K16 >= K16 ? 1u : 0u);
}

// A weight's terms in its old and its new cell, and what it adds to q; then the change of the lane's bins.  (Apart, so
// that the loads of several weights' constants stand before the first bin is written.)
struct Move { float from, to; };
__device__ __forceinline__ Move move_terms(const DeltaShared* sh, const uint32_t from, const uint32_t to, const float x, const float I, float& dq) {
    const float u0 = __fsub_rn(x, sh->c[from]), u1 = __fsub_rn(x, sh->c[to]);
    const Move m{__fmul_rn(I, u0), __fmul_rn(I, u1)};
    if (from != to) dq = __fmaf_rn(m.to, u1, __fmaf_rn(-m.from, u0, dq));
    return m;
}
__device__ __forceinline__ void move_weight(const uint32_t bins_lane, const uint32_t from, const uint32_t to, const Move& m, const float I) {
    const uint32_t a0 = bins_lane + from * kSlotBytes, a1 = bins_lane + to * kSlotBytes;
    float2 b0 = lds_bin(a0), b1 = lds_bin(a1);
    b0.x -= m.from;
    b0.y -= I;
    b1.x += m.to;
    b1.y += I;
    sts_bin(a0, b0);
    sts_bin(a1, b1);
}

struct DeltaArgs {                // what the list work needs of the layer
    const uint16_t* W;
    int64_t K, ldw;
    const uint8_t* scales;
    const float* I;
    uint32_t* kept;
    unsigned k16_inv;             // floor(2^32 / (K / 16))
};

// Works off the list's first `count` pieces, in which weights move within their table: first the moving weights are put
// into a row (most pieces have one, few more than two), then every lane takes one of them (two: 1 % slower).  Every lane
// calls; returns what the lane's weights add to q.
__device__ __noinline__ float apply_moves(const DeltaShared* sh, const DeltaArgs p, const uint32_t list_at, const int count,
                                          const uint32_t bins_lane, const int lane) {
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const unsigned K16 = (unsigned)p.K / 16u;
    const uint32_t row_at = list_at + kDeltaWeights, below = (1u << lane) - 1u;
    float dq = 0.f;
    uint32_t left = 0u, piece = 0u;
    int next = 0, n = 0;
    for (;;) {
        for (;;) {
            const unsigned some = __ballot_sync(kAll, left != 0u);
            if (some == 0u) {
                if (next >= count) break;
                piece = (uint32_t)(next + lane);
                if (next + lane < count) {
                    uint32_t at;
                    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(at), "=r"(left) : "r"(list_at + piece * 8u) : "memory");
                    left &= 0x55555555u;
                    atomicXor(p.kept + at, left);          // (nobody waits for it; the pass's loads of these words go past the L1)
                }
                next += 32;
                continue;
            }
            if (left) {
                const uint32_t j = (uint32_t)(__ffs(left) - 1) >> 1;
                left &= left - 1u;
                asm volatile("st.shared.u16 [%0], %1;" :: "r"(row_at + (uint32_t)(n + __popc(some & below)) * 2u), "h"((uint16_t)(piece | (j << 8))) : "memory");
            }
            n += __popc(some);
            if (n >= 32) break;
        }
        if (n == 0) return dq;
        const int take = min(n, 32);
        n -= take;
        __syncwarp();
        uint32_t w = 0u, table = 0u;
        float iv = 0.f, x = 0.f;
        if (lane < take) {
            uint32_t ej, at, word;
            asm volatile("ld.shared.u16 %0, [%1];" : "=r"(ej) : "r"(row_at + (uint32_t)(n + lane) * 2u) : "memory");
            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(at), "=r"(word) : "r"(list_at + (ej & 255u) * 8u) : "memory");
            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x) : "r"(list_at + kDeltaScales + (ej & 255u) * 4u) : "memory");
            const unsigned row = row_of(at, K16, p.k16_inv), col = (at - row * K16) * 16u + (ej >> 8);
            w = __ldg(p.W + (row * (unsigned)p.ldw + col));
            iv = __ldg(p.I + col);
            table = (word & 2u) ? (uint32_t)kM : 0u;
        }
        x = __fmul_rn(__uint_as_float(w << 16), x);
        const uint32_t in = (entries_of(sh, x) >> (table / 4u)) & kIdxMask, to = table + in;
        const uint32_t from = table + ((x > sh->mid_old[to] ? in + 1u : in - 1u) & kIdxMask);
        const Move m = move_terms(sh, from, to, x, iv, dq);
        if (lane < take) move_weight(bins_lane, from, to, m, iv);
        __syncwarp();
    }
}

// Works off the list's last `count` pieces, whose selection has changed or is open: all their weights move.  A lane takes
// a piece, four weights side by side.  Every lane calls; returns what the lane's weights add to q.
__device__ __noinline__ float apply_flips(const DeltaShared* sh, const DeltaArgs p, const uint32_t list_at, const int count,
                                          const uint32_t bins_lane, const int lane) {
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const FitTables& S = sh->t;
    const unsigned K16 = (unsigned)p.K / 16u;
    const uint32_t list_addr = list_at + (uint32_t)(kDeltaCap - count) * 8u, scales_at = list_at + (uint32_t)(kDeltaScales + (kDeltaCap - count) * 4);
    // the open ones: Eq. 8 in double, a weight per lane, in the order of resolve_deferred
    for (int first = 0; first < count; first += 32) {
        uint32_t at = 0u;
        if (first + lane < count) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(at) : "r"(list_addr + (uint32_t)(first + lane) * 8u) : "memory");
        unsigned open = __ballot_sync(kAll, (at & kUndecided) != 0u);
        for (; open; open &= open - 1u) {
            const int who = __ffs(open) - 1;
            const unsigned a = __shfl_sync(kAll, at, who) & kPieceMask;
            double e0 = 0.0, e1 = 0.0;
            if (lane < 16) {
                const unsigned r = row_of(a, K16, p.k16_inv), col = (a - r * K16) * 16u + (unsigned)lane;
                const uint32_t wb = p.W[r * (unsigned)p.ldw + col];
                const float x = __fmul_rn(__uint_as_float(wb << 16), S.rlut[p.scales[a] & 0x7Fu]);
                const double2 pq = S.PQ[find_interval(S.bp, x)];
                const double xd = (double)x, id = (double)__ldg(p.I + col);
                const double d0 = __dsub_rn(xd, pq.x), d1 = __dsub_rn(xd, pq.y);
                e0 = __dmul_rn(id, __dmul_rn(d0, d0));
                e1 = __dmul_rn(id, __dmul_rn(d1, d1));
            }
#pragma unroll
            for (int o = 8; o; o >>= 1) {
                e0 = __dadd_rn(e0, __shfl_xor_sync(kAll, e0, o));
                e1 = __dadd_rn(e1, __shfl_xor_sync(kAll, e1, o));
            }
            const bool second = __shfl_sync(kAll, (int)(e1 < e0), 0) != 0;
            if (lane == who) {
                at = second ? at | kSelected : at & ~kSelected;
                asm volatile("st.shared.u32 [%0], %1;" :: "r"(list_addr + (uint32_t)(first + lane) * 8u), "r"(at) : "memory");
            }
        }
    }
    __syncwarp();
    float dq = 0.f;
    for (int first = 0; first < count; first += 32) {
        if (first + lane >= count) continue;
        uint32_t at, old;
        float rinv;
        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(at), "=r"(old) : "r"(list_addr + (uint32_t)(first + lane) * 8u) : "memory");
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(rinv) : "r"(scales_at + (uint32_t)(first + lane) * 4u) : "memory");
        const uint32_t tn = (at & kSelected) ? (uint32_t)kM : 0u, to = (old & 2u) ? (uint32_t)kM : 0u;
        at &= kPieceMask;
        const unsigned row = row_of(at, K16, p.k16_inv), col = (at - row * K16) * 16u;
        const uint16_t* const W = p.W + (row * (unsigned)p.ldw + col);
        const float* const I = p.I + col;
        uint32_t word = tn ? 2u : 0u;
        uint4 w = __ldg(reinterpret_cast<const uint4*>(W));
#pragma unroll 1
        for (uint32_t q = 0; q < 2; ++q) {
            const uint4 wc = w;
            if (q == 0) w = __ldg(reinterpret_cast<const uint4*>(W + 8));      // (the next eight are asked for meanwhile)
            const uint32_t ws[4] = {wc.x, wc.y, wc.z, wc.w}, was = old >> (16u * q);
            const float4 i0 = __ldg(reinterpret_cast<const float4*>(I + 8u * q)), i1 = __ldg(reinterpret_cast<const float4*>(I + 8u * q + 4u));
            const float Iv[8] = {i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, i1.z, i1.w};
            uint32_t bits = 0u;
#pragma unroll
            for (int h = 0; h < 8; h += 4) {
                uint32_t from[4], into[4];
                float x[4];
                Move m[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    x[t] = __fmul_rn((t & 1) ? bf16_hi(ws[(h + t) / 2]) : bf16_lo(ws[(h + t) / 2]), rinv);
                    const uint32_t c = entries_of(sh, x[t]);
                    const uint32_t in = (c >> (tn / 4u)) & kIdxMask;
                    uint32_t io = (c >> (to / 4u)) & kIdxMask;
                    if (((was >> (2 * (h + t))) ^ io) & 1u) io = (x[t] > sh->mid_old[to + io] ? io + 1u : io - 1u) & kIdxMask;
                    from[t] = to + io;
                    into[t] = tn + in;
                    bits |= (in & 1u) << (2 * (h + t));
                }
#pragma unroll
                for (int t = 0; t < 4; ++t) m[t] = move_terms(sh, from[t], into[t], x[t], Iv[h + t], dq);
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (from[t] != into[t]) move_weight(bins_lane, from[t], into[t], m[t], Iv[h + t]);
            }
            word |= bits << (16u * q);
        }
        p.kept[at] = word;
    }
    return dq;
}

// The incremental passes of one layer, from the first after the kKeep launch to p.n_rounds, run by the blocks
// bid = 0 .. nblk - 1.  Layout in shared memory as in fit_rounds_body.
__device__ __forceinline__ void delta_rounds_body(const FitParams& p, const unsigned bid, const unsigned nblk) {
    constexpr int NW = kFitWarps, NB = kNBins, REP = kRep, NT = NW * 32;
    constexpr unsigned kAll = 0xFFFFFFFFu;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ DeltaShared sh;
    FitTables& S = sh.t;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    const uint32_t dyn_at = (uint32_t)__cvta_generic_to_shared(dyn);
    const uint32_t sm_base = (dyn_at + 255u) & ~255u;
    uint32_t dyn_size;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn_size));
    const int n_low = min(NW, (int)((kLut1At - sm_base) / (uint32_t)kDeltaBins));
    const uint32_t hi_base = kLut1At + kLut1Bytes;
    const uint32_t lut2_addr = hi_base + (uint32_t)(NW - n_low) * kDeltaBins;
    const uint32_t lists_at = lut2_addr + kLut2Bytes;
    if (sm_base > kLut1At || lists_at + NW * kDeltaList > dyn_at + dyn_size) {
        if (bid == 0 && threadIdx.x == 0 && p.dev_status) atomicOr(p.dev_status, AAAC_DEV_TIMEOUT);
        return;
    }
    const uint32_t lut1_or = kLut1At | ((lane & (REP - 1)) * 8);
    const uint32_t bins_warp = warp < n_low ? sm_base + warp * kDeltaBins : hi_base + (uint32_t)(warp - n_low) * kDeltaBins;
    const uint32_t bins_lane = bins_warp + lane * 8;
    const uint32_t list_at = lists_at + warp * kDeltaList;
    constexpr int kSumStride = kDeltaList / 8;
    static_assert(kDeltaList % 8 == 0 && kSumStride >= 2 * kCells + 2, "a warp's sums fit its lists' place");
    double* const wsums = reinterpret_cast<double*>(dyn + (lists_at - dyn_at));

    Ctrl& ctl = *p.ctrl;
    const int first_round = (int)ctl.next_round;
    if (!ctl.keep_ok || first_round >= p.n_rounds) return;
    unsigned pass_no = ctl.passes;

    const int N = (int)p.N, K = (int)p.K;
    const unsigned K16 = (unsigned)K / 16u;
    const int nrb = (N + NW - 1) / NW, slabs = (K + kDeltaCols - 1) / kDeltaCols;
    const int64_t units = (int64_t)slabs * nrb;
    const int t0 = (int)(units * bid / nblk), n_units = (int)(units * (bid + 1) / nblk) - t0;
    const int slab0 = t0 / nrb, rb0 = t0 - slab0 * nrb;

    // Row registers of two units, refilled as soon as they are unpacked with the unit after next; behind the last
    // unit of a pass come the first ones again.
    uint4 v[2][2];
    uint32_t sc[2], kw[2];
    int lslab = slab0, lrb = rb0, lleft = n_units;         // the unit to be loaded next
    auto offsets = [&](unsigned& wo, unsigned& ko) {       // elements of W; scales and kept words
        const unsigned row = (unsigned)min(lrb * NW + warp, N - 1);
        const unsigned piece = min((unsigned)(lslab * 32 + lane), K16 - 1u);
        wo = row * (unsigned)p.ldw + piece * 16u;
        ko = row * K16 + piece;
    };
    auto load_unit = [&](int s) {
        unsigned wo, ko;
        offsets(wo, ko);
        asm volatile("ld.global.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(v[s][0].x), "=r"(v[s][0].y), "=r"(v[s][0].z), "=r"(v[s][0].w), "=r"(v[s][1].x), "=r"(v[s][1].y), "=r"(v[s][1].z),
                       "=r"(v[s][1].w)
                     : "l"(p.W + wo));
        asm volatile("ld.global.u8 %0, [%1];" : "=r"(sc[s]) : "l"(p.scales + ko));
        asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(kw[s]) : "l"(p.kept + ko) : "memory");
        if (--lleft == 0) {
            lleft = n_units;
            lslab = slab0;
            lrb = rb0;
        } else if (++lrb == nrb) {
            lrb = 0;
            ++lslab;
        }
    };
    if (n_units > 0) {
        load_unit(0);
        load_unit(1);
    }

    if (tid >= 64 && tid < 192) {
        const int c = tid - 64;
        const float sv = __fmul_rn(e4m3_value((uint32_t)c), ctl.s_t);
        S.rlut[c] = c ? __frcp_rn(sv) : 0.f;
    }
    {
        const double2 fix = fixed_point_scale(p, wsums, kSumStride, tid);
        if (warp == 0) {
            const double before = ctl.keep_T[lane], T = ctl.T[lane];
            derive_tables(S, lane, before);
            __syncwarp();
            bool good = S.no_dup != 0;
            sh.mid_old[lane] = S.tmp_b[lane];
            __syncwarp();
            derive_tables(S, lane, T);
            __syncwarp();
            derive_differences(sh, lane);
            const double bp = __shfl_up_sync(kAll, before, 1);
            good = interlaced(sh.mid_old, S.tmp_b, lane) && good && S.no_dup && !__any_sync(kAll, (lane & 15) != 0 && !(bp <= before));
            sh.sx[lane] = ctl.keep_sx[lane];
            sh.sw[lane] = sh.sw_most[lane] = ctl.keep_sw[lane];
            sh.c[lane] = ctl.keep_c[lane];
            if (lane == 0) {
                sh.q = sh.q_most = ctl.keep_q;
                sh.fix_scale = fix.x;
                sh.fix_unscale = fix.y;
                sh.failed = 0;
                sh.stop = !good;
            }
        }
    }
    for (int b = 0; b < kCells; ++b) sts_bin(bins_lane + b * kSlotBytes, make_float2(0.f, 0.f));
    __syncthreads();
    if (sh.stop) return;                                   // (the control block says that every round is left)
    write_tables<NT, false>(S, sh.ab, tid, kLut1At, lut2_addr, sh.low);
    __syncthreads();

    constexpr float kBinsPerUnit = (float)(NB / 16);
    constexpr float kMagic = (float)(NB / 2) + 1.5f * (float)(1 << 23) / (float)(REP * 8);
    constexpr uint32_t kBinMask = (uint32_t)(NB - 1) * (REP * 8);
    const DeltaArgs args{p.W, p.K, p.ldw, p.scales, p.I, p.kept, (unsigned)((1ull << 32) / (unsigned long long)K16)};

    uint64_t II[8];           // importances of the lane's columns, in pairs
    float isum = 0.f;         // sum of |I| over the lane's group (rounded up a little)
    int have_slab = -1;
#pragma unroll
    for (int j = 0; j < 8; ++j) II[j] = 0ull;

    int round = first_round;  // counts passes
    int inner = first_round % p.n_inner;
    for (;;) {
        const bool frozen = inner != 0;                    // a further inner iteration: the selection stands
        // (block 0 clears the buffer of the next pass, as in fit_rounds_body)
        static_assert(NT >= 256 + kCells * 4 + kLimbs, "threads 256.. of block 0 clear the next buffer");
        if (bid == 0 && tid >= 256 && tid < 256 + kCells * 4 + kLimbs) {
            const int w = tid - 256;
            p.acc[(size_t)((pass_no + 1u) % 3u) * kAccBuffer + (size_t)(w >> 2) * kAccStride + (w & 3)] = 0ull;
            __threadfence();
        }
        const float margin = sh.margin;
        float tau = __fmul_ru(isum, margin);
        double dq = 0.0;
        int n_moves = 0, n_flips = 0;

        // Stages of half a unit (8 weights): L1 the bins' entries; L2 the second lookups; E the difference of the errors and the index
        // bits.  D, per unit: the group's difference, its selection, and the lists.  L1 of the next half comes before L2 of this one.
        float x[2][8];
        uint64_t ab[2][8];
        uint64_t sum = 0ull;
        uint32_t bits = 0;
        auto L1 = [&](const uint4& vv, const float rinv, const int b) {
            const uint32_t w[4] = {vv.x, vv.y, vv.z, vv.w};
            const uint64_t rr = pack2(rinv, rinv);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint64_t xx = mul2(pack2(bf16_lo(w[j]), bf16_hi(w[j])), rr);
                const uint64_t bb = fma2(xx, pack2(kBinsPerUnit, kBinsPerUnit), pack2(kMagic, kMagic));
                unpack2(xx, x[b][2 * j], x[b][2 * j + 1]);
                ab[b][2 * j] = lds_table_b64((__float_as_uint(lo2(bb)) & kBinMask) | lut1_or);
                ab[b][2 * j + 1] = lds_table_b64((__float_as_uint(hi2(bb)) & kBinMask) | lut1_or);
            }
        };
        auto L2 = [&](const int b) {
#pragma unroll
            for (int j = 0; j < 8; ++j) ab[b][j] = lds_table_b64(above_addr((uint32_t)ab[b][j], x[b][j], (uint32_t)(ab[b][j] >> 32)));
        };
        auto E = [&](const int b) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint64_t d = pack2(__fmaf_rn(x[b][2 * j], lo2(ab[b][2 * j]), hi2(ab[b][2 * j])),
                                         __fmaf_rn(x[b][2 * j + 1], lo2(ab[b][2 * j + 1]), hi2(ab[b][2 * j + 1])));
                sum = fma2(II[4 * b + j], d, sum);
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) bits = __funnelshift_r(bits, __float_as_uint(lo2(ab[b][j])), 2);
        };
        auto rinv_of = [&](uint32_t s) { return S.rlut[s & 0x7Fu]; };

        int slab = slab0, rb = rb0;
        float rinv = 0.f;
        // one unit; true if the lists have to be worked off before the next
        auto unit = [&](const int s) {
            if (slab != have_slab) {
                have_slab = slab;
                const int col0 = slab * kDeltaCols + lane * 16;
                isum = 0.f;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 a = col0 < K ? __ldg(reinterpret_cast<const float4*>(p.I + col0) + j) : make_float4(0.f, 0.f, 0.f, 0.f);
                    II[2 * j] = pack2(a.x, a.y);
                    II[2 * j + 1] = pack2(a.z, a.w);
                    isum += (fabsf(a.x) + fabsf(a.y)) + (fabsf(a.z) + fabsf(a.w));
                }
                isum *= 1.0001f;
                tau = __fmul_ru(isum, margin);
            }
            const uint32_t old = kw[s];
            const int row = rb * NW + warp;
            const uint32_t piece = (uint32_t)(slab * 32 + lane);
            L1(v[s][1], rinv, 1);
            load_unit(s);
            sum = 0ull;
            L2(0);
            E(0);
            const float rinv_now = rinv;
            rinv = rinv_of(sc[s ^ 1]);
            L1(v[s ^ 1][0], rinv, 0);                      // (for nothing at the end of a pass, or before the lists are worked off)
            L2(1);
            E(1);
            const float d = lo2(sum) + hi2(sum);
            // (a NaN, from a poisoned row, counts as a flip also where the selection stands)
            const bool near = !(fabsf(d) > tau) && !(frozen && d == d);
            const uint32_t sg = frozen ? (old >> 1) & 1u : d > 0.f ? 1u : 0u;
            const uint32_t now = ((bits >> sg) & 0x55555555u) | (sg << 1);
            const uint32_t diff = now ^ old;
            const bool ok = row < N && piece < K16;
            const bool flip = ok && (near || (diff & 2u) != 0u), move = ok && !flip && diff != 0u;
            const unsigned fm = __ballot_sync(kAll, flip), mm = __ballot_sync(kAll, move);
            const uint32_t at = (uint32_t)row * K16 + piece;
            const int e = move ? n_moves + __popc(mm & ((1u << lane) - 1u)) : kDeltaCap - n_flips - __popc(fm & ((2u << lane) - 1u));
            if (flip || move) {
                sts_u2(list_at + (uint32_t)e * 8u, move ? at : at | (sg ? kSelected : 0u) | (near && !frozen ? kUndecided : 0u),
                       move ? (diff & 0x55555555u) | (sg << 1) : old);
                asm volatile("st.shared.f32 [%0], %1;" :: "r"(list_at + (uint32_t)(kDeltaScales + e * 4)), "f"(rinv_now) : "memory");
            }
            n_moves += __popc(mm);
            n_flips += __popc(fm);
            if (++rb == nrb) { rb = 0; ++slab; }
            return n_moves + n_flips > kDeltaCap - 32 || n_flips >= 32;
        };
        for (int i = 0; i < n_units;) {
            rinv = rinv_of(sc[0]);
            L1(v[0][0], rinv, 0);
            for (;;) {
                const bool full0 = unit(0);
                if (++i == n_units || full0) {             // the next unit is in the second registers
#pragma unroll
                    for (int h = 0; h < 2; ++h) { const uint4 a = v[0][h]; v[0][h] = v[1][h]; v[1][h] = a; }
                    uint32_t a = sc[0];
                    sc[0] = sc[1];
                    sc[1] = a;
                    a = kw[0];
                    kw[0] = kw[1];
                    kw[1] = a;
                    break;
                }
                const bool full1 = unit(1);
                if (++i == n_units || full1) break;
            }
            // (out of the loop above, whose registers would be spilled in its midst)
            __syncwarp();
            if (n_moves > 0) dq += (double)apply_moves(&sh, args, list_at, n_moves, bins_lane, lane);
            n_moves = 0;
            if (n_flips > (i < n_units ? kLeastFlips - 1 : 0)) {
                dq += (double)apply_flips(&sh, args, list_at, n_flips, bins_lane, lane);
                n_flips = 0;
            }
            __syncwarp();
        }
        __syncwarp();
        // (the first two units' kept words were loaded ahead, perhaps before their last listed pieces were worked off)
        if (n_units > 0) {
            const int s_slab = lslab, s_rb = lrb;
            lslab = slab0;
            lrb = rb0;
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                unsigned wo, ko;
                offsets(wo, ko);
                asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(kw[s]) : "l"(p.kept + ko) : "memory");
                if (n_units > 1 && ++lrb == nrb) { lrb = 0; ++lslab; }
            }
            lslab = s_slab;
            lrb = s_rb;
        }
        {
            const double2 ws = warp_sums(bins_warp, lane);
            double* const row = wsums + warp * kSumStride;
            row[lane] = ws.x;
            row[kCells + lane] = ws.y;
#pragma unroll
            for (int s = 16; s; s >>= 1) dq += __shfl_xor_sync(kAll, dq, s);
            if (lane == 0) row[2 * kCells] = dq;
        }
        __syncthreads();
        unsigned long long* const acc = p.acc + (size_t)(pass_no % 3u) * kAccBuffer;
        put_block_sums(wsums, kSumStride, acc, sh.fix_scale, warp, lane);
        if (warp) {
#pragma unroll 8
            for (int b = 0; b < kCells; ++b) sts_bin(bins_lane + b * kSlotBytes, make_float2(0.f, 0.f));
            if (warp == 1) {
#pragma unroll 8
                for (int b = 0; b < kCells; ++b) sts_bin((n_low > 0 ? sm_base : hi_base) + lane * 8 + b * kSlotBytes, make_float2(0.f, 0.f));
            }
        }
        ++pass_no;
        if (warp == 0) {
            Totals t;
            if (!await_totals(t, acc, p, lane)) {
                if (lane == 0) sh.failed = 1;
            } else {
                const double sx = sh.sx[lane] + total_of(t.x, nblk, sh.fix_unscale), sw = sh.sw[lane] + total_of(t.y, nblk, sh.fix_unscale);
                const double most = sh.sw_most[lane], c = (double)sh.c[lane], before = S.Td[lane], d = before - c;
                double f = d * (2.0 * sx - d * sw);
#pragma unroll
                for (int s = 16; s; s >>= 1) f += __shfl_xor_sync(kAll, f, s);
                const double q = sh.q + 16.0 * total_of(t.e, nblk, sh.fix_unscale), q_most = fmax(sh.q_most, q), err = q - f;
                const bool used = (most > 0.0 ? sw > 0.25 * most : most == 0.0 && sw == 0.0) && (lane || err >= 0.0625 * q_most);
                if (!__all_sync(kAll, used)) {
                    if (lane == 0) sh.stop = 1;                    // this round is not used
                } else {
                    double T = sw > 0.0 ? c + __ddiv_rn(sx, sw) : before;
                    if (lane == 0) {
                        sh.q = q;
                        sh.q_most = q_most;
                        if (bid == 0 && !frozen && p.err_trace) p.err_trace[round / p.n_inner] = err;
                    }
                    sh.sx[lane] = sx;
                    sh.sw[lane] = sw;
                    sh.sw_most[lane] = fmax(most, sw);
                    sh.mid_old[lane] = S.tmp_b[lane];
                    const bool moved = sort_tables(S, T, lane);
                    __syncwarp();
                    derive_tables(S, lane, T);
                    __syncwarp();
                    derive_differences(sh, lane);
                    const bool good = interlaced(sh.mid_old, S.tmp_b, lane) && !moved && S.no_dup;
                    if (lane == 0 && !good) sh.stop = 2;           // this round is; the next needs a full pass
                }
            }
        }
        __syncthreads();
        if (sh.failed) {
            if (tid == 0) {
                atomicExch(&ctl.abort, 1u);
                if (p.dev_status) atomicOr(p.dev_status, AAAC_DEV_TIMEOUT);
            }
            return;
        }
        if (sh.stop != 1) ++round;
        if (++inner == p.n_inner) inner = 0;
        if (sh.stop || round >= p.n_rounds) break;
        write_tables<NT, false>(S, sh.ab, tid, kLut1At, lut2_addr, sh.low);
        __syncthreads();
    }
    if (bid == 0 && tid < 2 * kM) {
        ctl.T[tid] = S.Td[tid];
        if (p.T01_out) p.T01_out[tid] = (float)S.Td[tid];
        if (tid == 0) {
            ctl.first_incremental = (uint32_t)first_round;
            ctl.next_round = ctl.end_incremental = (uint32_t)round;
            ctl.passes = pass_no;
        }
    }
}

__global__ void __launch_bounds__(kFitWarps * 32, 1) delta_kernel(const __grid_constant__ FitBatch b) {
    if (b.first[1] == gridDim.x) { delta_rounds_body(b.L[0], blockIdx.x, gridDim.x); return; }
    int l = 0;
    while (l + 1 < kMaxBatch && blockIdx.x >= b.first[l + 1]) ++l;
    delta_rounds_body(b.L[l], blockIdx.x - b.first[l], b.first[l + 1] - b.first[l]);
}
