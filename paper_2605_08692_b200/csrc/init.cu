// Initial tables (Algorithm 1 lines 4-5).
//
// Quantile initialisation (Eq. 9, Eq. 10): T0[i] = Quantile_{i/15}, T1[i] = Quantile_{d + (1-d) i/15},
// d = 1/30, of all N*K normalised weights, with linear interpolation at position q (n - 1).
// That needs up to 64 exact order statistics of n values.  They are selected without sorting:
//   1. histogram of every w~ over 16384 uniform bins on [-8, 8): counted by the scales pass
//      (scales_hist_kernel);
//   2. one block turns the histogram into a prefix sum, finds the bin and the rank inside the
//      bin of every requested order statistic, and gives each distinct bin a slot;
//   3. a second pass over W appends the (order-preserving integer keys of the) values that fall
//      into a slotted bin to that slot's list -- the lists' sizes are known from step 1.  A block
//      stages its candidates in shared memory and reserves list space once per slot, so the
//      global counters see one atomic per block and slot instead of one per candidate;
//   4. one block per slot selects the requested ranks of its list by an 11-bit radix select (the
//      list is read once into registers when it is short enough, else streamed per pass);
//   5. the table entries are interpolated in double and rounded to FP32.
// Integer atomics only, so the result does not depend on scheduling.
//
// Grid initialisation: T0 = the format's table (INT4: -8..7, NVFP4: signed E2M1 with both
// zeros), T1[i] = (T0[i] + T0[i+1]) / 2 and T1[15] = T0[15] + (T0[15] - T0[14]) / 2.
#include <algorithm>

#include "internal.cuh"

namespace aaac {

namespace {

__device__ __forceinline__ uint32_t float_key(float f) {      // order-preserving; -0 and +0 share a key
    uint32_t u = __float_as_uint(f);
    if (u == 0x80000000u) u = 0u;
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
constexpr uint32_t kSlotOver = 0x40u;      // bin -> slot table: the slot's candidates have no room in the list
__device__ __forceinline__ float key_float(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}
// Step 3: candidates of the slotted bins, staged per block.
//
// One lane in eight holds a candidate among their eight weights, nearly always a single one, so working on
// candidates where they are found leaves most of a warp idle for half of the pass's instructions.  Such lanes put
// their weights on a queue of the warp, and the warp works on 32 of them at a time (14336 x 4096 NVFP4: scales + start 150.9 -> 143.2 us, INT4 135.4 -> 126.7).
constexpr int kStageCap = 3072;                  // staged candidates per block
constexpr int kStageEvery = 4;                   // loop iterations between two looks at the stage's fill
constexpr int kQueue = 64;                       // queued lanes per warp: up to 31 left over and 32 more

template <int MODE, bool DENSE>
__global__ void __launch_bounds__(256)
quantile_collect_kernel(const uint16_t* __restrict__ W, unsigned n_pieces, unsigned per_row, int64_t ldw,
                        const void* __restrict__ scales, Ctrl* ctrl, const uint8_t* __restrict__ slot_of_bin,
                        uint32_t* __restrict__ list) {
    constexpr int G = MODE == AAAC_INT4 ? 128 : 16;
    extern __shared__ uint32_t sm[];                      // kQBins bytes of slot ids
    __shared__ uint32_t buf_key[kStageCap];
    __shared__ uint8_t buf_slot[kStageCap];
    __shared__ uint16_t buf_pos[kStageCap];
    __shared__ uint4 queue_w[8][kQueue];                  // eight weights, their slot bytes and their group's fl32(1 / s)
    __shared__ uint2 queue_s[8][kQueue];
    __shared__ float queue_r[8][kQueue];
    __shared__ uint32_t cnt[kQReq];
    __shared__ unsigned long long base[kQReq];
    __shared__ uint32_t room[kQReq];                      // what a slot's list has left for the block's keys
    __shared__ uint32_t nbuf;
    __shared__ uint32_t okmin[kQReq], okmax[kQReq];       // smallest / largest key of the slots without list space
    __shared__ float rl[128];                             // fl32(1 / s) per E4M3 code, or per mantissa of a BF16 scale
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    chain_next();
    chain_wait();
    const float s_t = ctrl->s_t;
    if (tid < 128) rl[tid] = MODE == AAAC_NVFP4 ? __frcp_rn(__fmul_rn(e4m3_value((uint32_t)tid), s_t)) : bf16_rcp_entry((uint32_t)tid);
    {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(slot_of_bin);
        for (int i = tid; i < kQBins / 4; i += blockDim.x) sm[i] = src[i];
        if (tid == 0) nbuf = 0;
        if (tid < kQReq) { okmin[tid] = 0xFFFFFFFFu; okmax[tid] = 0u; }
    }
    __syncthreads();
    const uint8_t* sm_slot = reinterpret_cast<const uint8_t*>(sm);
    constexpr int LPG = G / 8;                            // lanes per scale group
    const unsigned step = gridDim.x * blockDim.x;
    const unsigned iters = (n_pieces + 2 * step - 1) / (2 * step);     // two pieces per thread and iteration

    // Reserves n places of slot s's list; returns how many of them the list has.  (All of them: its size was counted
    // from the same weights.  The check keeps a layer that is written to meanwhile from spoiling other memory.)
    auto reserve = [&](uint32_t s, uint32_t n, unsigned long long& at) {
        const unsigned long long off = ctrl->slot_off[s];
        const uint32_t size = (uint32_t)(ctrl->slot_off[s + 1] - off), before = atomicAdd(&ctrl->slot_fill[s], n);
        at = off + before;
        return before < size ? min(size - before, n) : 0u;
    };
    auto flush = [&]() {                                  // called by the whole block, after a barrier
        const uint32_t n = min(nbuf, (uint32_t)kStageCap);
        if (tid < kQReq) cnt[tid] = 0;
        __syncthreads();
        for (uint32_t i = tid; i < n; i += blockDim.x) buf_pos[i] = (uint16_t)atomicAdd(&cnt[buf_slot[i]], 1u);
        __syncthreads();
        if (tid < kQReq && cnt[tid]) room[tid] = reserve(tid, cnt[tid], base[tid]);
        __syncthreads();
        for (uint32_t i = tid; i < n; i += blockDim.x)
            if (buf_pos[i] < room[buf_slot[i]]) list[base[buf_slot[i]] + buf_pos[i]] = buf_key[i];
        __syncthreads();
        if (tid == 0) nbuf = 0;
        __syncthreads();
    };

    unsigned next = blockIdx.x * blockDim.x + tid;
    // (the scale travels as its stored bits: nothing waits for the load before the piece is worked on)
    auto fetch = [&](uint4& vv, uint32_t& ss, bool& okk) {
        okk = next < n_pieces;
        if (okk) {
            vv = load_piece<DENSE>(W, next, per_row, ldw);
            if (MODE == AAAC_INT4) ss = __ldg(reinterpret_cast<const uint16_t*>(scales) + next / LPG);
            else ss = __ldg(reinterpret_cast<const uint8_t*>(scales) + next / LPG);
        }
        next += step;
    };
    // The candidates of the first n queued lanes (called by the whole warp).  A slot byte has bit 7 set where
    // the bin is not asked for; the candidates are found by a bit scan of the packed bytes.
    uint32_t q_head = 0, q_fill = 0;                      // the same in every lane of the warp
    auto drain = [&](uint32_t n) {
        __syncwarp();
        if ((uint32_t)lane < n) {
            const uint32_t e = (q_head + lane) % kQueue;
            const uint4 v = queue_w[warp][e];
            const uint2 sb = queue_s[warp][e];
            const float r = queue_r[warp][e];
            const uint64_t bytes = ((uint64_t)sb.y << 32) | sb.x;
            uint64_t todo = ~bytes & 0x8080808080808080ull;
            while (todo) {
                const int j = (__ffsll((long long)todo) - 1) >> 3;
                todo &= todo - 1;
                const uint32_t s = (uint32_t)(bytes >> (8 * j)) & 0xFFu;
                const uint32_t ww = (j >> 1) == 0 ? v.x : (j >> 1) == 1 ? v.y : (j >> 1) == 2 ? v.z : v.w;
                const uint32_t key = float_key(__fmul_rn((j & 1) ? bf16_hi(ww) : bf16_lo(ww), r));
                if (s & kSlotOver) {
                    // no list space for this slot: keep only the extremes of its keys (lanes with the
                    // same slot combine first, so that a heavy bin costs one atomic per warp step)
                    const uint32_t so = s & (kSlotOver - 1u);
                    const unsigned peers = __match_any_sync(__activemask(), so);
                    const uint32_t mn = __reduce_min_sync(peers, key), mx = __reduce_max_sync(peers, key);
                    if (lane == __ffs(peers) - 1) { atomicMin(&okmin[so], mn); atomicMax(&okmax[so], mx); }
                } else {
                    const uint32_t pos = atomicAdd(&nbuf, 1u);
                    if (pos < (uint32_t)kStageCap) {
                        buf_key[pos] = key;
                        buf_slot[pos] = (uint8_t)s;
                    } else {
                        // the stage is full until the block next looks at it: straight to the slot's list
                        unsigned long long at;
                        if (reserve(s, 1u, at)) list[at] = key;
                    }
                }
            }
        }
        __syncwarp();
        q_head += n;
        q_fill -= n;
    };
    // The slots of a lane's eight weights: the AND of their bytes tells whether the lane holds a candidate.
    auto take = [&](const uint4& v, uint32_t ss, bool ok) {
        // fl32(1 / s) for these scale bits
        const float r = MODE == AAAC_INT4 ? bf16_rcp(rl, ss & 0x7FFFu) : rl[ss & 0x7Fu];
        uint32_t bin[8], sl[8];
        qbins(v, r, bin);
#pragma unroll
        for (int j = 0; j < 8; ++j) sl[j] = sm_slot[bin[j]];
        const uint32_t none = 0x80u & (sl[0] & sl[1] & sl[2]) & (sl[3] & sl[4] & sl[5]) & (sl[6] & sl[7]);
        const bool hit = ok && !none;
        const unsigned hits = __ballot_sync(0xFFFFFFFFu, hit);
        if (hit) {
            const uint32_t e = (q_head + q_fill + __popc(hits & ((1u << lane) - 1u))) % kQueue;
            queue_w[warp][e] = v;
            queue_s[warp][e] = make_uint2(__byte_perm(__byte_perm(sl[0], sl[1], 0x0040), __byte_perm(sl[2], sl[3], 0x0040), 0x5410),
                                          __byte_perm(__byte_perm(sl[4], sl[5], 0x0040), __byte_perm(sl[6], sl[7], 0x0040), 0x5410));
            queue_r[warp][e] = r;
        }
        q_fill += __popc(hits);
        if (q_fill >= 32) drain(32);
    };

    // Two pieces per thread are in flight: the loads of iteration k + 1 are issued before iteration k
    // is processed.  The warps of a block meet only every kStageEvery iterations, to empty the
    // stage once it is half full (the vote makes the decision the same for every thread).
    uint4 va{}, vb{};
    uint32_t ra = 0, rb = 0;
    bool oka, okb;
    fetch(va, ra, oka);
    fetch(vb, rb, okb);
    for (unsigned k = 0; k < iters; ++k) {
        uint4 vna{}, vnb{};
        uint32_t rna = 0, rnb = 0;
        bool okna, oknb;
        fetch(vna, rna, okna);
        fetch(vnb, rnb, oknb);
        take(va, ra, oka);
        take(vb, rb, okb);
        if ((k % kStageEvery) == kStageEvery - 1 && __syncthreads_or(nbuf > (uint32_t)kStageCap / 2)) flush();
        va = vna; ra = rna; oka = okna;
        vb = vnb; rb = rnb; okb = oknb;
    }
    drain(q_fill);
    __syncthreads();
    flush();
    if (tid < kQReq && okmin[tid] <= okmax[tid]) {
        atomicMin(&ctrl->slot_kmin[tid], okmin[tid]);
        atomicMax(&ctrl->slot_kmax[tid], okmax[tid]);
    }
}

struct Requests {                     // the order statistics asked for (host-computed from N K alone)
    uint32_t rank[kQReq];             // ascending
    uint8_t id[kQReq];                // which table entry's neighbour it is: 2 entry, 2 entry + 1
    double frac[2 * kM];
};

// One block of 1024 threads: prefix sum, bin + local rank of every request, slots.  All latency: the
// counts are read once, 16 bins per thread; then every warp finds two of the requests side by side, in
// three steps of 32 (or 16) compares at once, and one warp gives the distinct bins their slots by scans
// over the requests in ascending order (4 to 5 us less than where a thread walked its bins for
// every rank in them and 64 threads compared all pairs of requests: 11.3 us).  Counts fit 32 bits: a layer has fewer than
// 2^32 weights.
__device__ __forceinline__ uint32_t warp_inclusive(uint32_t v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

__global__ void __launch_bounds__(1024)
quantile_plan_kernel(Ctrl* ctrl, const uint32_t* __restrict__ hist, uint8_t* __restrict__ slot_of_bin,
                     unsigned long long qcap, const __grid_constant__ Requests rq) {
    __shared__ uint32_t chunk[1024];                        // weights before a thread's bins
    __shared__ uint32_t wtot[32];
    __shared__ uint32_t req_bin[kQReq], req_cnt[kQReq];     // in ascending order of rank
    __shared__ uint32_t cnt_of[kQReq];                      // by the request's id
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int per = kQBins / 1024;
    static_assert(per == 16 && kQReq == 64, "four 16-byte loads per thread, two requests per warp");
    chain_next();
    chain_wait();
    uint32_t s = 0;
    {
        const uint4* src = reinterpret_cast<const uint4*>(hist + tid * per);
#pragma unroll
        for (int i = 0; i < per / 4; ++i) {
            const uint4 v = __ldg(src + i);
            s += v.x + v.y + v.z + v.w;
        }
    }
    if (tid < 2 * kM) ctrl->frac[tid] = rq.frac[tid];
    if (tid == 0) ctrl->done = 0u;                          // blocks of the selection kernel that have finished
    reinterpret_cast<uint4*>(slot_of_bin)[tid] = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
    // exclusive prefix of the 1024 chunk sums: warp scans, then every warp scans the 32 warp totals
    const uint32_t v = warp_inclusive(s, lane);
    if (lane == 31) wtot[warp] = v;
    __syncthreads();
    {
        const uint32_t w = warp_inclusive(wtot[lane], lane);
        const uint32_t before = __shfl_sync(0xFFFFFFFFu, w, (warp + 31) & 31);
        chunk[tid] = v - s + (warp ? before : 0u);
    }
    __syncthreads();
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const int q = half * 32 + warp;
        const uint32_t r = rq.rank[q];
        // the last chunk with at most r weights before it holds rank r (chunk[0] is 0, so there is one)
        const int b = 31 - __clz(__ballot_sync(0xFFFFFFFFu, chunk[32 * lane] <= r));
        const int c = 32 * b + 31 - __clz(__ballot_sync(0xFFFFFFFFu, chunk[32 * b + lane] <= r));
        const uint32_t h = lane < per ? __ldg(hist + c * per + lane) : 0u;
        const uint32_t upto = chunk[c] + warp_inclusive(h, lane);
        const int i = __popc(__ballot_sync(0xFFFFFFFFu, lane < per - 1 && upto <= r));
        if (lane == i) {
            req_bin[q] = c * per + i;
            req_cnt[q] = cnt_of[rq.id[q]] = h;
            ctrl->req_local[rq.id[q]] = r - (upto - h);
        }
    }
    __syncthreads();
    if (warp) return;
    // A slot per distinct bin.  A slot gets list space while the list has room for all of its bin's weights;
    // otherwise it is marked and only the extremes of its keys will be kept.
    const int q0 = 2 * lane, q1 = q0 + 1;
    const uint32_t bin0 = req_bin[q0], bin1 = req_bin[q1];
    const bool lead0 = lane == 0 || req_bin[max(q0 - 1, 0)] != bin0, lead1 = bin1 != bin0;
    const uint32_t c0 = lead0 ? req_cnt[q0] : 0u, c1 = lead1 ? req_cnt[q1] : 0u;
    const uint32_t slots = warp_inclusive((uint32_t)lead0 + (uint32_t)lead1, lane);     // up to and with request q1
    const uint32_t room = warp_inclusive(c0 + c1, lane);
    const uint32_t ns = __shfl_sync(0xFFFFFFFFu, slots, 31), tot = __shfl_sync(0xFFFFFFFFu, room, 31);
    const uint32_t slot1 = slots - 1u, slot0 = slot1 - (uint32_t)lead1;
    ctrl->req_slot[rq.id[q0]] = slot0;
    ctrl->req_slot[rq.id[q1]] = slot1;
    const bool all_fit = tot <= qcap;
    if (all_fit) {
        auto open = [&](uint32_t slot, uint32_t bin, uint32_t off) {
            ctrl->slot_off[slot] = off;
            ctrl->slot_fill[slot] = 0;
            ctrl->slot_over[slot] = 0u;
            slot_of_bin[bin] = (uint8_t)slot;
        };
        if (lead0) open(slot0, bin0, room - c0 - c1);
        if (lead1) open(slot1, bin1, room - c1);
    }
    __syncwarp();                                            // lane 0 reads every lane's req_slot
    if (lane) return;
    if (!all_fit) {
        uint64_t seen = 0, fit = 0;                          // bins take their space in the order of the table entries
        unsigned long long used = 0;
        for (int e = 0; e < kQReq; ++e) {
            const uint32_t slot = ctrl->req_slot[e];
            if (seen >> slot & 1) continue;
            seen |= 1ull << slot;
            if (used + cnt_of[e] > qcap) continue;
            used += cnt_of[e];
            fit |= 1ull << slot;
        }
        unsigned long long off = 0;
        uint32_t slot = 0;
        for (int q = 0; q < kQReq; ++q) {
            if (q && req_bin[q] == req_bin[q - 1]) continue;
            const bool fits = fit >> slot & 1;
            ctrl->slot_off[slot] = off;
            ctrl->slot_fill[slot] = 0;
            ctrl->slot_over[slot] = fits ? 0u : 1u;
            ctrl->slot_kmin[slot] = 0xFFFFFFFFu;
            ctrl->slot_kmax[slot] = 0u;
            slot_of_bin[req_bin[q]] = (uint8_t)(fits ? slot : (slot | kSlotOver));
            if (fits) off += req_cnt[q];
            ++slot;
        }
        ctrl->slot_off[ns] = off;
    } else {
        ctrl->slot_off[ns] = tot;
    }
    ctrl->nslots = ns;
    ctrl->scratch_short = 0u;
}

// one block per slot: radix select of every request that lives in this slot.
//  - The first kKeep * 1024 keys of the list are read once and stay in registers for every sweep;
//    only what is beyond them is streamed from memory, eight loads in flight per thread.
//  - The keys of a slot lie in one narrow bin, so they share their leading bits: one sweep finds
//    the bits on which all keys agree, and only the digits of 11 bits below them need a radix pass: two,
//    mostly, or none where the keys are all equal (8-bit digits took three, and combining equal digits within a
//    warp before counting cost more than the counting).  A thread counts its keys in 32 bits and tests nothing else
//    about them: the longest lists of a layer hold some 60 000 keys and are bound by instructions.
//  - The two neighbours that one table entry interpolates between are consecutive ranks: the
//    second is the first's key again, or the next larger key, which the last pass's counters name
//    unless it differs in a higher digit; then one sweep finds it.
__device__ __forceinline__ void select_slot(Ctrl* ctrl, const uint32_t* __restrict__ list) {
    constexpr int kDigit = 11, kDigits = 1 << kDigit;
    __shared__ uint32_t hist[kDigits];
    __shared__ uint32_t wsum[32];
    __shared__ uint32_t sh_digit, sh_left, sh_in, sh_next;
    __shared__ uint32_t asked[kQReq / 32];                 // the requests that live in this slot
    __shared__ uint32_t req_local[kQReq];
    __shared__ uint32_t sh_or, sh_and, sh_cnt, sh_min;
    const uint32_t slot = blockIdx.x;
    // (read side by side: the launch is all latency for most lists)
    const uint32_t nslots = ctrl->nslots, over = ctrl->slot_over[slot];
    const unsigned long long begin = ctrl->slot_off[slot];
    const uint32_t n = (uint32_t)(ctrl->slot_off[slot + 1] - begin);       // (a layer has fewer than 2^32 weights)
    const uint32_t my_slot = threadIdx.x < kQReq ? ctrl->req_slot[threadIdx.x] : ~0u;
    const uint32_t my_local = threadIdx.x < kQReq ? (uint32_t)ctrl->req_local[threadIdx.x] : 0u;
    if (slot >= nslots) return;
    if (over) {
        // the bin's weights had no room in the list: if they all share one value, that value is every
        // order statistic of the bin; otherwise the scratch was too small for this layer
        const uint32_t kmin = ctrl->slot_kmin[slot], kmax = ctrl->slot_kmax[slot];
        if (my_slot == slot) {
            if (kmin == kmax) ctrl->rank_val[threadIdx.x] = key_float(kmin);
            else { ctrl->rank_val[threadIdx.x] = 0.f; ctrl->scratch_short = 1u; }
        }
        return;
    }
    if (threadIdx.x < kQReq) {
        const unsigned m = __ballot_sync(0xFFFFFFFFu, my_slot == slot);
        if ((threadIdx.x & 31) == 0) asked[threadIdx.x >> 5] = m;
        req_local[threadIdx.x] = my_local;
    }
    if (threadIdx.x == 0) { sh_or = 0u; sh_and = 0xFFFFFFFFu; }
    const uint32_t* keys = list + begin;
    const int lane = threadIdx.x & 31;
    constexpr uint32_t kThreads = 1024;
    constexpr int kKeep = 24, kAhead = 8;
    const uint32_t* mine = keys + threadIdx.x;             // this thread's keys are kThreads apart
    const uint32_t n_mine = threadIdx.x < n ? (n - threadIdx.x - 1) / kThreads + 1 : 0u;
    uint32_t kc[kKeep];
#pragma unroll
    for (int u = 0; u < kKeep; ++u) kc[u] = u < n_mine ? mine[u * kThreads] : 0u;
    // f(key) for every key of this thread's part of the list
    auto for_each_key = [&](auto f) {
#pragma unroll
        for (int u = 0; u < kKeep; ++u) {
            if (u >= n_mine) return;
            f(kc[u]);
        }
        const uint32_t* p = mine + kKeep * kThreads;
        uint32_t left = n_mine - kKeep;
        for (; left >= kAhead; left -= kAhead, p += kAhead * kThreads) {
            uint32_t kk[kAhead];
#pragma unroll
            for (int u = 0; u < kAhead; ++u) kk[u] = p[u * kThreads];
#pragma unroll
            for (int u = 0; u < kAhead; ++u) f(kk[u]);
        }
        for (; left; --left, p += kThreads) f(*p);
    };
    __syncthreads();
    {
        uint32_t o = 0u, a = 0xFFFFFFFFu;
        for_each_key([&](uint32_t k) { o |= k; a &= k; });
        o = __reduce_or_sync(0xFFFFFFFFu, o);
        a = __reduce_and_sync(0xFFFFFFFFu, a);
        if (lane == 0) { atomicOr(&sh_or, o); atomicAnd(&sh_and, a); }
    }
    __syncthreads();
    int top = 31;                                          // highest bit on which keys of the list differ
    uint32_t first_mask = 0u, first_prefix = 0u;           // ... and the bits above it, the same in all
    if (n > 0) {
        const uint32_t diff = sh_or ^ sh_and;
        if (!diff) {                                       // one value (many a bin of scaled BF16 weights)
            if (my_slot == slot) ctrl->rank_val[threadIdx.x] = key_float(sh_and);
            return;
        }
        top = 31 - __clz(diff);
        first_mask = top == 31 ? 0u : ~((2u << top) - 1u);
        first_prefix = sh_and & first_mask;
    }
    bool have_prev = false;                                // rank and key of the request answered last
    uint32_t prev_k = 0;
    uint32_t prev_key = 0u, prev_next = 0u;                // the next larger key, if the counters named it (else 0)
    bool prev_last = false;                                // no further key equal to it comes after that rank
    unsigned long long todo = asked[1];
    for (todo = todo << 32 | asked[0]; todo; todo &= todo - 1) {      // uniform across the block
        const int q = __ffsll((long long)todo) - 1;
        if (have_prev && (req_local[q] == prev_k || req_local[q] == prev_k + 1)) {
            // the same or the next order statistic: it equals the previous key unless every key
            // up to that one is already counted, in which case it is the smallest larger key
            uint32_t key = prev_key;
            if (req_local[q] == prev_k + 1 && prev_last && prev_next) {
                key = prev_next;
            } else if (req_local[q] == prev_k + 1 && prev_last) {
                if (threadIdx.x == 0) { sh_cnt = 0u; sh_min = 0xFFFFFFFFu; }
                __syncthreads();
                uint32_t c = 0u, m = 0xFFFFFFFFu;
                for_each_key([&](uint32_t k) {
                    if (k <= prev_key) ++c;
                    else m = min(m, k);
                });
                c = __reduce_add_sync(0xFFFFFFFFu, c);
                m = __reduce_min_sync(0xFFFFFFFFu, m);
                if (lane == 0) { atomicAdd(&sh_cnt, c); atomicMin(&sh_min, m); }
                __syncthreads();
                if (req_local[q] >= sh_cnt && sh_min != 0xFFFFFFFFu) key = sh_min;
                __syncthreads();
            }
            if (threadIdx.x == 0) ctrl->rank_val[q] = key_float(key);
            // (at most two consecutive ranks belong together; a third is selected anew)
            have_prev = req_local[q] == prev_k;
            continue;
        }
        uint32_t prefix = first_prefix, mask = first_mask;
        uint32_t k_left = req_local[q];                    // rank among the keys with this prefix
        for (int hi = top; hi >= 0;) {
            const int shift = hi >= kDigit ? hi - (kDigit - 1) : 0;
            const uint32_t width = (2u << (hi - shift)) - 1u;
            for (int i = threadIdx.x; i < kDigits; i += blockDim.x) hist[i] = 0;
            if (threadIdx.x == 0) { sh_digit = width; sh_left = 0u; sh_in = 1u; sh_next = 0xFFFFFFFFu; }   // (ranks beyond the list are never requested)
            __syncthreads();
            for_each_key([&](uint32_t k) {
                if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & width], 1u);
            });
            __syncthreads();
            // the digit that holds the rank: thread t owns digits 2 t and 2 t + 1
            const uint32_t c0 = hist[2 * threadIdx.x], c1 = hist[2 * threadIdx.x + 1], tot = c0 + c1;
            uint32_t incl = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane == 31) wsum[threadIdx.x >> 5] = incl;
            __syncthreads();
            uint32_t before = lane < (int)(threadIdx.x >> 5) ? wsum[lane] : 0u;
            before = __reduce_add_sync(0xFFFFFFFFu, before) + incl - tot;
            if (k_left >= before && k_left < before + tot) {
                const bool second = k_left - before >= c0;
                sh_digit = 2 * threadIdx.x + second;
                sh_left = k_left - before - (second ? c0 : 0u);
                sh_in = second ? c1 : c0;
            }
            __syncthreads();
            const uint32_t digit = sh_digit;
            if (shift == 0) {
                // the next larger digit in use names the next larger key
                const uint32_t d0 = 2 * threadIdx.x;
                const uint32_t nx = d0 > digit && c0 ? d0 : d0 + 1 > digit && c1 ? d0 + 1 : 0xFFFFFFFFu;
                const uint32_t wnx = __reduce_min_sync(0xFFFFFFFFu, nx);
                if (lane == 0 && wnx != 0xFFFFFFFFu) atomicMin(&sh_next, wnx);
                __syncthreads();
                prev_last = sh_left + 1 >= sh_in;
                prev_next = sh_next == 0xFFFFFFFFu ? 0u : prefix | sh_next;
            }
            k_left = sh_left;
            prefix |= digit << shift;
            mask |= width << shift;
            hi = shift - 1;
            __syncthreads();                               // (sh_* and hist are written again)
        }
        if (threadIdx.x == 0) ctrl->rank_val[q] = key_float(prefix);
        have_prev = true;
        prev_k = req_local[q];
        prev_key = prefix;
    }
}

// One block per slot; the last block to finish interpolates the table entries: entry e uses requests
// 2e (lower neighbour) and 2e+1 (upper neighbour), in double, rounded to FP32.
__global__ void __launch_bounds__(1024)
quantile_select_kernel(Ctrl* ctrl, const uint32_t* __restrict__ list, uint32_t* dev_status) {
    __shared__ int last;
    chain_next();
    chain_wait();
    select_slot(ctrl, list);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&ctrl->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int e = threadIdx.x;
    if (e == 0) {
        ctrl->done = 0u;
        if (__ldcg(&ctrl->scratch_short) && dev_status) atomicOr(dev_status, AAAC_DEV_SCRATCH);
    }
    if (e >= 2 * kM) return;
    const double lo = (double)__ldcg(&ctrl->rank_val[2 * e]), hi = (double)__ldcg(&ctrl->rank_val[2 * e + 1]);
    const double v = __dadd_rn(lo, __dmul_rn(ctrl->frac[e], __dsub_rn(hi, lo)));
    ctrl->T[e] = (double)(float)v;
}

__global__ void grid_init_kernel(Ctrl* ctrl, int mode, const float* T01_user) {
    const int t = threadIdx.x;
    chain_next();
    chain_wait();
    if (t >= 2 * kM) return;
    if (T01_user) {
        const float T = T01_user[t];
        const uint32_t tmax = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(fabsf(T)));
        const float reach = fmaxf(16.f, 8.f + __uint_as_float(tmax)) * 0.0625f;         // |w~| < 8; a round only brings entries in
        ctrl->T[t] = (double)T;
        if (t == 0) ctrl->reach = __fmul_ru(reach, reach);
        return;
    }
    const double e2m1[kM] = {-6, -4, -3, -2, -1.5, -1, -0.5, 0, 0, 0.5, 1, 1.5, 2, 3, 4, 6};
    auto base = [&](int i) { return mode == AAAC_INT4 ? (double)(i - 8) : e2m1[i]; };
    const int i = t & 15;
    if (t < kM) ctrl->T[t] = base(i);
    else ctrl->T[t] = (i < 15) ? 0.5 * (base(i) + base(i + 1)) : base(15) + 0.5 * (base(15) - base(14));
}

}  // namespace

cudaError_t launch_init(const uint16_t* W, int64_t N, int64_t K, int64_t ldw, int mode, int init,
                        const void* scales, const float* T01_user, uint32_t* dev_status, const Workspace& ws, cudaStream_t st) {
    if (init != AAAC_INIT_QUANTILE) {
        note_launch();
        return launch_chained(grid_init_kernel, 1, 32, 0, st, ws.ctrl, mode, init == AAAC_INIT_USER ? T01_user : nullptr);
    }
    // positions of the 32 quantiles, as the definition states them
    Requests rq;
    uint32_t rank[kQReq];
    const double n1 = (double)(N * K - 1);
    const double d = 1.0 / (2.0 * (kM - 1));
    for (int e = 0; e < 2 * kM; ++e) {
        const int i = e & 15;
        const double q = (e < kM) ? (double)i / (double)(kM - 1) : d + (1.0 - d) * (double)i / (double)(kM - 1);
        const double pos = q * n1;
        double lo = floor(pos), hi = ceil(pos);
        if (lo < 0) lo = 0;
        if (hi > n1) hi = n1;
        if (lo > hi) lo = hi;
        rank[2 * e] = (uint32_t)lo;
        rank[2 * e + 1] = (uint32_t)hi;
        rq.frac[e] = pos - lo;
    }
    for (int q = 0; q < kQReq; ++q) rq.id[q] = (uint8_t)q;
    std::stable_sort(rq.id, rq.id + kQReq, [&](uint8_t a, uint8_t b) { return rank[a] < rank[b]; });
    for (int q = 0; q < kQReq; ++q) rq.rank[q] = rank[rq.id[q]];
    cudaError_t e = launch_chained(quantile_plan_kernel, 1, 1024, 0, st, ws.ctrl, ws.qhist, ws.qslot_of_bin, (unsigned long long)ws.qcap, rq);
    note_launch();
    if (e != cudaSuccess) return e;
    const bool dense = ldw == K;
    auto collect = mode == AAAC_INT4 ? (dense ? quantile_collect_kernel<AAAC_INT4, true> : quantile_collect_kernel<AAAC_INT4, false>)
                                     : (dense ? quantile_collect_kernel<AAAC_NVFP4, true> : quantile_collect_kernel<AAAC_NVFP4, false>);
    static std::atomic<size_t> ready[4][kMaxDevices];
    if ((e = allow_smem(collect, kQBins, ready[2 * (mode == AAAC_NVFP4) + dense])) != cudaSuccess) return e;
    e = launch_chained(collect, sm_count() * 4, 256, kQBins, st, W, (unsigned)(N * (K / 8)), (unsigned)(K / 8), ldw, scales, ws.ctrl,
                       ws.qslot_of_bin, ws.qlist);
    note_launch();
    if (e != cudaSuccess) return e;
    note_launch();
    return launch_chained(quantile_select_kernel, kQReq, 1024, 0, st, ws.ctrl, ws.qlist, dev_status);
}

}  // namespace aaac
