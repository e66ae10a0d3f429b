// Per-policy reductions over a grid of plain policies, budgets by migration overheads: dispatch decision (Algorithms 2-3,
// wait-then-race), TTFT, which decode stream applies (migration trigger, Eq. 4), tokens per endpoint.
//
// The distinct budgets of the policies are the grid's COLUMNS (ascending), the distinct overheads its ROWS.  What a
// request comes to under a policy, but for the hand-off, depends on the column alone, and along the columns thresholds
// are ordered: Algorithm 3's l_th does not increase, Algorithm 2's l* does not decrease, its w_tail does not increase.
// So a request falls into at most three runs of columns that dispatch it alike:
//   Algorithm 3:  columns [0, k) have l_th > l  -> device only;     [k, K) race at once (wait 0);
//   Algorithm 2:  columns [0, k1) have l* < l   -> wait w_tail;     [k1, k2) have l* = l -> wait their own w*;
//                 [k2, K) have l* > l           -> wait 0.
// k, k1, k2 depend on the prompt length alone, and the requests of a group are stored by prompt length: a chunk of
// requests splits into a few SEGMENTS of consecutive requests that share them.  A block sweeps a segment once per run
// with a lane per request, sums up what the requests come to in registers and shared-memory histograms, and enters the
// run's totals ONCE into a table of differences along the columns (row q is carried to the columns from q on: a run of the
// columns [a, b) is entered into row a and taken back in row b).  k_spread adds the rows up and writes every policy's
// sums and histograms.
// Under Algorithm 2 the first columns (budgets below the tail ratio) may wait longer than the others: for the few
// requests that the common w_tail does not cover (at most a share alpha of them) the block keeps a list, and each of
// those columns gets the list's totals under its own wait in place of the common one.
//
// The rows differ in the hand-off alone: a race won by the endpoint that may hand over migrates in the rows whose
// overhead is below the request's saving.  Every sweep adds what migration changes to each row whose overhead it passes
// (three additions a row); the hand-off stall is counted at the level of the last such row, and the levels are summed
// up when the run is entered.
//
// Bound: integer issue.  Against one sweep per 128 policies of one overhead, with what differs between neighbouring
// policies entered into their histograms one by one, a request is visited once per run instead of once per run and
// overhead: 16 M requests in six groups under 128 budgets by 8 overheads took 2,300 us (and 450 more pair by pair), now
// 349 and k_spread 18; a million in one group under 256 by 4 took 220 us, now 35 and 15.
#include <algorithm>
#include <cstddef>
#include <type_traits>

#include "tile.cuh"

namespace disco {

namespace {

constexpr int kThreads = 256;
constexpr int kListCap = 8192;           // requests a block lists for the columns with longer waits
constexpr int kListStep = 4096;          // ... and looks after the list's room every so many requests
constexpr int kMaxSeg = 2 * kGridCols + 2;
constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr uint32_t kNoPolicy = 0xFFFFFFFFu;
static_assert(kNBins % 32 == 0 && kNBins / 32 < 32, "a bit for each group of bins");

// Blocks to a multiprocessor by the rows a kernel is built for: as many as its registers allow with few spills (64 registers:
// 136 bytes in k_grid<1, true>, 16 in <2, false>; 80: 8 in <2, true>, 20 in <4, true>; the others none).
__host__ __device__ constexpr int blocks_for(int rows, bool wide) { return rows == 1 || (rows == 2 && !wide) ? 4 : rows <= 4 ? 3 : 2; }
// The rows of the kernel that takes a slab of T.
constexpr int rows_for(int T) { return T <= 1 ? 1 : T <= 2 ? 2 : T <= 4 ? 4 : 8; }

// Sums of a run: what every row gets, and per row what migration changes.
enum Base { B_TD = 0, B_PS, B_PD, B_DO, B_RACE, B_DW, B_TAU, B_TT, kBase };
enum Lev { V_A = 0, V_B, V_C, V_N, V_TAU, kLev };      // tokens handed over, prefill of the target, delayed, count, TBTs in tau's bin
__host__ __device__ constexpr int sum_fields(int T) { return kBase + T * kLev; }

struct Seg { uint16_t pa, pb, k1, k2; };               // requests [pa, pb) of the chunk

struct Smem {                                          // fixed part; the TBT histograms [T][kNBins] follow, and one more for
                                                       // the device-only run where windows are counted
    uint32_t sum[kBase + kGridRows * kLev];            // totals of the run in work
    uint32_t only_sum[4];                              // ... of the device-only run: requests, tokens, prompt tokens, TBTs in tau's bin
    uint32_t tt[3], only_tt[3];                        // ... and the sums of TTFTs, in parts of 20 bits
    uint32_t ttft[kNBins], only_ttft[kNBins];
    uint32_t used[2][3];                               // groups of bins with counts: TTFT, stall, device only; by turns
    uint32_t n_seg, n_runs, n_list, flagged, ticket;
    int32_t key[kGridCols];                            // the columns' length thresholds
    uint32_t w_star[kGridCols], w_tail[kGridCols];
    Seg seg[kMaxSeg];
    uint16_t list[kListCap];
};

template <int NT>
struct Acc {                                           // a lane's share of a run
    uint32_t td, ps, pd, tau, race, dw;
    unsigned long long tt;
    uint32_t bins, stalls;                             // groups of 32 bins with counts: of the TTFTs, of the hand-off stalls
    uint32_t a[NT], b[NT], cn[NT], tx[NT];             // cn: delayed tokens | requests << 22 (at most 255 requests a lane)
};

struct Only { uint32_t cnt, n, l, tau, bins; unsigned long long tt; };   // ... of a device-only run

struct Ctx {                                           // a (chunk, slab)
    uint32_t start, len;
    uint32_t kappa, c0;
    float delta_c;
    int cand, g;
    int K, T;
    bool may_migrate, mixed;
    float th_lo;                                       // mixed: smallest overhead
    int E0, x_from;
    uint32_t even;
    const ClassConst* cc;
    const uint2* hand;
    size_t win_at;                                     // bytes from the windows of slot 0
};

struct Args {
    TraceDev tr;
    TimelineRec rec;
    const GroupConst* gcs;
    size_t rec_stride;
    const ClassConst* classes;
    const Prep* prep;
    uint32_t P;
    const Slab* slabs;
    uint32_t n_slabs;
    const uint32_t* tab;
    const Chunk* chunks;
    uint32_t n_chunks;
    GridTables gt;
    LeftLists left;
    uint32_t k0;
    uint32_t* ticket;
    unsigned long long* work;
    bool beside;
};

__device__ __forceinline__ void hist_add(uint32_t* h, int bin) {
    if (DBG_OK(bin, kNBins, DBG_K_GRID, DBG_BIN)) atomicAdd(&h[bin], 1u);
}

// Adds (or, sub, takes) the rows of window counts of the lanes' requests that are in the mask: a lane sums up a bin over
// the requests, with eight loads in flight, and adds once.
__device__ __forceinline__ void add_rows(const uint16_t* __restrict__ win, int W, int lo, uint32_t mask, uint32_t kk, bool sub,
                                         uint32_t* hist) {
    if (mask == 0u) return;
    const int lane = threadIdx.x & 31;
    if (W <= 16) {
        // short rows: several requests' at a time, which mostly lie side by side
        const int per = 32 / W, mine = lane / W, b = lane - mine * W;
        const bool in = mine < per && DBG_OK(lo + b, kNBins, DBG_K_GRID, DBG_BIN);
        uint32_t sum = 0;
#pragma unroll 4
        for (int r0 = 0; r0 < 32; r0 += per) {
            const int r = r0 + mine;
            const uint32_t k = __shfl_sync(FULL, kk, r & 31);
            if (in && r < 32 && ((mask >> r) & 1u)) sum += win[(size_t)k * W + b];
        }
        if (sum) atomicAdd(&hist[lo + b], sub ? 0u - sum : sum);
        return;
    }
    for (int b0 = 0; b0 < W; b0 += 32) {
        const int b = b0 + lane;
        const bool in = b < W && DBG_OK(lo + b, kNBins, DBG_K_GRID, DBG_BIN);
        uint32_t sum = 0;
#pragma unroll 1
        for (int r0 = 0; r0 < 32; r0 += 8) {
            if (((mask >> r0) & 255u) == 0u) continue;
            uint32_t v[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const uint32_t k = __shfl_sync(FULL, kk, r0 + r);
                v[r] = (in && ((mask >> (r0 + r)) & 1u)) ? win[(size_t)k * W + b] : 0u;
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) sum += v[r];
        }
        if (sum) atomicAdd(&hist[lo + b], sub ? 0u - sum : sum);
    }
}

// The windows of the lanes' requests whose streams' intervals are not all tau: the base stream (device or server) goes to
// every row of the grid but those that migrate, [0, t), which get the stream after the hand-off.
__device__ __forceinline__ void add_windows(const Args& a, const Ctx& c, uint32_t* tbt, bool valid, uint32_t kk, bool device, int t,
                                            uint32_t orig) {
    const ClassConst& cc = *c.cc;
    const auto win = [&](int s) { return reinterpret_cast<const uint16_t*>(reinterpret_cast<const char*>(a.rec.win[s]) + c.win_at); };
    uint32_t* all = tbt + (c.T - 1) * kNBins;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        if ((c.even >> s) & 1u) continue;
        const bool mine = valid && (int)device == s;
        const int W = cc.W[s], lo = cc.lo[c.g][s];
        add_rows(win(s), W, lo, __ballot_sync(FULL, mine && t < c.T), kk, false, all);
        for (int r = 1; r < c.T; ++r)
            add_rows(win(s), W, lo, __ballot_sync(FULL, mine && t == r), kk, true, tbt + (r - 1) * kNBins);
    }
    if (c.even & 4u) return;
    const int from = c.x_from >= 0 ? c.x_from : 2;
    for (int r = 1; r <= c.T; ++r)
        add_rows(win(from), cc.W[from], cc.lo[c.g][from], __ballot_sync(FULL, valid && t == r), kk, false, tbt + (r - 1) * kNBins);
    if (c.x_from >= 0 && valid && t > 0) {
        const int bin = first_bin(a.gcs[c.g], c.x_from, a.k0, orig);
        if (DBG_OK(bin, kNBins, DBG_K_GRID, DBG_BIN)) atomicSub(&tbt[(t - 1) * kNBins + bin], 1u);
    }
}

// One sweep over the requests [pa, pb) of the chunk, or (list) of the block's list: what they come to when the device
// starts after the wait w, added up in `s` and in the shared histograms.  push: requests with S > w go on the list.
// ONLY: the segment is Algorithm 3's; `race` says whether some columns race (w = 0), `only` whether some run the device
// alone, which is added up in `o` and histograms of its own.
template <int NT, bool WIDE, bool ONLY>
__device__ __forceinline__ void sweep(const Args& a, const Ctx& c, const float (&th)[NT], Smem& sm, uint32_t* tbt, uint32_t pa,
                                      uint32_t pb, uint32_t w, bool list, bool push, bool race, bool only, Acc<NT>& s, Only& o) {
    const int lane = threadIdx.x & 31;
    // The kernel of eight rows has too few warps a multiprocessor to hide the loads' latency: there they run an iteration
    // ahead (16 M requests under 128 budgets by 8 overheads, with k_spread, 369 us instead of 435; the others have the
    // warps, and no registers left: 3 % slower).
    constexpr bool kAhead = NT == 8 && !WIDE;
    uint32_t pos;
    uint4 q, q_ahead;
    uint2 hand, hand_ahead;
    uint32_t ahead;
    auto fetch = [&](uint32_t i0, uint32_t& at, uint4& to, uint2& to_hand) {
        const uint32_t i = min(i0 + lane, pb - 1);
        at = list ? (uint32_t)sm.list[i] : i;
        to = a.tr.req[c.start + at];
        to_hand = c.may_migrate ? c.hand[c.start + at] : make_uint2(0u, 0u);
    };
    const uint32_t first = pa + (threadIdx.x & ~31u);
    if (kAhead && first < pb) fetch(first, ahead, q_ahead, hand_ahead);
    for (uint32_t i0 = first; i0 < pb; i0 += kThreads) {              // a warp's lanes iterate together
        if (kAhead) {
            pos = ahead; q = q_ahead; hand = hand_ahead;
            if (i0 + kThreads < pb) fetch(i0 + kThreads, ahead, q_ahead, hand_ahead);
        } else {
            fetch(i0, pos, q, hand);
        }
        const uint32_t kk = c.start + pos;
        bool valid = i0 + lane < pb && DBG_OK(kk, a.tr.n, DBG_K_GRID, DBG_REQUEST);
        const uint32_t S = q.x, l = q.y & 0xFFFFu, n = q.y >> 16, m = hand.x & 0xFFFFu, dly = hand.x >> 16;
        const uint32_t Td = c.kappa * l + c.c0;
        // Eq. 4's projected saving, on the true remainder or on what is left of the expected length; a request may only
        // hand over if its buffer filled (m != 0)
        float saving = m ? c.delta_c * (float)(c.E0 ? max(c.E0 - (int)m, 0) : (int)(n - m)) : -1.0f;
        if (c.mixed) valid = valid && !(saving > c.th_lo && !(saving > th[0]));       // left to the pair kernel
        if (ONLY) {
            if (only) {
                const int bin = bin_of_ticks(Td);
                const uint32_t live = __ballot_sync(FULL, valid);
                // requests of one prompt length share the device's TTFT: mostly the whole warp counts in one bin
                if (__shfl_sync(FULL, l, 0) == __shfl_sync(FULL, l, 31)) {
                    if (lane == 0 && live && DBG_OK(bin, kNBins, DBG_K_GRID, DBG_BIN)) atomicAdd(&sm.only_ttft[bin], (uint32_t)__popc(live));
                } else if (valid) hist_add(sm.only_ttft, bin);
                if (!WIDE && valid) o.bins |= 1u << (bin >> 5);
                if (valid) { o.cnt += 1u; o.n += n; o.l += l; o.tt += Td; o.tau += (!WIDE || (c.even & 2u)) ? n - 1u : 0u; }
                if (WIDE && !(c.even & 2u)) add_rows(reinterpret_cast<const uint16_t*>(reinterpret_cast<const char*>(a.rec.win[1]) + c.win_at), c.cc->W[1], c.cc->lo[c.g][1], live, kk, false, tbt + NT * kNBins);
            }
            if (!race) continue;
        }
        const bool started = S > w, dev_wins = S > w + Td;            // the device starts after the wait; a tie goes to the server
        const uint32_t tt = min(S, w + Td);
        const bool pace = ((c.even >> (dev_wins ? 1 : 0)) & 1u) != 0; // the base stream's intervals are all tau
        if (valid) {
            s.td += dev_wins ? n : 0u; s.ps += l; s.pd += started ? l : 0u;
            s.race += started ? 1u : 0u; s.dw += dev_wins ? 1u : 0u;
            s.tt += tt;
            s.tau += (!WIDE || pace) ? n - 1u : 0u;
            const int bin = bin_of_ticks(tt);
            hist_add(sm.ttft, bin);
            if (!WIDE) s.bins |= 1u << (bin >> 5);
        }
        if (!ONLY && push) {
            const bool mine = valid && S > w;
            const uint32_t all = __ballot_sync(FULL, mine);
            if (all) {
                uint32_t at = 0;
                if (lane == 0) at = atomicAdd(&sm.n_list, (uint32_t)__popc(all));
                at = __shfl_sync(FULL, at, 0) + __popc(all & ((1u << lane) - 1u));
                if (mine && DBG_OK(at, kListCap, DBG_K_GRID, DBG_SLOT)) sm.list[at] = (uint16_t)pos;
            }
        }
        if (!(valid && started && (dev_wins ? 2 : 1) == c.cand)) saving = -1.0f;      // not won by the endpoint that may hand over
        const uint32_t handed = n - m, refill = l + m, cn = dly | 1u << 22;
        const uint32_t tx = WIDE ? ((c.even & 4u) ? n - 2u : 0u) - (pace ? n - 1u : 0u) : 0u;
        int t = 0;                                                    // rows that migrate: [0, t)
#pragma unroll
        for (int r = 0; r < NT; ++r)
            if (saving > th[r]) {
                s.a[r] += handed; s.b[r] += refill; s.cn[r] += cn; ++t;
                if (WIDE) s.tx[r] += tx;
            }
        if (t > 0) {
            const int bin = bin_of_ticks(hand.y);
            hist_add(tbt + (t - 1) * kNBins, bin);
            if (!WIDE) s.stalls |= 1u << (bin >> 5);
        }
        if (WIDE) add_windows(a, c, tbt, valid, kk, dev_wins, t, q.z);
    }
}

// Adds the lanes' 64-bit shares (below 2^40 each) to a total kept in parts of 20 bits: three warp sums instead of a tree of
// shuffles, and 32-bit additions in shared memory, which has no 64-bit ones of its own.
__device__ __forceinline__ void add_wide(uint32_t (&to)[3], unsigned long long v) {
    const uint32_t a = __reduce_add_sync(FULL, (uint32_t)v & 0xFFFFFu), b = __reduce_add_sync(FULL, (uint32_t)(v >> 20) & 0xFFFFFu);
    const int lane = threadIdx.x & 31;
    const unsigned long long t = (unsigned long long)a + ((unsigned long long)b << 20);
    if (lane < 3) {
        const uint32_t part = lane == 0 ? (uint32_t)t & 0xFFFFFu : lane == 1 ? (uint32_t)(t >> 20) & 0xFFFFFu : (uint32_t)(t >> 40);
        if (part) atomicAdd(&to[lane], part);
    }
}
__device__ __forceinline__ unsigned long long take_wide(uint32_t (&from)[3]) {
    const unsigned long long v = from[0] + ((unsigned long long)from[1] << 20) + ((unsigned long long)from[2] << 40);
    from[0] = from[1] = from[2] = 0;
    return v;
}

// The lanes' shares of a run go to the block's totals (32-bit: at most 65,280 requests of at most 12,288 tokens).  Lane f
// of a warp adds field f.
template <int NT, bool WIDE>
__device__ __forceinline__ void share_out(Smem& sm, const Acc<NT>& s, int turn) {
    const int lane = threadIdx.x & 31;
    if (!WIDE) {
        const uint32_t bins = __reduce_or_sync(FULL, s.bins), stalls = __reduce_or_sync(FULL, s.stalls);
        if (lane == 0 && bins) atomicOr(&sm.used[turn][0], bins);
        if (lane == 0 && stalls) atomicOr(&sm.used[turn][1], stalls);
    }
    uint32_t lo = 0, hi = 0;
    auto put = [&](int f, uint32_t v) {
        v = __reduce_add_sync(FULL, v);
        if (f < 32) { if (lane == f) lo = v; } else if (lane == f - 32) hi = v;
    };
    put(B_TD, s.td); put(B_PS, s.ps); put(B_PD, s.pd); put(B_RACE, s.race); put(B_DW, s.dw); put(B_TAU, s.tau);
#pragma unroll
    for (int r = 0; r < NT; ++r) {
        const int f = kBase + r * kLev;
        put(f + V_A, s.a[r]); put(f + V_B, s.b[r]); put(f + V_C, s.cn[r] & 0x3FFFFFu); put(f + V_N, s.cn[r] >> 22);
        if (WIDE) put(f + V_TAU, s.tx[r]);
    }
    if (lo) atomicAdd(&sm.sum[lane], lo);
    if (NT * kLev + kBase > 32 && hi) atomicAdd(&sm.sum[32 + lane], hi);
    add_wide(sm.tt, s.tt);
}
__device__ __forceinline__ void share_only(Smem& sm, const Only& o, int turn) {
    const uint32_t bins = __reduce_or_sync(FULL, o.bins);
    if ((threadIdx.x & 31) == 0 && bins) atomicOr(&sm.used[turn][2], bins);
    const uint32_t c = __reduce_add_sync(FULL, o.cnt), n = __reduce_add_sync(FULL, o.n), l = __reduce_add_sync(FULL, o.l),
                   tau = __reduce_add_sync(FULL, o.tau);
    add_wide(sm.only_tt, o.tt);
    if ((threadIdx.x & 31) == 0 && c) {
        atomicAdd(&sm.only_sum[0], c); atomicAdd(&sm.only_sum[1], n); atomicAdd(&sm.only_sum[2], l); atomicAdd(&sm.only_sum[3], tau);
    }
}

// A slab's difference tables: row q is carried to the columns from q on.
template <bool WIDE>
struct Tables {
    using word = typename std::conditional<WIDE, unsigned long long, unsigned int>::type;   // windows hold more than 2^32 TBTs
    uint32_t* ttft;                      // [K][kNBins]
    word* tbt;                           // [T][K][kNBins]
    unsigned long long* sums;            // [G][K][fields]
    int K, T, G;
    __device__ Tables(const GridTables& gt, const Slab& sl, int G_)
        : ttft(gt.ttft + sl.ttft), tbt((word*)gt.tbt + sl.tbt), sums(gt.sums + sl.sums), K(sl.K), T(sl.T), G(G_) {}
    __device__ uint32_t* ttft_row(int q) const { return ttft + (size_t)q * kNBins; }
    __device__ word* tbt_row(int q, int r) const { return tbt + ((size_t)r * K + q) * kNBins; }
    __device__ unsigned long long* sum_row(int g, int q) const { return sums + ((size_t)g * K + q) * sum_fields(T); }
};

// Calls f(bin) for every bin of the groups of 32 in the mask, a warp a group (ALL: for every bin; windows may lie anywhere).
template <bool ALL, class F>
__device__ __forceinline__ void each_bin(uint32_t groups, F f) {
    if (ALL) {
        for (int b = threadIdx.x; b < kNBins; b += kThreads) f(b);
        return;
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int k = 0; groups; groups &= groups - 1u, ++k)
        if (k % (kThreads / 32) == w) f((__ffs(groups) - 1) * 32 + lane);
}

// Enters what the block has totalled for a run of the columns [q0, q1), or takes it from them (neg), and clears it.  All
// threads call; barriers before and after.  Only groups of 32 bins that the run has counts in are looked at (a run over all
// bins of nine histograms took longer than the sweep of a few hundred requests).
template <int NT, bool WIDE>
__device__ __forceinline__ void enter(Smem& sm, uint32_t* tbt, const Tables<WIDE>& tb, int g, int q0, int q1, bool neg, int turn) {
    using word = typename Tables<WIDE>::word;
    const bool back = q1 < tb.K;
    each_bin<WIDE>(sm.used[turn][0], [&](int b) {
        const uint32_t x = sm.ttft[b];
        if (x) {
            sm.ttft[b] = 0;
            const uint32_t y = neg ? 0u - x : x;
            atomicAdd(&tb.ttft_row(q0)[b], y);
            if (back) atomicAdd(&tb.ttft_row(q1)[b], 0u - y);
        }
    });
    each_bin<WIDE>(sm.used[turn][1], [&](int b) {
        int32_t y[NT], level = 0;                                      // counts at a level go to every row below it
#pragma unroll
        for (int r = 0; r < NT; ++r) y[r] = (int32_t)tbt[r * kNBins + b];      // (rows beyond the slab's have none)
#pragma unroll
        for (int r = NT - 1; r >= 0; --r) {
            if (y[r]) { tbt[r * kNBins + b] = 0; level += y[r]; }
            if (level) {
                const word z = (word)(long long)(neg ? -level : level);
                atomicAdd(&tb.tbt_row(q0, r)[b], z);
                if (back) atomicAdd(&tb.tbt_row(q1, r)[b], (word)0 - z);
            }
        }
    });
    const int F = sum_fields(tb.T);
    for (int f = threadIdx.x; f < F; f += kThreads) {
        unsigned long long x = (f >= kBase && (f - kBase) % kLev == V_TAU) ? (unsigned long long)(long long)(int32_t)sm.sum[f] : sm.sum[f];
        sm.sum[f] = 0;
        if (f == B_TT) x = take_wide(sm.tt);
        if (!x) continue;
        if (neg) x = 0ull - x;
        atomicAdd(&tb.sum_row(g, q0)[f], x);
        if (back) atomicAdd(&tb.sum_row(g, q1)[f], 0ull - x);
    }
    if (threadIdx.x < 3) sm.used[turn ^ 1][threadIdx.x] = 0;          // (of the run before; all have read them)
}

// The same for a device-only run of the columns below q1.
template <bool WIDE>
__device__ __forceinline__ void enter_only(Smem& sm, uint32_t* only_tbt, const Tables<WIDE>& tb, int g, int q1, int turn) {
    using word = typename Tables<WIDE>::word;
    const bool back = q1 < tb.K;
    each_bin<WIDE>(sm.used[turn][2], [&](int b) {
        const uint32_t x = sm.only_ttft[b];
        if (x) {
            sm.only_ttft[b] = 0;
            atomicAdd(&tb.ttft_row(0)[b], x);
            if (back) atomicAdd(&tb.ttft_row(q1)[b], 0u - x);
        }
        if (WIDE) {
            const word y = only_tbt[b];
            if (y) {
                only_tbt[b] = 0;
                for (int r = 0; r < tb.T; ++r) {
                    atomicAdd(&tb.tbt_row(0, r)[b], y);
                    if (back) atomicAdd(&tb.tbt_row(q1, r)[b], (word)0 - y);
                }
            }
        }
    });
    if (threadIdx.x < 3) sm.used[turn ^ 1][threadIdx.x] = 0;
    if (threadIdx.x < 5) {
        const int k = threadIdx.x;
        const unsigned long long x = k < 4 ? (unsigned long long)sm.only_sum[k] : take_wide(sm.only_tt);
        if (k < 4) sm.only_sum[k] = 0;
        const int f = k == 0 ? B_DO : k == 1 ? B_TD : k == 2 ? B_PD : k == 3 ? B_TAU : B_TT;
        if (x) {
            atomicAdd(&tb.sum_row(g, 0)[f], x);
            if (back) atomicAdd(&tb.sum_row(g, q1)[f], 0ull - x);
        }
    }
}

// A chunk whose runs have few requests each, request by request: a thread enters what its request comes to in every run by
// itself.  A run swept by the whole block costs its barriers and a walk over all bins (a microsecond or more), which pays
// only with enough requests to share it.  Bound: the chain of atomics per request, and, with many of them, the L2 slices
// that the hottest sums live in (lanes that add up first were tried: shorter there, but longer where the lanes' columns
// differ).  A step of 1,000 requests under 256 budgets 465 -> 114 us, of 10,000 requests under 256 policies with
// migration 785 -> 185 us.
//
// Taken below so many requests to a run: where every block has at most one item the step waits for the slowest item, and
// the runs' latency decides (64; nothing changes beyond); with more items than blocks the atomics' rate does, and at 24
// requests to a run 300,000 requests under 128 policies with migration already lose (286 us against 230, 202 at 16).
constexpr uint32_t kDirectAlone = 64, kDirectMany = 16;

template <int NT>
__device__ __noinline__ void enter_requests(const Args& a, const Ctx& c, const float (&th)[NT], const Smem& sm,
                                            const Tables<false>& tb, bool waits, uint32_t wt_min, int n_low) {
    const int K = c.K;
    for (uint32_t i = threadIdx.x; i < c.len; i += kThreads) {
        const uint32_t kk = c.start + i;
        const uint4 q = a.tr.req[kk];
        const uint2 hand = c.may_migrate ? c.hand[kk] : make_uint2(0u, 0u);
        const uint32_t S = q.x, l = q.y & 0xFFFFu, n = q.y >> 16, m = hand.x & 0xFFFFu, dly = hand.x >> 16;
        const uint32_t Td = c.kappa * l + c.c0;
        const float saving = m ? c.delta_c * (float)(c.E0 ? max(c.E0 - (int)m, 0) : (int)(n - m)) : -1.0f;
        if (c.mixed && saving > c.th_lo && !(saving > th[0])) continue;               // left to the pair kernel
        // adds (or takes) a count to a histogram of the columns [q0, q1), a value to a sum
        auto count = [&](uint32_t* at, int q0, int q1) {
            atomicAdd(at + (size_t)q0 * kNBins, 1u);
            if (q1 < K) atomicAdd(at + (size_t)q1 * kNBins, ~0u);
        };
        const size_t F = sum_fields(c.T);
        auto add = [&](int f, unsigned long long v, int q0, int q1) {
            unsigned long long* at = tb.sum_row(c.g, 0) + f;
            atomicAdd(at + q0 * F, v);
            if (q1 < K) atomicAdd(at + q1 * F, 0ull - v);
        };
        // what the request comes to under the columns [q0, q1), which start the device after w
        auto enter_run = [&](uint32_t w, int q0, int q1) {
            const bool started = S > w, dev_wins = S > w + Td;
            const uint32_t tt = min(S, w + Td);
            const int bin = bin_of_ticks(tt);
            if (DBG_OK(bin, kNBins, DBG_K_GRID, DBG_BIN)) count(tb.ttft + bin, q0, q1);
            if (dev_wins) { add(B_TD, n, q0, q1); add(B_DW, 1ull, q0, q1); }
            add(B_PS, l, q0, q1);
            if (started) { add(B_PD, l, q0, q1); add(B_RACE, 1ull, q0, q1); }
            add(B_TAU, n - 1u, q0, q1); add(B_TT, tt, q0, q1);
            if (!started || (dev_wins ? 2 : 1) != c.cand) return;
            const int stall = bin_of_ticks(hand.y);
#pragma unroll
            for (int r = 0; r < NT; ++r) {
                if (!(saving > th[r])) break;                                          // (overheads ascend)
                const int f = kBase + r * kLev;
                add(f + V_A, n - m, q0, q1); add(f + V_B, l + m, q0, q1); add(f + V_N, 1ull, q0, q1);
                if (dly) add(f + V_C, dly, q0, q1);
                if (DBG_OK(stall, kNBins, DBG_K_GRID, DBG_BIN)) count(tb.tbt + (size_t)r * K * kNBins + stall, q0, q1);
            }
        };
        // the columns on either side of the request's length
        int k1 = 0, k2;
        for (int hi = K; k1 < hi;) { const int mid = (k1 + hi) >> 1; if (waits ? sm.key[mid] < (int)l : sm.key[mid] > (int)l) k1 = mid + 1; else hi = mid; }
        k2 = k1;
        if (waits) {
            while (k2 < K && sm.key[k2] == (int)l) { enter_run(sm.w_star[k2], k2, k2 + 1); ++k2; }
            const int low = S > wt_min ? min(n_low, k1) : 0;
            for (int p = 0; p < low; ++p) enter_run(sm.w_tail[p], p, p + 1);
            if (low < k1) enter_run(wt_min, low, k1);
        } else if (k1 > 0) {                                                           // the device alone
            const int bin = bin_of_ticks(Td);
            if (DBG_OK(bin, kNBins, DBG_K_GRID, DBG_BIN)) count(tb.ttft + bin, 0, k1);
            add(B_DO, 1ull, 0, k1); add(B_TD, n, 0, k1); add(B_PD, l, 0, k1); add(B_TAU, n - 1u, 0, k1); add(B_TT, Td, 0, k1);
        }
        if (k2 < K) enter_run(0u, k2, K);
    }
}

template <int NT, bool WIDE>
__global__ void __launch_bounds__(kThreads, blocks_for(NT, WIDE))
k_grid(const __grid_constant__ Args a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
    uint32_t* tbt = (uint32_t*)(smem_raw + sizeof(Smem));
    // Beside the slope search of Eq. 1-2 (k_prep_beta), which no plain policy needs: what this kernel reads was complete before that
    // one let it start.  It then waits at its end, for the kernels behind.  (Under 48 such searches, 79 us on 48
    // multiprocessors, 300,000 requests by 16 budgets take 27.)
    for (int i = threadIdx.x; i < (int)(offsetof(Smem, key) / 4); i += kThreads) ((uint32_t*)&sm)[i] = 0;
    for (int i = threadIdx.x; i < (NT + (WIDE ? 1 : 0)) * kNBins; i += kThreads) tbt[i] = 0;
    if (!a.beside) grid_dependency_wait();

    int turn = 0;                                                     // which of the two sets of used bins is in use
    const uint32_t direct = a.n_chunks * a.n_slabs <= gridDim.x ? kDirectAlone : kDirectMany;
    // A block starts with a (chunk, slab) item of its own and then draws the next ones from a counter (zero at launch): items
    // differ in cost.  (Drawn ahead, when the one in front begins, they are no longer dealt to who is free: 16 M requests by
    // 128 and 8 policies 348 -> 385 us.  Beside another kernel not all blocks are there at once: all items are drawn.)
    const uint32_t n_items = a.n_chunks * a.n_slabs, dealt = a.beside ? 0u : gridDim.x;
    uint32_t item = blockIdx.x;
    __syncthreads();
    if (a.beside) {
        if (threadIdx.x == 0) sm.ticket = atomicAdd(a.ticket, 1u);
        __syncthreads();
        item = sm.ticket;
    }
    for (; item < n_items; item = sm.ticket) {
        const uint32_t slab_id = item % a.n_slabs;
        const Slab& sl = a.slabs[slab_id];
        const Chunk ch = a.chunks[item / a.n_slabs];
        const int g = ch.g;
        if (!DBG_OK(g, a.tr.n_groups, DBG_K_GRID, DBG_GROUP) ||
            (ch.len && !DBG_OK((unsigned long long)ch.start + ch.len - 1, a.tr.n, DBG_K_GRID, DBG_REQUEST)))
            break;
        const GroupConst& gc = a.gcs[g];
        const Tables<WIDE> tb(a.gt, sl, a.tr.n_groups);
        Ctx c;
        c.start = ch.start; c.len = ch.len; c.kappa = (uint32_t)gc.kappa; c.c0 = (uint32_t)gc.c0;
        c.delta_c = gc.delta_c; c.cand = gc.candidate; c.g = g; c.K = sl.K; c.T = sl.T;
        c.may_migrate = sl.mig && gc.candidate != 0;
        c.mixed = sl.mixed && c.may_migrate;
        c.cc = a.classes + sl.cls;
        c.hand = reinterpret_cast<const uint2*>(reinterpret_cast<const char*>(a.rec.hand) + sl.slot * a.rec_stride);
        c.win_at = sl.win_slot * a.rec_stride;
        c.E0 = (int)sl.expected_len; c.even = c.cc->even[g];
        c.x_from = x_stream(*c.cc, gc);
        float th[NT];                                                  // rows beyond the slab's never migrate
#pragma unroll
        for (int r = 0; r < NT; ++r) th[r] = (c.may_migrate && r < c.T) ? sl.theta[sl.mixed ? 1 : r] : __int_as_float(0x7F800000);
        c.th_lo = sl.theta[0];
        bool waits = false;
        {
            const Prep& pr = a.prep[(size_t)g * a.P + a.tab[sl.cols]];
            waits = pr.device_constrained != 0;
        }
        for (int p = threadIdx.x; p < c.K; p += kThreads) {
            if (!DBG_OK(a.tab[sl.cols + p], a.P, DBG_K_GRID, DBG_POLICY)) continue;
            const Prep& pr = a.prep[(size_t)g * a.P + a.tab[sl.cols + p]];
            sm.key[p] = waits ? pr.l_star : pr.l_th;
            sm.w_star[p] = (uint32_t)pr.w_star; sm.w_tail[p] = (uint32_t)pr.w_tail;
        }
        if (c.mixed) {
            // ---- requests whose saving lies between the policies' overheads: to the pair kernel's list
            const uint32_t first = a.tr.grp_off[g];
            uint32_t mine = 0;
            for (uint32_t i0 = threadIdx.x & ~31u; i0 < ch.len; i0 += kThreads) {
                const uint32_t i = min(i0 + (threadIdx.x & 31), ch.len - 1), kk = ch.start + i;
                const uint4 q = a.tr.req[kk];
                const uint32_t m = c.hand[kk].x & 0xFFFFu, n = q.y >> 16;
                const float saving = m ? c.delta_c * (float)(c.E0 ? max(c.E0 - (int)m, 0) : (int)(n - m)) : -1.0f;
                const bool out = i0 + (threadIdx.x & 31) < ch.len && saving > c.th_lo && !(saving > th[0]);
                const uint32_t all = __ballot_sync(FULL, out);
                if (!all) continue;
                uint32_t at = 0;
                if ((threadIdx.x & 31) == 0) at = atomicAdd(&a.left.count[slab_id * a.tr.n_groups + g], (uint32_t)__popc(all));
                at = first + __shfl_sync(FULL, at, 0) + __popc(all & ((1u << (threadIdx.x & 31)) - 1u));
                if (out && DBG_OK(at, a.tr.n, DBG_K_GRID, DBG_REQUEST)) a.left.list[(size_t)slab_id * a.tr.n + at] = kk;
                mine += (uint32_t)__popc(all);
            }
            if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&sm.flagged, mine);
        }
        __syncthreads();

        // ---- the segments: stretches of prompt lengths between two thresholds and (Algorithm 2) the thresholds
        //      themselves; a thread per candidate looks up where its lengths lie in the chunk
        const int K = c.K;
        for (int q = threadIdx.x; q < (waits ? 2 * K + 1 : K + 1); q += kThreads) {
            auto cl = [](int x) { return min(max(x, 0), kMaxPrompt + 1); };
            int la, lb, k1, k2;
            bool any = true;
            if (waits) {                                             // thresholds ascend
                const int p = q >> 1;
                k1 = k2 = p;
                if (q == 2 * K) { la = cl(sm.key[K - 1] + 1); lb = kMaxPrompt + 1; }
                else if (q & 1) {
                    la = cl(sm.key[p]); lb = cl(sm.key[p] + 1); any = p == 0 || sm.key[p] != sm.key[p - 1];
                    if (any && la < lb) while (k2 < K && sm.key[k2] == sm.key[p]) ++k2;
                }
                else { la = p ? cl(sm.key[p - 1] + 1) : 0; lb = cl(sm.key[p]); }
            } else {                                                 // thresholds descend
                la = q ? cl(sm.key[K - q]) : 0;
                lb = q < K ? cl(sm.key[K - 1 - q]) : kMaxPrompt + 1;
                k1 = k2 = K - q;
            }
            if (any && la < lb) {
                // first request of the group with a prompt of at least L tokens: where the shorter ones end
                const uint32_t* ends = a.tr.len_end + (size_t)g * (kMaxPrompt + 1);
                const uint32_t at_a = la ? ends[la - 1] : a.tr.grp_off[g], at_b = ends[lb - 1];
                const uint32_t lo = ch.start, hi = ch.start + ch.len;
                const uint32_t pa = min(max(at_a, lo), hi) - lo, pb = min(max(at_b, lo), hi) - lo;
                if (pa < pb) {
                    const uint32_t at = atomicAdd(&sm.n_seg, 1u);
                    atomicAdd(&sm.n_runs, waits ? (uint32_t)(k2 - k1) + (k1 > 0) + (k2 < K) : 1u);
                    if (DBG_OK(at, kMaxSeg, DBG_K_GRID, DBG_SLOT))
                        sm.seg[at] = Seg{(uint16_t)pa, (uint16_t)pb, (uint16_t)k1, (uint16_t)k2};
                }
            }
        }
        const uint32_t wt_min = waits ? sm.w_tail[K - 1] : 0u;
        int n_low = 0;                                                // columns that wait longer than the others: the first ones
        for (int p0 = 0; waits && p0 < K; p0 += kThreads) {
            const int p = p0 + (int)threadIdx.x;
            n_low += __syncthreads_count(p < K && sm.w_tail[p] > wt_min);
        }
        __syncthreads();
        const int n_seg = (int)min(sm.n_seg, (uint32_t)kMaxSeg);
        uint32_t passes = 0;

        // one run: sweep and enter; `list` and `push` as in sweep
        auto run = [&](uint32_t pa, uint32_t pb, uint32_t w, bool list, bool push, int q0, int q1, bool neg) {
            Acc<NT> s = {};
            Only none = {};
            sweep<NT, WIDE, false>(a, c, th, sm, tbt, pa, pb, w, list, push, true, false, s, none);
            share_out<NT, WIDE>(sm, s, turn);
            __syncthreads();
            enter<NT, WIDE>(sm, tbt, tb, g, q0, q1, neg, turn);
            __syncthreads();
            ++passes; turn ^= 1;
        };
        bool by_request = false;
        if constexpr (!WIDE) {
            by_request = c.len < (sm.n_runs + (n_low ? (uint32_t)n_low + 1u : 0u)) * direct;
            if (by_request) {
                const Ctx its = c;                                    // (copies: what is handed over by address lives in memory)
                const Tables<false> tables = tb;
                float rows[NT];
#pragma unroll
                for (int r = 0; r < NT; ++r) rows[r] = th[r];
                enter_requests<NT>(a, its, rows, sm, tables, waits, wt_min, n_low);
                passes = 1;
            }
        }
        if (by_request) {
        } else if (!waits) {
            for (int si = 0; si < n_seg; ++si) {
                const Seg sg = sm.seg[si];
                const bool race = (int)sg.k2 < K, only = sg.k1 > 0;
                Acc<NT> s = {};
                Only o = {};
                sweep<NT, WIDE, true>(a, c, th, sm, tbt, sg.pa, sg.pb, 0u, false, false, race, only, s, o);
                if (race) share_out<NT, WIDE>(sm, s, turn);
                if (only) share_only(sm, o, turn);
                __syncthreads();
                if (race) enter<NT, WIDE>(sm, tbt, tb, g, sg.k2, K, false, turn);
                if (only) enter_only<WIDE>(sm, tbt + NT * kNBins, tb, g, sg.k1, turn);
                __syncthreads();
                ++passes; turn ^= 1;
            }
        } else {
            // segment by segment, run by run: [k2, K) waits 0, each column of [k1, k2) its own w*, [0, k1) w_tail -- and,
            // when the list is full or the chunk is done, the list for the columns that wait longer
            uint32_t pa = 0;                                          // (of the segment in work: where the sweep goes on)
            int si = 0, ri = 0;
            for (;;) {
                uint32_t from = 0, to = 0, w = 0;
                int q0 = 0, q1 = 0;
                bool push = false;
                const bool done = si >= n_seg;
                if (!done) {
                    const Seg sg = sm.seg[si];
                    const int n_pts = (int)sg.k2 - (int)sg.k1;
                    if (ri == 0) pa = sg.pa;
                    if (ri == 0 && (int)sg.k2 >= K) { ++ri; continue; }
                    if (ri > n_pts && sg.k1 == 0) { ri = 0; ++si; continue; }
                    from = pa; to = sg.pb;
                    if (ri == 0) { q0 = sg.k2; q1 = K; ++ri; }
                    else if (ri <= n_pts) { q0 = (int)sg.k1 + ri - 1; q1 = q0 + 1; w = sm.w_star[q0]; ++ri; }
                    else {
                        w = wt_min; q1 = sg.k1; push = n_low > 0;
                        if (push && to - from > (uint32_t)kListStep) { to = from + kListStep; pa = to; }
                        else { ri = 0; ++si; }
                    }
                    run(from, to, w, false, push, q0, q1, false);
                } else if (sm.n_list == 0) break;
                if (done || (push && sm.n_list > (uint32_t)(kListCap - kListStep))) {
                    const uint32_t k = sm.n_list;                     // (barriers inside run: all threads agree)
                    __syncthreads();
                    if (threadIdx.x == 0) sm.n_list = 0;
                    for (int p = -1; p < n_low; ++p)                  // the common wait's totals go, each column's own come
                        run(0u, k, p < 0 ? wt_min : sm.w_tail[p], true, false, max(p, 0), p < 0 ? n_low : p + 1, p < 0);
                }
            }
        }
        if (threadIdx.x == 0 && a.work) {
            const unsigned long long settled = ch.len - sm.flagged;
            atomicAdd(&a.work[0], settled * (unsigned long long)sl.policies);      // pairs settled run by run
            atomicAdd(&a.work[2], settled);                            // requests settled, per slab
            atomicAdd(&a.work[3], (unsigned long long)passes);         // sweeps over segments
        }
        if (n_items <= dealt) break;
        __syncthreads();
        if (threadIdx.x == 0) {
            sm.n_seg = 0; sm.n_runs = 0; sm.n_list = 0; sm.flagged = 0;
            sm.ticket = dealt + atomicAdd(a.ticket, 1u);
        }
        __syncthreads();
    }
    if (a.beside) grid_dependency_wait();
}

// Adds up the difference rows: what a policy gets is the sum of the rows up to its column.  A block takes 32 histogram
// bins (or sums) of one row of the grid, a lane each, and all columns, a few consecutive ones a warp: the warps add up
// their own rows, the totals meet in shared memory, and every warp writes its columns' policies.  Bound: L2 and the
// stores (the tables are read once, every policy's histograms written once).  (256 x 4 policies: 15 us; one thread a bin,
// walking the columns, 202.  The 64 registers that 1,024 threads leave spill 204 bytes, 68 with windows.)
constexpr int kSpreadWarps = 32;
constexpr int kSpreadPer = kGridCols / kSpreadWarps;                   // columns a warp may have
static_assert(kNBins % 32 == 0, "a block's bins");

template <class W, class F, class E>
__device__ __forceinline__ void spread_columns(unsigned long long* s_part, int K, F at /* (q) */, E emit /* (column, value) */) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int per = (K + kSpreadWarps - 1) / kSpreadWarps, q0 = min(K, w * per), q1 = min(K, q0 + per);
    W x[kSpreadPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kSpreadPer; ++k) x[k] = q0 + k < q1 ? (W)at(q0 + k) : (W)0;
#pragma unroll
    for (int k = 0; k < kSpreadPer; ++k) { sum += x[k]; x[k] = sum; }
    s_part[w * 33 + lane] = sum;
    __syncthreads();
    // the warps' totals in front of each: a warp scans one bin's 32 totals
    {
        unsigned long long v = s_part[lane * 33 + w];
        const unsigned long long own = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned long long up = __shfl_up_sync(FULL, v, off);
            if (lane >= off) v += up;
        }
        s_part[lane * 33 + w] = v - own;
    }
    __syncthreads();
    const W before = (W)s_part[w * 33 + lane];
#pragma unroll
    for (int k = 0; k < kSpreadPer; ++k) if (q0 + k < q1) emit(q0 + k, (W)(before + x[k]));
}

template <bool WIDE>
__global__ void __launch_bounds__(kSpreadWarps * 32)
k_spread(TraceDev tr, const GroupConst* __restrict__ gcs, const Slab* __restrict__ slabs,
         const uint32_t* __restrict__ tab, GridTables gt, unsigned long long* __restrict__ acc,
         unsigned long long* __restrict__ hist_ttft, unsigned long long* __restrict__ hist_tbt) {
    __shared__ unsigned long long s_part[kSpreadWarps * 33];
    grid_dependency_wait();
    const Slab& sl = slabs[blockIdx.y];
    const int K = sl.K, T = sl.T, bin_tau = sl.bin_tau, lane = threadIdx.x & 31;
    const Tables<WIDE> tb(gt, sl, tr.n_groups);
    using word = typename Tables<WIDE>::word;
    const uint32_t* cells = tab + sl.cells;
    constexpr int kParts = kNBins / 32;
    int part = blockIdx.x;
    if (part < T * kParts) {                                           // TTFT: the same for every row
        const int r = part / kParts, b = (part - r * kParts) * 32 + lane;
        spread_columns<uint32_t>(s_part, K, [&](int q) { return tb.ttft_row(q)[b]; }, [&](int c, uint32_t x) {
            const uint32_t p = cells[c * T + r];
            if (p != kNoPolicy) hist_ttft[(size_t)p * kNBins + b] = x;
        });
        return;
    }
    part -= T * kParts;
    if (part < T * kParts) {                                           // TBT
        const int r = part / kParts, b = (part - r * kParts) * 32 + lane;
        // (in 64 bits: tau's bin holds all regular TBTs; a 32-bit row is a difference of at most 2^31 requests)
        using big = unsigned long long;
        spread_columns<big>(s_part, K, [&](int q) {
            const word y = tb.tbt_row(q, r)[b];
            big x = WIDE ? (big)y : (big)(long long)(int32_t)y;
            if (b == bin_tau)                                          // the regular TBTs of streams that keep the pace
                for (int g = 0; g < tr.n_groups; ++g) {
                    const unsigned long long* row = tb.sum_row(g, q);
                    x += row[B_TAU] + (WIDE ? row[kBase + r * kLev + V_TAU] : 0ull - row[kBase + r * kLev + V_N]);
                }
            return x;
        }, [&](int c, big x) {
            const uint32_t p = cells[c * T + r];
            if (p != kNoPolicy) hist_tbt[(size_t)p * kNBins + b] = x;
        });
        return;
    }
    part -= T * kParts;
    const int k = part * 32 + lane;                                    // sums
    if (part * 32 >= tr.n_groups * T * kNAcc) return;
    const bool mine = k < tr.n_groups * T * kNAcc;
    const int s = mine ? k % kNAcc : 0, r = mine ? (k / kNAcc) % T : 0, g = mine ? k / (kNAcc * T) : 0;
    const int cand = gcs[g].candidate;
    const int fb = s == A_DEVICE_ONLY ? B_DO : s == A_RACE ? B_RACE : s == A_DEVICE_WON ? B_DW : s == A_TOK_DEVICE ? B_TD
                 : s == A_PRE_SERVER ? B_PS : s == A_PRE_DEVICE ? B_PD : s == A_TTFT_SUM ? B_TT : -1;
    int fl = -1;
    bool minus = false;
    if (s == A_TOK_DEVICE) { fl = V_A; minus = cand == 2; }            // the server's tokens go to the device, or the device's to the server
    else if (s == A_PRE_SERVER && cand == 2) fl = V_B;
    else if (s == A_PRE_DEVICE && cand == 1) fl = V_B;
    else if (s == A_DELAYED) fl = V_C;
    else if (s == A_MIGR) fl = V_N;
    const int f2 = fl < 0 ? -1 : kBase + r * kLev + fl;
    spread_columns<unsigned long long>(s_part, K, [&](int q) {
        const unsigned long long* row = tb.sum_row(g, q);
        unsigned long long y = fb >= 0 ? row[fb] : 0ull;
        if (f2 >= 0) y += minus ? 0ull - row[f2] : row[f2];
        return y;
    }, [&](int c, unsigned long long x) {
        const uint32_t p = mine ? cells[c * T + r] : kNoPolicy;
        if (p == kNoPolicy) return;
        acc[((size_t)p * tr.n_groups + g) * kNAcc + s] = x;
    });
}

size_t grid_smem(int NT, bool wide) { return sizeof(Smem) + (size_t)(NT + (wide ? 1 : 0)) * kNBins * 4; }

template <int NT, bool WIDE>
cudaError_t launch_one(const Args& a, int sms, cudaStream_t st) {
    const size_t smem = grid_smem(NT, WIDE);
    cudaError_t e = allow_smem((const void*)k_grid<NT, WIDE>, smem);
    if (e) return e;
    const uint64_t items = (uint64_t)a.n_chunks * a.n_slabs;
    const uint32_t blocks = (uint32_t)std::min<uint64_t>(items, (uint64_t)sms * blocks_for(NT, WIDE));
    return launch_after(k_grid<NT, WIDE>, dim3(blocks), kThreads, smem, st, a);
}

}  // namespace

DBG_TRANSLATION_UNIT()

uint64_t grid_ttft_words(int K) { return (uint64_t)K * kNBins; }
uint64_t grid_tbt_words(int K, int T) { return (uint64_t)K * T * kNBins; }
uint64_t grid_sum_words(int K, int T, int G) { return (uint64_t)G * K * sum_fields(T); }
uint32_t grid_blocks_per_sm(int T) { return (uint32_t)blocks_for(rows_for(T), false); }
int grid_rows(int T) { return rows_for(T); }

cudaError_t launch_grid(const TraceDev& tr, const GroupConst* gc, const ClassConst* classes, const Prep* prep, uint32_t P,
                        const Slab* slabs, uint32_t n_slabs, int T, bool wide, const uint32_t* tab,
                        const Chunk* chunks, uint32_t n_chunks, TimelineRec rec, size_t rec_stride, GridTables gt, LeftLists left,
                        uint32_t k0, uint32_t* ticket, uint64_t* work, bool beside, int sms, cudaStream_t st) {
    if (n_chunks == 0 || n_slabs == 0) return cudaSuccess;
    if ((uint64_t)n_chunks * n_slabs > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
    const Args a = {tr, rec, gc, rec_stride, classes, prep, P, slabs, n_slabs, tab, chunks, n_chunks, gt, left, k0, ticket,
                    (unsigned long long*)work, beside};
    switch (rows_for(T)) {
        case 1: return wide ? launch_one<1, true>(a, sms, st) : launch_one<1, false>(a, sms, st);
        case 2: return wide ? launch_one<2, true>(a, sms, st) : launch_one<2, false>(a, sms, st);
        case 4: return wide ? launch_one<4, true>(a, sms, st) : launch_one<4, false>(a, sms, st);
        default: return wide ? launch_one<8, true>(a, sms, st) : launch_one<8, false>(a, sms, st);
    }
}

cudaError_t launch_spread(const TraceDev& tr, const GroupConst* gc, const Slab* slabs, uint32_t n_slabs, int T,
                          bool wide, const uint32_t* tab, GridTables gt, uint64_t* acc, uint64_t* hist_ttft,
                          uint64_t* hist_tbt, cudaStream_t st) {
    if (n_slabs == 0) return cudaSuccess;
    const dim3 grid((uint32_t)(2 * T * (kNBins / 32) + (tr.n_groups * T * kNAcc + 31) / 32), n_slabs);
    auto* kernel = wide ? k_spread<true> : k_spread<false>;
    return launch_after(kernel, grid, kSpreadWarps * 32, 0, st, tr, gc, slabs, tab, gt, (unsigned long long*)acc,
                        (unsigned long long*)hist_ttft, (unsigned long long*)hist_tbt);
}

}  // namespace disco
