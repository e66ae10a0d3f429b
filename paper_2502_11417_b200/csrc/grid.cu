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
// requests splits into a few SEGMENTS of consecutive requests that share them.  A block sweeps a segment with a lane per
// request, sums up what the requests come to in registers and shared-memory histograms, and enters a run's totals ONCE into a
// table of differences along the columns (row q is carried to the columns from q on: a run of the columns [a, b) is entered
// into row a and taken back in row b).  k_spread adds the rows up and writes every policy's sums and histograms.
// The last run of a segment and the first are swept together: where the device runs alone, or where the common w_tail covers a
// request (S <= w_tail: the server answers alone), the first run adds little to what is read.  The requests that w_tail does not
// cover (at most a share alpha of them) go on a list of the block's, swept again for the first run, and once for each of the
// columns that wait longer (budgets below the tail ratio).  With windows Algorithm 2's segments are swept run by run.
// Small traces leave a run few requests: there a lane takes a request with all its runs (see below).
//
// The rows differ in the hand-off alone: a race won by the endpoint that may hand over migrates in the rows whose
// overhead is below the request's saving.  Every sweep adds what migration changes to each row whose overhead it passes
// (three additions a row), or, with eight rows, to the last of them; the hand-off stall is counted at the level of the last such
// row, and the levels are summed up when the run is entered.
//
// Bound: a run's barriers and its latency, then integer issue (half of the slots).  16 M requests in six groups under 128 budgets by 8
// overheads: 347 us with a sweep for each run and every row's sums in registers (122 of them, two blocks to a multiprocessor), 240 now
// (80, three); 5 M under 40 by 8 113 -> 85; a million in one group under 256 by 4 32 -> 28.  (Kernels that also held the way of small traces had to spill: 283 and 99.)
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <type_traits>

#include "tile.cuh"

namespace disco {

namespace {

constexpr int kThreads = 256;
constexpr int kListCap = 4096;           // requests a block lists whose TTFT the common wait does not cover
// ... of a segment that are entered by warps, a wait each: a handful is not worth a run for every column that waits longer (600,000 requests
// in six groups under 32 by 2 34 us, now 30).  Not with more rows: the additions to their histograms are as many as the rows, and the call
// costs registers.
__host__ __device__ constexpr int list_few(int NT) { return NT > 2 ? 0 : 256 / (1 + NT); }
// Requests that may be swept at once where any may be listed: whole rounds of the block, so that what a lane takes of a chunk in several
// sweeps is no more than in one.
__device__ __forceinline__ uint32_t list_room(uint32_t listed) { return ((uint32_t)kListCap - listed) / kThreads * kThreads; }
constexpr int kMaxSeg = 2 * kGridCols + 2;
constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr uint32_t kNoPolicy = 0xFFFFFFFFu;
static_assert(kNBins % 32 == 0 && kNBins / 32 < 32, "a bit for each group of bins");

// Blocks to a multiprocessor by the rows a kernel is built for: as many as its registers allow with few spills (with windows up to
// 44 bytes, without up to 20).
enum GridMode { M_RACES = 0, M_WAITS, M_JOINED };
__host__ __device__ constexpr int blocks_for(int rows, bool wide, int mode) { return mode == M_JOINED ? (rows <= 2 ? 4 : 3) : rows <= (wide ? 1 : 2) ? 4 : rows <= 4 || !wide ? 3 : 2; }
// The rows of the kernel that takes a slab of T.
constexpr int rows_for(int T) { return T <= 1 ? 1 : T <= 2 ? 2 : T <= 4 ? 4 : 8; }

// Sums of a run: what every row gets, and per row what migration changes.
enum Base { B_TD = 0, B_PS, B_PD, B_DO, B_RACE, B_DW, B_TAU, B_TT, kBase };
enum Lev { V_A = 0, V_B, V_C, V_N, V_TAU, kLev };      // tokens handed over, prefill of the target, delayed, count, TBTs in tau's bin
__host__ __device__ constexpr int sum_fields(int T) { return kBase + T * kLev; }

struct Seg { uint16_t pa, pb, k1, k2; };               // requests [pa, pb) of the chunk

// Whether a lane's shares of what migration changes lie in shared memory, level by level (see Levels).
__host__ __device__ constexpr bool has_levels(int NT, bool wide) { return NT >= 8 && !wide; }

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

// Whether the bins of the TTFTs that a run has counts in are remembered: not where windows may lie anywhere, nor in the kernel of eight
// rows, which has no registers left for it.
__host__ __device__ constexpr bool knows_bins(int NT, bool wide) { return !wide && !has_levels(NT, wide); }

struct __align__(16) Smem {                            // fixed part; the TBT histograms [T][kNBins] follow, and one more for
                                                       // the run beside where windows are counted, or the warps' levels
    uint32_t sum[2][kBase + kGridRows * kLev];         // totals of the run in work; by turns
    uint32_t side_sum[4];                              // ... of the run beside it: requests, tokens, prompt tokens, TBTs in tau's bin
    uint32_t tt[3], side_tt[3];                        // ... and the sums of TTFTs, in parts of 20 bits
    uint32_t ttft[kNBins], side_ttft[kNBins];
    uint32_t used[2][3];                               // groups of bins with counts: TTFT, stall, TTFT of the run beside; by turns
    uint32_t n_seg, n_list, flagged, ticket;
    int32_t key[kGridCols];                            // the columns' length thresholds
    uint32_t w_star[kGridCols], w_tail[kGridCols];
    Seg seg[kMaxSeg];
    uint16_t list[kListCap];
    Ctx ctx;                                           // of the item, and its overheads, for what is called and not inlined
    float rows[kGridRows];
    uint32_t slab;
};

static_assert(sizeof(Smem) % 16 == 0 && kNBins % 2 == 0, "the levels are read in words of eight bytes");

template <int NT, bool WIDE>
struct Acc {                                           // a lane's share of a run
    static constexpr int kRows = has_levels(NT, WIDE) ? 0 : NT;
    uint32_t td, ps, pd, tau, race, dw;
    unsigned long long tt;
    uint32_t bins, stalls;                             // groups of 32 bins with counts: of the TTFTs, of the hand-off stalls
    uint32_t levels;                                   // a bit a level with requests
    uint32_t a[kRows + 1], b[kRows + 1], cn[kRows + 1], tx[kRows + 1];   // cn: delayed tokens | requests << 22 (at most 255 requests a lane)
};

struct Side { uint32_t cnt, n, l, tau, bins; unsigned long long tt; };   // ... of the run beside it

// With eight rows a request does not go to every row that it migrates in but to the last of them, its level, and the levels are
// added up when the run is entered.  (With four, registers do: a million requests under 256 by 4 28 us, by levels 36.)  A lane's shares lie in shared memory, a column of the warp's for each lane, which nobody else
// touches: handed-over tokens and prefill side by side, then delayed tokens | requests << 22.
template <int NT>
struct Levels {
    uint2* ab;                                         // [NT][32]
    uint32_t* cn;                                      // [NT][32]
    static constexpr int kWords = NT * 96;             // of a warp
    __device__ explicit Levels(uint32_t* at) : ab(reinterpret_cast<uint2*>(at)), cn(at + NT * 64) {}
};

// Words behind the fixed part: the TBT histograms and what follows them.
__host__ __device__ constexpr int tbt_words(int NT, bool wide) { return (NT + (wide ? 1 : 0)) * kNBins + (has_levels(NT, wide) ? kThreads / 32 * NT * 96 : 0); }

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
    bool beside, early;
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
// starts after the wait w, added up in `s` and in the shared histograms.
// SIDE: a segment's requests under its last columns, which wait 0 (`race`: there are such columns), and beside them under its first
// ones (`side`), added up in `o` and histograms of its own: Algorithm 3's, where the device runs alone (S_DEVICE), or Algorithm 2's
// (S_SERVER), which wait w: there the server alone answers the requests with S <= w, and the others go on the list.
// push: requests with S > w go on the list (without a run beside).
enum SideKind { S_NONE = 0, S_DEVICE, S_SERVER };
template <int NT, bool WIDE, int SIDE>
__device__ __forceinline__ void sweep(const Args& a, const Ctx& c, const float (&th)[NT], Smem& sm, uint32_t* tbt, const Levels<NT>& lv,
                                      uint32_t pa, uint32_t pb, uint32_t w, bool list, bool push, bool race, bool side, Acc<NT, WIDE>& s, Side& o) {
    constexpr bool waits = SIDE == S_SERVER;
    const int lane = threadIdx.x & 31;
    // The kernel of eight rows has too few warps a multiprocessor to hide the loads' latency: there they run an iteration ahead.
    constexpr bool kAhead = NT == 8 && !WIDE;
    constexpr bool kLevels = has_levels(NT, WIDE);
    uint32_t pos;
    uint4 q, q_ahead;
    uint2 hand, hand_ahead;
    uint32_t ahead;
    auto fetch = [&](uint32_t i0, uint32_t& at, uint4& to, uint2& to_hand) {
        const uint32_t i = min(i0 + lane, pb - 1);
        at = !SIDE && list ? (uint32_t)sm.list[i] : i;
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
        if (NT == 1 && c.mixed) valid = valid && !(saving > c.th_lo && !(saving > th[0]));       // left to the pair kernel
        if (SIDE && side) {
            constexpr int stream = 1;                                 // (with windows a run beside is the device's)
            const bool mine = valid && !(waits && S > w);
            const uint32_t tt = waits ? S : Td;
            const uint32_t live = __ballot_sync(FULL, mine);
            const int bin = bin_of_ticks(tt);
            // requests of one prompt length share the device's TTFT: mostly the whole warp counts in one bin
            if (!waits && __shfl_sync(FULL, l, 0) == __shfl_sync(FULL, l, 31)) {
                if (lane == 0 && live && DBG_OK(bin, kNBins, DBG_K_GRID, DBG_BIN)) atomicAdd(&sm.side_ttft[bin], (uint32_t)__popc(live));
            } else if (mine) hist_add(sm.side_ttft, bin);
            if (knows_bins(NT, WIDE) && mine) o.bins |= 1u << (bin >> 5);
            if (mine) { o.cnt += 1u; o.n += n; o.l += l; o.tt += tt; o.tau += (!WIDE || ((c.even >> stream) & 1u)) ? n - 1u : 0u; }
            if (WIDE && !((c.even >> stream) & 1u))
                add_rows(reinterpret_cast<const uint16_t*>(reinterpret_cast<const char*>(a.rec.win[stream]) + c.win_at), c.cc->W[stream], c.cc->lo[c.g][stream], live, kk, false, tbt + NT * kNBins);
        }
        if (waits || (WIDE && push)) {
            const bool longer = valid && S > w;
            const uint32_t all = __ballot_sync(FULL, longer);
            if (all) {
                uint32_t at = 0;
                if (lane == 0) at = atomicAdd(&sm.n_list, (uint32_t)__popc(all));
                at = __shfl_sync(FULL, at, 0) + __popc(all & ((1u << lane) - 1u));
                if (longer && DBG_OK(at, kListCap, DBG_K_GRID, DBG_SLOT)) sm.list[at] = (uint16_t)pos;
            }
        }
        if (SIDE && !race) continue;
        const uint32_t wait = SIDE ? 0u : w;
        const bool started = S > wait, dev_wins = S > wait + Td;      // the device starts after the wait; a tie goes to the server
        const uint32_t tt = min(S, wait + Td);
        const bool pace = ((c.even >> (dev_wins ? 1 : 0)) & 1u) != 0; // the base stream's intervals are all tau
        if (valid) {
            s.td += dev_wins ? n : 0u; s.ps += l; s.pd += started ? l : 0u;
            s.race += started ? 1u : 0u; s.dw += dev_wins ? 1u : 0u;
            s.tt += tt;
            s.tau += (!WIDE || pace) ? n - 1u : 0u;
            const int bin = bin_of_ticks(tt);
            hist_add(sm.ttft, bin);
            if (knows_bins(NT, WIDE)) s.bins |= 1u << (bin >> 5);
        }
        if (!(valid && started && (dev_wins ? 2 : 1) == c.cand)) saving = -1.0f;      // not won by the endpoint that may hand over
        const uint32_t handed = n - m, refill = l + m, cn = dly | 1u << 22;
        const uint32_t tx = WIDE ? ((c.even & 4u) ? n - 2u : 0u) - (pace ? n - 1u : 0u) : 0u;
        int t = 0;                                                    // rows that migrate: [0, t)
        if constexpr (kLevels) {
            if (saving > th[0]) {
                static_assert(NT == 8, "a search in steps of four, two and one");
                const bool p4 = saving > th[4], p2 = saving > (p4 ? th[6] : th[2]);
                t = (p4 ? 5 : 1) + (p2 ? 2 : 0) + (saving > (p4 ? (p2 ? th[7] : th[5]) : (p2 ? th[3] : th[1])) ? 1 : 0);
                const int at = (t - 1) * 32 + lane;
                uint2 v = lv.ab[at];
                v.x += handed; v.y += refill;
                lv.ab[at] = v;
                lv.cn[at] += cn;
                s.levels |= 1u << (t - 1);
                const int bin = bin_of_ticks(hand.y);
                hist_add(tbt + (t - 1) * kNBins, bin);
                s.stalls |= 1u << (bin >> 5);
            }
        } else {
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
__device__ __forceinline__ void share_out(Smem& sm, const Acc<NT, WIDE>& s, const Levels<NT>& lv, int turn) {
    const int lane = threadIdx.x & 31;
    if (!WIDE) {
        const uint32_t bins = knows_bins(NT, WIDE) ? __reduce_or_sync(FULL, s.bins) : 0u, stalls = __reduce_or_sync(FULL, s.stalls);
        if (lane == 0 && bins) atomicOr(&sm.used[turn][0], bins);
        if (lane == 0 && stalls) atomicOr(&sm.used[turn][1], stalls);
    }
    uint32_t lo = 0, hi = 0;
    auto put = [&](int f, uint32_t v) {
        v = __reduce_add_sync(FULL, v);
        if (f < 32) { if (lane == f) lo = v; } else if (lane == f - 32) hi = v;
    };
    put(B_TD, s.td); put(B_PS, s.ps); put(B_PD, s.pd); put(B_RACE, s.race); put(B_DW, s.dw); put(B_TAU, s.tau);
    if constexpr (has_levels(NT, WIDE)) {
#pragma unroll 1
        for (uint32_t left = __reduce_or_sync(FULL, s.levels); left; left &= left - 1u) {
            const int r = __ffs(left) - 1, at = r * 32 + lane;
            const uint2 v = lv.ab[at];
            const uint32_t cn = lv.cn[at];
            lv.ab[at] = make_uint2(0u, 0u); lv.cn[at] = 0u;
            const uint32_t x = __reduce_add_sync(FULL, v.x), y = __reduce_add_sync(FULL, v.y), dly = __reduce_add_sync(FULL, cn & 0x3FFFFFu), num = __reduce_add_sync(FULL, cn >> 22);
            const uint32_t z = lane == V_A ? x : lane == V_B ? y : lane == V_C ? dly : num;
            if (lane < V_TAU && z) atomicAdd(&sm.sum[turn][kBase + r * kLev + lane], z);
        }
    } else {
#pragma unroll
        for (int r = 0; r < NT; ++r) {
            const int f = kBase + r * kLev;
            put(f + V_A, s.a[r]); put(f + V_B, s.b[r]); put(f + V_C, s.cn[r] & 0x3FFFFFu); put(f + V_N, s.cn[r] >> 22);
            if (WIDE) put(f + V_TAU, s.tx[r]);
        }
    }
    if (lo) atomicAdd(&sm.sum[turn][lane], lo);
    if (!has_levels(NT, WIDE) && NT * kLev + kBase > 32 && hi) atomicAdd(&sm.sum[turn][32 + lane], hi);
    add_wide(sm.tt, s.tt);
}
static_assert(V_A == 0 && V_B == 1 && V_C == 2 && V_N == 3 && V_TAU == 4, "a lane a field of a level");
template <int NT, bool WIDE>
__device__ __forceinline__ void share_side(Smem& sm, const Side& o, int turn) {
    if (knows_bins(NT, WIDE)) {
        const uint32_t bins = __reduce_or_sync(FULL, o.bins);
        if ((threadIdx.x & 31) == 0 && bins) atomicOr(&sm.used[turn][2], bins);
    }
    const uint32_t c = __reduce_add_sync(FULL, o.cnt), n = __reduce_add_sync(FULL, o.n), l = __reduce_add_sync(FULL, o.l),
                   tau = __reduce_add_sync(FULL, o.tau);
    add_wide(sm.side_tt, o.tt);
    if ((threadIdx.x & 31) == 0 && c) {
        atomicAdd(&sm.side_sum[0], c); atomicAdd(&sm.side_sum[1], n); atomicAdd(&sm.side_sum[2], l); atomicAdd(&sm.side_sum[3], tau);
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

// What the run before used is clear for the next one (all have read it).
__device__ __forceinline__ void clear_before(Smem& sm, int turn) {
    for (int f = threadIdx.x; f < kBase + kGridRows * kLev; f += kThreads) sm.sum[turn ^ 1][f] = 0;
    if (threadIdx.x < 3) sm.used[turn ^ 1][threadIdx.x] = 0;
}

// Enters what the block has totalled for a run of the columns [q0, q1), or takes it from them (neg), and clears it.  All
// threads call; barriers before and after.  Only groups of 32 bins that the run has counts in are looked at (a run over all
// bins of nine histograms took longer than the sweep of a few hundred requests).
template <int NT, bool WIDE>
__device__ __forceinline__ void enter(Smem& sm, uint32_t* tbt, const Tables<WIDE>& tb, int g, int q0, int q1, bool neg, int turn) {
    using word = typename Tables<WIDE>::word;
    const bool back = q1 < tb.K;
    each_bin<!knows_bins(NT, WIDE)>(sm.used[turn][0], [&](int b) {
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
        const uint32_t* sum = sm.sum[turn];
        unsigned long long x = (f >= kBase && (f - kBase) % kLev == V_TAU) ? (unsigned long long)(long long)(int32_t)sum[f] : sum[f];
        if (has_levels(NT, WIDE) && f >= kBase)
            for (int h = f + kLev; h < F; h += kLev) x += sum[h];      // (so do these)
        if (f == B_TT) x = take_wide(sm.tt);
        if (!x) continue;
        if (neg) x = 0ull - x;
        atomicAdd(&tb.sum_row(g, q0)[f], x);
        if (back) atomicAdd(&tb.sum_row(g, q1)[f], 0ull - x);
    }
    clear_before(sm, turn);
}

// The same for the run beside it, of the columns below q1: the device alone, or the server.
template <int NT, bool WIDE>
__device__ __forceinline__ void enter_side(Smem& sm, uint32_t* side_tbt, const Tables<WIDE>& tb, int g, int q1, bool server, int turn) {
    using word = typename Tables<WIDE>::word;
    const bool back = q1 < tb.K;
    each_bin<!knows_bins(NT, WIDE)>(sm.used[turn][2], [&](int b) {
        const uint32_t x = sm.side_ttft[b];
        if (x) {
            sm.side_ttft[b] = 0;
            atomicAdd(&tb.ttft_row(0)[b], x);
            if (back) atomicAdd(&tb.ttft_row(q1)[b], 0u - x);
        }
        if (WIDE) {
            const word y = side_tbt[b];
            if (y) {
                side_tbt[b] = 0;
                for (int r = 0; r < tb.T; ++r) {
                    atomicAdd(&tb.tbt_row(0, r)[b], y);
                    if (back) atomicAdd(&tb.tbt_row(q1, r)[b], (word)0 - y);
                }
            }
        }
    });
    if (threadIdx.x < 5) {
        const int k = threadIdx.x;
        const unsigned long long x = k < 4 ? (unsigned long long)sm.side_sum[k] : take_wide(sm.side_tt);
        if (k < 4) sm.side_sum[k] = 0;
        const int f = k == 0 ? B_DO : k == 1 ? B_TD : k == 2 ? (server ? B_PS : B_PD) : k == 3 ? B_TAU : B_TT;
        if (x && !(server && k < 2)) {                                 // (none of these requests runs on the device)
            atomicAdd(&tb.sum_row(g, 0)[f], x);
            if (back) atomicAdd(&tb.sum_row(g, q1)[f], 0ull - x);
        }
    }
    clear_before(sm, turn);
}

// ---- side by side: a lane a request, with what it comes to in all its runs.  A run swept by a block costs its barriers, its first
// loads' latency and a walk over its histograms, some 2.5 us, which pays only with enough requests to share it.  Here the lanes of
// a warp whose requests have the same runs -- neighbours do, the requests are stored by length -- enter each run together: the sums
// are added up over the lanes and entered by a lane a field, the histograms by a lane a request (one for all in the same bin).  What is
// left of a warp enters its runs lane by lane.  Bound: latency for small traces, then the atomic additions (some 250 a nanosecond on
// all of the GPU).  With every sum entered by every lane 20,000 requests in six groups under 64 budgets took some 40 us, run by run
// 147, together 11; 100,000 under 32 by 4 80 us, now 20.
constexpr int kJoin = 8;                               // lanes that join, at least

// Adds to the tables of a slab: a count to a histogram of the columns [q0, q1), a value to a sum.
struct Adder {
    unsigned long long* sums;
    size_t F;
    int K;
    __device__ __forceinline__ void count(uint32_t* at, int q0, int q1, uint32_t x) const {
        atomicAdd(at + (size_t)q0 * kNBins, x);
        if (q1 < K) atomicAdd(at + (size_t)q1 * kNBins, 0u - x);
    }
    __device__ __forceinline__ void add(int f, unsigned long long v, int q0, int q1) const {
        atomicAdd(sums + q0 * F + f, v);
        if (q1 < K) atomicAdd(sums + q1 * F + f, 0ull - v);
    }
};
struct Request {                                       // a lane's; level: rows that migrate where the winner may hand over, [0, level)
    uint32_t S, l, n, m, dly, Td;
    int stall, level;
};
template <int NT>
__device__ __forceinline__ Request request_of(const Ctx& c, const float* th, const uint4& q, const uint2& hand, float& saving) {
    Request r;
    r.S = q.x; r.l = q.y & 0xFFFFu; r.n = q.y >> 16; r.m = hand.x & 0xFFFFu; r.dly = hand.x >> 16;
    r.Td = c.kappa * r.l + c.c0;
    r.stall = bin_of_ticks(hand.y);
    saving = r.m ? c.delta_c * (float)(c.E0 ? max(c.E0 - (int)r.m, 0) : (int)(r.n - r.m)) : -1.0f;
    r.level = 0;
#pragma unroll
    for (int k = 0; k < NT; ++k) r.level += saving > th[k] ? 1 : 0;
    return r;
}
// What a request comes to under the columns [q0, q1), which start the device after w, entered by its lane alone.
__device__ __forceinline__ void enter_run(const Adder& t, const Tables<false>& tb, const Request& r, int cand, uint32_t w, int q0, int q1) {
    const bool started = r.S > w, dev_wins = r.S > w + r.Td;
    const uint32_t tt = min(r.S, w + r.Td);
    const int bin = bin_of_ticks(tt);
    if (DBG_OK(bin, kNBins, DBG_K_GRID, DBG_BIN)) t.count(tb.ttft + bin, q0, q1, 1u);
    if (dev_wins) { t.add(B_TD, r.n, q0, q1); t.add(B_DW, 1ull, q0, q1); }
    t.add(B_PS, r.l, q0, q1);
    if (started) { t.add(B_PD, r.l, q0, q1); t.add(B_RACE, 1ull, q0, q1); }
    t.add(B_TAU, r.n - 1u, q0, q1); t.add(B_TT, tt, q0, q1);
    if (!started || (dev_wins ? 2 : 1) != cand) return;
#pragma unroll 1
    for (int k = 0; k < r.level; ++k) {
        const int f = kBase + k * kLev;
        t.add(f + V_A, r.n - r.m, q0, q1); t.add(f + V_B, r.l + r.m, q0, q1); t.add(f + V_N, 1ull, q0, q1);
        if (r.dly) t.add(f + V_C, r.dly, q0, q1);
        if (DBG_OK(r.stall, kNBins, DBG_K_GRID, DBG_BIN)) t.count(tb.tbt + (size_t)k * t.K * kNBins + r.stall, q0, q1, 1u);
    }
}
// What the requests of the lanes `mine` come to under the columns [q0, q1), which start the device after w, together: the sums are added
// up over the lanes and entered once, a lane a field.  alone: the device alone answers.
template <int NT>
__device__ __forceinline__ void join_run(const Adder& t, const Tables<false>& tb, const Request& r, int cand, bool mine, bool alone, uint32_t w, int q0, int q1) {
    const int lane = threadIdx.x & 31;
    const uint32_t all = __ballot_sync(FULL, mine);
    if (!all) return;
    const bool started = mine && !alone && r.S > w, dev_wins = mine && (alone || r.S > w + r.Td);
    const uint32_t tt = alone ? r.Td : min(r.S, w + r.Td);
    const int bin = bin_of_ticks(tt), first = __shfl_sync(FULL, bin, __ffs(all) - 1);
    const uint32_t like = __ballot_sync(FULL, mine && bin == first);     // (one prompt length, one TTFT of the device)
    if (mine && (bin != first || lane == __ffs(all) - 1) && DBG_OK(bin, kNBins, DBG_K_GRID, DBG_BIN))
        t.count(tb.ttft + bin, q0, q1, bin == first ? (uint32_t)__popc(like) : 1u);
    uint32_t lo = 0, hi = 0;
    auto put = [&](int f, uint32_t v) { if (f < 32) { if (lane == f) lo = v; } else if (lane == f - 32) hi = v; };
    const uint32_t sum_l = __reduce_add_sync(FULL, mine ? r.l : 0u);
    put(B_TD, __reduce_add_sync(FULL, dev_wins ? r.n : 0u));
    put(B_TAU, __reduce_add_sync(FULL, mine ? r.n - 1u : 0u));
    if (alone) { put(B_PD, sum_l); put(B_DO, (uint32_t)__popc(all)); }
    else {
        put(B_PS, sum_l);
        put(B_PD, __reduce_add_sync(FULL, started ? r.l : 0u));
        put(B_RACE, (uint32_t)__popc(__ballot_sync(FULL, started)));
        put(B_DW, (uint32_t)__popc(__ballot_sync(FULL, dev_wins)));
    }
    const unsigned long long tt_sum = __reduce_add_sync(FULL, mine ? tt & 0xFFFFu : 0u) + ((unsigned long long)__reduce_add_sync(FULL, mine ? tt >> 16 : 0u) << 16);
    const int level = started && (dev_wins ? 2 : 1) == cand ? r.level : 0;
    const uint32_t movers = __ballot_sync(FULL, level > 0);
    const int leader = movers ? __ffs(movers) - 1 : 0, stall_0 = __shfl_sync(FULL, r.stall, leader);     // (mostly tau, where none stalls)
#pragma unroll
    for (int k = 0; k < NT; ++k) {
        const uint32_t go = __ballot_sync(FULL, level > k), alike = __ballot_sync(FULL, level > k && r.stall == stall_0);
        if (!go) break;
        const int f = kBase + k * kLev;
        put(f + V_A, __reduce_add_sync(FULL, level > k ? r.n - r.m : 0u)); put(f + V_B, __reduce_add_sync(FULL, level > k ? r.l + r.m : 0u));
        put(f + V_C, __reduce_add_sync(FULL, level > k ? r.dly : 0u)); put(f + V_N, (uint32_t)__popc(go));
        const bool by_one = alike != 0u && lane == __ffs(alike) - 1;
        if (level > k && (r.stall != stall_0 || by_one) && DBG_OK(r.stall, kNBins, DBG_K_GRID, DBG_BIN))
            t.count(tb.tbt + (size_t)k * t.K * kNBins + r.stall, q0, q1, by_one ? (uint32_t)__popc(alike) : 1u);
    }
    const unsigned long long x = lane == B_TT ? tt_sum : lo;
    if (x) t.add(lane, x, q0, q1);
    if (NT * kLev + kBase > 32 && hi) t.add(lane + 32, hi, q0, q1);
}

// The requests [from, to) of the block's list, a segment's, for the columns [0, k1).
// A warp a wait: the common one, and those of the columns that wait longer.
template <int NT>
__device__ __noinline__ void enter_listed(const Args& a, const Smem& sm, uint32_t from, uint32_t to, uint32_t wt_min, int n_low, int k1) {
    const Ctx& c = sm.ctx;
    const Tables<false> tb(a.gt, a.slabs[sm.slab], a.tr.n_groups);
    const Adder t = {tb.sum_row(c.g, 0), (size_t)sum_fields(c.T), c.K};
    const int lane = threadIdx.x & 31;
    for (int p = threadIdx.x >> 5; p <= n_low; p += kThreads / 32) {
        const uint32_t w = p < n_low ? sm.w_tail[p] : wt_min;
        const int q1 = p < n_low ? p + 1 : k1;
        if (p >= q1) continue;                                         // (every column waits longer)
#pragma unroll 1
        for (uint32_t i0 = from; i0 < to; i0 += 32) {
            const uint32_t i = min(i0 + lane, to - 1), kk = c.start + sm.list[i];
            if (!DBG_OK(kk, a.tr.n, DBG_K_GRID, DBG_REQUEST)) break;
            float saving;
            const Request r = request_of<NT>(c, sm.rows, a.tr.req[kk], c.may_migrate ? c.hand[kk] : make_uint2(0u, 0u), saving);
            join_run<NT>(t, tb, r, c.cand, i0 + lane < to, false, w, p, q1);
        }
    }
}

template <int NT>
__device__ __forceinline__ void enter_requests(const Args& a, const Ctx& c, const float (&th)[NT], const Smem& sm, const Tables<false>& tb,
                                               bool waits, uint32_t wt_min, int n_low) {
    const int K = c.K, lane = threadIdx.x & 31;
    const Adder t_ = {tb.sum_row(c.g, 0), (size_t)sum_fields(c.T), K};
#pragma unroll 1
    for (uint32_t i0 = threadIdx.x & ~31u; i0 < c.len; i0 += kThreads) {
        const uint32_t kk = c.start + min(i0 + lane, c.len - 1);
        float saving;
        const Request r = request_of<NT>(c, th, a.tr.req[kk], c.may_migrate ? c.hand[kk] : make_uint2(0u, 0u), saving);
        const uint32_t S = r.S, l = r.l, n = r.n, Td = r.Td;
        const bool valid = i0 + lane < c.len && !(c.mixed && saving > c.th_lo && !(saving > th[0]));       // (else left to the pair kernel)
        // the columns on either side of the request's length
        int k1 = 0;
        for (int hi = K; k1 < hi;) { const int mid = (k1 + hi) >> 1; if (waits ? sm.key[mid] < (int)l : sm.key[mid] > (int)l) k1 = mid + 1; else hi = mid; }
        int k2 = k1;
        if (waits) while (k2 < K && sm.key[k2] == (int)l) ++k2;
        const bool longer = waits && valid && S > wt_min && n_low > 0;         // (not covered by the common wait)
        bool joined = false;
        uint32_t todo = __ballot_sync(FULL, valid);
#pragma unroll 1
        while (todo) {
            const int lead = __ffs(todo) - 1, a1 = __shfl_sync(FULL, k1, lead), a2 = __shfl_sync(FULL, k2, lead);
            const uint32_t same = __ballot_sync(FULL, valid && k1 == a1 && k2 == a2);
            todo &= ~same;
            if (__popc(same) < kJoin) continue;
            const bool mine = (same >> lane) & 1u;
            joined = joined || mine;
            if (waits) {
#pragma unroll 1
                for (int p = a1; p < a2; ++p) join_run<NT>(t_, tb, r, c.cand, mine, false, sm.w_star[p], p, p + 1);
            }
            if (a1 > 0) join_run<NT>(t_, tb, r, c.cand, mine && !longer, !waits, waits ? wt_min : 0u, 0, a1);
            if (a1 > n_low) join_run<NT>(t_, tb, r, c.cand, mine && longer, false, wt_min, n_low, a1);
            if (a2 < K) join_run<NT>(t_, tb, r, c.cand, mine, false, 0u, a2, K);
        }
        // (the columns that wait longer have l* = 0: they are in front of every request's k1)
        if (__any_sync(FULL, longer)) {
#pragma unroll 1
            for (int p = 0; p < n_low; ++p) join_run<NT>(t_, tb, r, c.cand, longer, false, sm.w_tail[p], p, p + 1);
        }
        if (valid && !joined) {
            const int low = longer ? n_low : 0;
            for (int p = k1; p < k2; ++p) enter_run(t_, tb, r, c.cand, sm.w_star[p], p, p + 1);
            if (k2 < K) enter_run(t_, tb, r, c.cand, 0u, k2, K);
            if (waits) {
                if (low < k1) enter_run(t_, tb, r, c.cand, wt_min, low, k1);
            } else if (k1 > 0) {                                           // the device alone
                const int bin = bin_of_ticks(Td);
                if (DBG_OK(bin, kNBins, DBG_K_GRID, DBG_BIN)) t_.count(tb.ttft + bin, 0, k1, 1u);
                t_.add(B_DO, 1ull, 0, k1); t_.add(B_TD, n, 0, k1); t_.add(B_PD, l, 0, k1); t_.add(B_TAU, n - 1u, 0, k1); t_.add(B_TT, Td, 0, k1);
            }
        }
        __syncwarp();
    }
}

// MODE: run by run, where no group of the slabs is Algorithm 2's, or where some are (kernels of their own: the second has no registers
// to spare); or a chunk's requests side by side.
template <int NT, bool WIDE, int MODE>
__global__ void __launch_bounds__(kThreads, blocks_for(NT, WIDE, MODE))
k_grid(const __grid_constant__ Args a) {
    constexpr bool WAITS = MODE != M_RACES, JOINED = MODE == M_JOINED;
    static_assert(!(WIDE && JOINED), "windows are added up by runs");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
    uint32_t* tbt = (uint32_t*)(smem_raw + sizeof(Smem));
    const Levels<NT> lv(tbt + NT * kNBins + (has_levels(NT, WIDE) ? (threadIdx.x >> 5) * Levels<NT>::kWords : 0));
    // Beside the slope search of Eq. 1-2 (k_prep_beta), which no plain policy needs: what this kernel reads was complete before that
    // one let it start.  It then waits at its end, for the kernels behind.  (Under 48 such searches, 79 us on 48
    // multiprocessors, 300,000 requests by 16 budgets take 27.)
    for (int i = threadIdx.x; i < (int)(offsetof(Smem, key) / 4); i += kThreads) ((uint32_t*)&sm)[i] = 0;
    if (!JOINED) for (int i = threadIdx.x; i < tbt_words(NT, WIDE); i += kThreads) tbt[i] = 0;
    if (!a.beside) grid_dependency_wait();
    // Another grid beside this one: it has tables of its own, and what it reads was complete before this one's blocks came here.  (Waits
    // for it at its end.  250,000 requests in five classes, a kernel without windows and one with, a step 221 us -> 211.)
    if (a.early) let_next_start();

    int turn = 0;                                                     // which of the two sets of used bins is in use
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
        if (!WIDE && MODE == M_WAITS && list_few(NT) != 0 && threadIdx.x == 0) {
            sm.ctx = c; sm.slab = slab_id;
#pragma unroll
            for (int r = 0; r < NT; ++r) sm.rows[r] = th[r];
        }
        bool waits = false;
        {
            const Prep& pr = a.prep[(size_t)g * a.P + a.tab[sl.cols]];
            waits = WAITS && pr.device_constrained != 0;
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
        for (int q = threadIdx.x; !JOINED && q < (waits ? 2 * K + 1 : K + 1); q += kThreads) {
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

        if constexpr (JOINED) {
            enter_requests<NT>(a, c, th, sm, tb, waits, wt_min, n_low);
            passes = 1;
        }
        // a segment's last columns, which wait 0, and beside them its first ones: the device alone
        if (MODE == M_RACES || (MODE == M_WAITS && !waits)) {
            for (int si = 0; si < n_seg; ++si) {
                const Seg sg = sm.seg[si];
                const bool race = (int)sg.k2 < K, side = sg.k1 > 0;
                Acc<NT, WIDE> s = {};
                Side o = {};
                sweep<NT, WIDE, S_DEVICE>(a, c, th, sm, tbt, lv, sg.pa, sg.pb, 0u, false, false, race, side, s, o);
                if (race) share_out<NT, WIDE>(sm, s, lv, turn);
                if (side) share_side<NT, WIDE>(sm, o, turn);
                __syncthreads();
                if (race) enter<NT, WIDE>(sm, tbt, tb, g, sg.k2, K, false, turn);
                if (side) enter_side<NT, WIDE>(sm, tbt + NT * kNBins, tb, g, sg.k1, false, turn);
                __syncthreads();
                ++passes; turn ^= 1;
            }
        } else if constexpr (WIDE) {
            // Windows: run by run, [k2, K), each column of [k1, k2), [0, k1), and, when the list is half full or the chunk is done, the list
            // for the columns that wait longer, with the common wait's totals taken back from them.  (A sweep for two runs, and the
            // turns of the kernels below, cost registers that are short here: 250,000 requests in five classes, those with windows 46.7 us
            // instead of 42.0.)
            auto run = [&](uint32_t pa, uint32_t pb, uint32_t w, bool list, bool push, int q0, int q1, bool neg) {
                Acc<NT, WIDE> s = {};
                Side none = {};
                sweep<NT, WIDE, S_NONE>(a, c, th, sm, tbt, lv, pa, pb, w, list, push, true, false, s, none);
                share_out<NT, WIDE>(sm, s, lv, turn);
                __syncthreads();
                enter<NT, WIDE>(sm, tbt, tb, g, q0, q1, neg, turn);
                __syncthreads();
                ++passes; turn ^= 1;
            };
            constexpr uint32_t kListStep = kListCap / 2;
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
                bool full = done;
                if (push) {                                           // all threads see the same, and only then may the next run add to it
                    full = sm.n_list > (uint32_t)(kListCap - kListStep);
                    __syncthreads();
                }
                if (full) {
                    const uint32_t k = sm.n_list;                     // (nobody adds to it from here to the runs' end)
                    __syncthreads();
                    if (threadIdx.x == 0) sm.n_list = 0;
                    for (int p = -1; p < n_low; ++p)                  // the common wait's totals go, each column's own come
                        run(0u, k, p < 0 ? wt_min : sm.w_tail[p], true, false, max(p, 0), p < 0 ? n_low : p + 1, p < 0);
                }
            }
        } else if constexpr (MODE == M_WAITS) {
            // Algorithm 2, segment by segment: each column of [k1, k2) under its own w*; then [k2, K), which waits 0, in one sweep with [0, k1),
            // which waits w_tail.  (Groups of Algorithm 3 have the way above: with one for both 300,000 requests of six groups under 32 policies took
            // 26.1 us instead of 24.8, 600,000 under 32 by 2 30.0 instead of 28.4, 2 M under 64 by 2 48.8 instead of 47.0.)  The few requests that w_tail does not cover have been listed.  A handful is
            // entered request by request; more are entered for [0, k1) from the list, and when it is half full or the chunk is done,
            // the columns that wait longer get what they come to there under their own wait in place of the common one.
            enum { POINTS, MAIN, LISTED, LONGER } at = POINTS;
            uint32_t pos = 0, listed = 0, n_list = 0;                  // where the segment's sweep goes on; the list: entered for [0, k1), all
            int si = 0, ri = 0;                                       // segment, point or column
#pragma unroll 1
            for (;;) {
                uint32_t from = 0, to = 0, w = 0;
                int q0 = 0, q1 = 0;
                bool list = false;
                if (at == POINTS) {
                    if (si >= n_seg) {
                        if (n_list == 0) break;
                        at = LONGER; ri = 0;
                        continue;
                    }
                    const Seg sg = sm.seg[si];
                    if (ri >= (int)sg.k2 - (int)sg.k1) { at = MAIN; pos = sg.pa; continue; }
                    from = sg.pa; to = sg.pb; q0 = (int)sg.k1 + ri; q1 = q0 + 1; w = sm.w_star[q0];
                    ++ri;
                } else if (at == MAIN) {
                    const Seg sg = sm.seg[min(si, kMaxSeg - 1)];
                    const bool race = (int)sg.k2 < K, side = sg.k1 > 0;
                    if (pos >= sg.pb || !(race || side)) { at = POINTS; ri = 0; ++si; continue; }
                    if (!side || (!race && n_low == 0)) {
                        // no two runs to sweep at once, and no column that wants the list: a run of its own, without one (six groups under one policy,
                        // evaluation and reduction: 100,000 requests 39.4 us -> 38.1, a million 57.9 -> 57.0, under 1 by 8 300,000 51.1 -> 48.9)
                        from = sg.pa; to = sg.pb;
                        if (side) { w = wt_min; q1 = sg.k1; } else { q0 = sg.k2; q1 = K; }
                        at = POINTS; ri = 0; ++si;
                    } else {
                        Acc<NT, WIDE> s = {};
                        Side o = {};
                        for (;;) {
                            const uint32_t end = min((uint32_t)sg.pb, pos + list_room(n_list));
                            sweep<NT, WIDE, S_SERVER>(a, c, th, sm, tbt, lv, pos, end, wt_min, false, false, race, true, s, o);
                            pos = end;
                            __syncthreads();
                            n_list = sm.n_list;
                            __syncthreads();
                            if (pos >= sg.pb || list_room(n_list) == 0u) break;
                        }
                        if (race) share_out<NT, WIDE>(sm, s, lv, turn);
                        share_side<NT, WIDE>(sm, o, turn);
                        if constexpr (list_few(NT) != 0) {
                            if (n_list > listed && n_list - listed <= (uint32_t)list_few(NT)) {
                                enter_listed<NT>(a, sm, listed, n_list, wt_min, n_low, sg.k1);
                                n_list = listed;
                            }
                        }
                        __syncthreads();
                        if (threadIdx.x == 0) sm.n_list = n_list;
                        if (race) enter<NT, WIDE>(sm, tbt, tb, g, sg.k2, K, false, turn);
                        enter_side<NT, WIDE>(sm, tbt + NT * kNBins, tb, g, sg.k1, true, turn);
                        __syncthreads();
                        ++passes; turn ^= 1;
                        if (n_list > listed) at = LISTED;
                        continue;
                    }
                } else if (at == LISTED) {
                    const int k1 = sm.seg[si].k1;
                    list = true; from = listed; to = n_list; w = wt_min; q0 = n_low; q1 = k1;
                    listed = n_list;
                    at = MAIN;
                    if (n_low == 0) listed = n_list = 0;
                    else if (n_list > (uint32_t)kListCap / 2) { at = LONGER; ri = 0; }
                    if (q0 >= k1) continue;                            // (every column waits longer)
                } else {
                    list = true; to = n_list; w = sm.w_tail[ri]; q0 = ri; q1 = ri + 1;
                    if (++ri == n_low) { listed = n_list = 0; at = si >= n_seg ? POINTS : MAIN; }
                }
                Acc<NT, WIDE> s = {};
                Side none = {};
                sweep<NT, WIDE, S_NONE>(a, c, th, sm, tbt, lv, from, to, w, list, false, true, false, s, none);
                share_out<NT, WIDE>(sm, s, lv, turn);
                __syncthreads();
                if (n_list == 0 && threadIdx.x == 0) sm.n_list = 0;
                enter<NT, WIDE>(sm, tbt, tb, g, q0, q1, false, turn);
                __syncthreads();
                ++passes; turn ^= 1;
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
            sm.n_seg = 0; sm.n_list = 0; sm.flagged = 0;
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
         unsigned long long* __restrict__ hist_ttft, unsigned long long* __restrict__ hist_tbt, bool beside, bool early) {
    __shared__ unsigned long long s_part[kSpreadWarps * 33];
    // (beside another such kernel, which began when the tables were complete: the last block waits for it)
    if (!beside || (blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1)) grid_dependency_wait();
    if (early) let_next_start();
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

size_t grid_smem(int NT, bool wide) { return sizeof(Smem) + (size_t)tbt_words(NT, wide) * 4; }

template <int NT, bool WIDE, int MODE>
cudaError_t launch_one(const Args& a, int sms, cudaStream_t st) {
    const size_t smem = MODE == M_JOINED ? sizeof(Smem) : grid_smem(NT, WIDE);
    auto* kernel = k_grid<NT, WIDE, MODE>;
    cudaError_t e = allow_smem((const void*)kernel, smem);
    if (e) return e;
    const uint64_t items = (uint64_t)a.n_chunks * a.n_slabs;
    const uint32_t blocks = (uint32_t)std::min<uint64_t>(items, (uint64_t)sms * blocks_for(NT, WIDE, MODE));
    return launch_after(kernel, dim3(blocks), kThreads, smem, st, a);
}
template <int NT>
cudaError_t launch_rows(const Args& a, bool wide, int mode, int sms, cudaStream_t st) {
    if (wide) return mode == M_RACES ? launch_one<NT, true, M_RACES>(a, sms, st) : launch_one<NT, true, M_WAITS>(a, sms, st);
    return mode == M_RACES ? launch_one<NT, false, M_RACES>(a, sms, st) : mode == M_WAITS ? launch_one<NT, false, M_WAITS>(a, sms, st)
                                                                                         : launch_one<NT, false, M_JOINED>(a, sms, st);
}

}  // namespace

DBG_TRANSLATION_UNIT()

// Side by side or run by run.  Run by run a threshold of a group costs a run's latency, in the chunks that it falls into; side by side the
// requests add to the same rows of the tables, two runs each (under one policy setting one), and the fewer columns there are the more
// of them meet.  (Evaluation and reduction, us, run by run and side by side: one group, 60,000 requests under budgets of 0 and 1 31 and 40, under 4 34 and 36,
// 130,000 under 64 40 and 41, 220,000 under 256 62 and 58, 400,000 63 and 68; six groups, 60,000 under 0 and 1 36 and 49, under one 80,000 37 and 39,
// 130,000 under 16 51 and 47, 220,000 53 and 55, 400,000 under 64 75 and 77, under 128 113 and 91, 550,000 101 and 117, 750,000 under 256 175 and 142,
// 1.3 million 194 and 216, under 16 by 8 170,000 72 and 64, 400,000 74 and 86, under 128 by 8 750,000 174 and 172.  How fast the rows are
// added to depends on where they lie -- k_grid of 400,000 requests of six groups under 64 by 2 took 59 us in one context, run by run 44 there, and as
// long as run by run in others --: the line lies in front of where both meet.)
// It is asked slab by slab: a narrow grid beside a wide one goes its own way (six groups, a million requests under 256 by 4, and sixteen times 2 by 4
// of other expected lengths, 779 us all side by side, now 484; under 256 by 4 and one 300, now 248; one group, 150,000 under 128 by 8 and eight
// times 4 164, now 141).
// Budgets of 0 and 1 alone part no requests: a chunk is one run or two, and side by side all requests meet in the same rows.
bool grid_joins(uint32_t n, int groups, int K, int T, bool inner) {
    return n <= (K == 1 ? 60000.0 : !inner ? 16000.0 : 10000.0 * std::pow((double)K * groups, 0.6)) * (1.0 + T / 16.0);
}
uint64_t grid_ttft_words(int K) { return (uint64_t)K * kNBins; }
uint64_t grid_tbt_words(int K, int T) { return (uint64_t)K * T * kNBins; }
uint64_t grid_sum_words(int K, int T, int G) { return (uint64_t)G * K * sum_fields(T); }
uint32_t grid_blocks_per_sm(int T) { return (uint32_t)blocks_for(rows_for(T), false, M_WAITS); }
int grid_rows(int T) { return rows_for(T); }

cudaError_t launch_grid(const TraceDev& tr, const GroupConst* gc, const ClassConst* classes, const Prep* prep, uint32_t P,
                        const Slab* slabs, uint32_t n_slabs, int T, bool wide, const uint32_t* tab,
                        const Chunk* chunks, uint32_t n_chunks, TimelineRec rec, size_t rec_stride, GridTables gt, LeftLists left,
                        uint32_t k0, uint32_t* ticket, uint64_t* work, bool beside, bool early, bool waits, bool joined, int sms, cudaStream_t st) {
    if (n_chunks == 0 || n_slabs == 0) return cudaSuccess;
    if ((uint64_t)n_chunks * n_slabs > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
    const Args a = {tr, rec, gc, rec_stride, classes, prep, P, slabs, n_slabs, tab, chunks, n_chunks, gt, left, k0, ticket,
                    (unsigned long long*)work, beside, early};
    const int mode = joined ? M_JOINED : waits ? M_WAITS : M_RACES;
    switch (rows_for(T)) {
        case 1: return launch_rows<1>(a, wide, mode, sms, st);
        case 2: return launch_rows<2>(a, wide, mode, sms, st);
        case 4: return launch_rows<4>(a, wide, mode, sms, st);
        default: return launch_rows<8>(a, wide, mode, sms, st);
    }
}

cudaError_t launch_spread(const TraceDev& tr, const GroupConst* gc, const Slab* slabs, uint32_t n_slabs, int T,
                          bool wide, const uint32_t* tab, GridTables gt, uint64_t* acc, uint64_t* hist_ttft,
                          uint64_t* hist_tbt, bool beside, bool early, cudaStream_t st) {
    if (n_slabs == 0) return cudaSuccess;
    const dim3 grid((uint32_t)(2 * T * (kNBins / 32) + (tr.n_groups * T * kNAcc + 31) / 32), n_slabs);
    auto* kernel = wide ? k_spread<true> : k_spread<false>;
    return launch_after(kernel, grid, kSpreadWarps * 32, 0, st, tr, gc, slabs, tab, gt, (unsigned long long*)acc,
                        (unsigned long long*)hist_ttft, (unsigned long long*)hist_tbt, beside, early);
}

}  // namespace disco
