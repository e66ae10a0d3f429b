// Decode play-out (Sec. 4.3) of the groups whose streams are delivered as they are generated (G_FREE): pacing is off, or
// every token takes at least tau, so that the reader always waits for it (d_j = g_j, TBT_j = x_j); a stream that cannot
// clamp beside it keeps the pace and is not played.  Every token's interval goes to a sum, a maximum and a window of
// histogram bins.
//
// Bound: integer issue (a hash, a range map and a bin per token and stream; 40 cycles for 32 tokens of two streams, where about
// thirty instructions are issued).  A warp plays a request, a lane every 32nd token.  The counters are [bin][8] in shared
// memory: four lanes share a column, by atomic additions that nobody waits for.  Two requests share a counter's halves
// before the columns are added up (a lane a bin, four counters at a time) and written as rows of 16-bit counts.  The stream
// after a hand-off stores no window: it is the target's without token 2, which the reductions take away (x_stream in
// disco_internal.cuh).  200,000 requests of 200 tokens, two streams: 95 us with a column a lane, read and written (23 of
// them to add up and clear eight times the counters) and batches of eight dealt out in turn, 76 now; 4 or 16 columns equal, but one bin
// for all tokens 89 with four.  125,000 with one stream, chosen as it went: 63 us, 44 in a kernel of its own.  Five or
// six blocks a multiprocessor: 78 and 82 us.
#include <algorithm>

#include "disco_internal.cuh"

namespace disco {

namespace {

constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr int kFreeWarps = 8;
constexpr int kFreeBlocks = 4;            // to a multiprocessor
constexpr int kCols = 8;                  // columns of counters a warp has
constexpr uint32_t kFreeBatch = 16;       // requests a warp takes at a time, at most (a lane each)

// Where a stream's window of counters starts for this lane, and the bin in front of it.
struct Counters { uint32_t* at; int lo, W; };

// One interval of x ticks more.  SMALL: intervals below 32 ticks occur, which have bins of their own (bin_of_ticks).
template <bool SMALL>
__device__ __forceinline__ void count_in(const Counters& c, uint32_t x, uint32_t inc) {
    const int b = (SMALL ? bin_of_ticks(x) : (int)(__float_as_uint(__uint2float_rz(x)) >> 18) - ((127 + 4) << 5)) - c.lo;
    if (DBG_OK(b, c.W, DBG_K_PLAYOUT, DBG_WINDOW)) atomicAdd(&c.at[b * kCols], inc);
}
// PLAY: which streams are played.  P_BOTH: pacing is off, both, and a hand-off may follow the first token.  Otherwise pacing is
// on, a stream or two clamp at every token and no buffer fills: the server's or the device's in all groups, or what a group's
// are.  (Kernels of their own: in one kernel for all cases the warps waited for instructions four cycles of every ten.)
enum Play { P_GROUP = 0, P_SERVER, P_DEVICE, P_BOTH };

template <int PLAY, bool SMALL>
__global__ void __launch_bounds__(kFreeWarps * 32, kFreeBlocks)
k_playout_free(TraceDev tr, const GroupConst* __restrict__ gcs, const __grid_constant__ ClassConst cc,
               const int32_t* __restrict__ knots, uint32_t k0, TimelineRec rec, const __grid_constant__ FreeMore more,
               uint32_t* __restrict__ ticket, uint32_t batches, uint32_t size, bool beside, bool early) {
    constexpr bool BOTH = PLAY == P_BOTH;
    extern __shared__ __align__(16) uint32_t s_win[];         // per warp: [W0 + W1][kCols] counters
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, warps = blockDim.x >> 5;
    // (beside the play-out of other classes, which began when the load was complete: the last block waits for it)
    if (!beside || blockIdx.x == gridDim.x - 1) grid_dependency_wait();
    if (early) let_next_start();
    const int W0 = cc.W[0], W1 = cc.W[1], WW = W0 + W1;
    uint32_t* win = s_win + wib * (WW * kCols);
    for (int b = lane; b < WW * kCols; b += 32) win[b] = 0;
    __syncwarp();
    // A warp starts with a batch of its own and then draws the next one, ahead of time: each batch draws once, so that the
    // counter is zero again behind the last.
    uint32_t batch = blockIdx.x * warps + wib;
    while (batch < batches) {
        uint32_t drawn = 0;
        if (lane == 0) drawn = atomicInc(ticket, batches - 1u);
        int g;
        uint32_t k_lo, n_here;
        if (!batch_of_kind(tr, cc, G_FREE, size, batch, g, k_lo, n_here)) break;
        const GroupConst& gc = gcs[g];
        const uint32_t mul0 = 2u * (uint32_t)gc.J_srv + 1u, mul1 = 2u * (uint32_t)gc.J_dev + 1u;
        const uint32_t base0 = (uint32_t)(gc.T_srv - gc.J_srv), base1 = (uint32_t)(gc.T_dev - gc.J_dev);   // x = base + ((h * mul) >> 32)
        const Counters ct0 = {win + lane % kCols, cc.lo[g][0], W0}, ct1 = {win + W0 * kCols + lane % kCols, cc.lo[g][1], W1};
        const bool on0 = PLAY != P_GROUP ? (PLAY & 1) != 0 : !(cc.even[g] & 1u), on1 = PLAY != P_GROUP ? (PLAY & 2) != 0 : !(cc.even[g] & 2u);
        // without pacing the buffer is empty and the dearer winner hands over after its first token
        const int cand = (BOTH && cc.mig_any) ? gc.candidate : 0;
        const bool to_dev = cand == 1;
        // ---- one request per lane: inputs, results
        uint32_t n_l = 1, l_l = 1, key_l = 0;
        if (lane < n_here) {
            const uint4 q = tr.req[k_lo + lane];
            n_l = q.y >> 16; l_l = q.y & 0xFFFFu;
            key_l = mix32(k0 + q.z * kHashReq);
        }
        // sums of the intervals, and the largest hash from token 3 on (an interval grows with its hash)
        uint32_t o_s0 = 0, o_s1 = 0, o_h = 0;
        const int b_lo = on0 ? 0 : W0, b_hi = on1 ? WW : W0;      // the bins in use
        for (int r0 = 0; r0 < (int)n_here; r0 += 2) {
            const int pair = min(2, (int)n_here - r0);
#pragma unroll 1
            for (int half = 0; half < pair; ++half) {
                const int r = r0 + half;
                const uint32_t n = __shfl_sync(FULL, n_l, r), inc = half ? 65536u : 1u;
                uint32_t hin = __shfl_sync(FULL, key_l, r) + (2u + lane) * kHashTok;
                uint32_t s0 = 0, s1 = 0, most = 0, j = 2u + lane;
                // one token: its interval in each stream that is played
                auto token = [&]() {
                    const uint32_t h = mix32(hin);
                    hin += 32u * kHashTok;
                    if (on0) { const uint32_t x = mad_hi(h, mul0, base0); s0 += x; count_in<SMALL>(ct0, x, inc); }
                    if (on1) { const uint32_t x = mad_hi(h, mul1, base1); s1 += x; count_in<SMALL>(ct1, x, inc); }
                    return h;
                };
                if (j <= n) {
                    const uint32_t h = token();
                    if (lane != 0) most = h;                      // (lane 0 had token 2)
#pragma unroll 2
                    for (j += 32u; j <= n; j += 32u) most = max(most, token());
                }
                if (on0) s0 = __reduce_add_sync(FULL, s0);
                if (on1) s1 = __reduce_add_sync(FULL, s1);
                most = __reduce_max_sync(FULL, most);
                if (lane == r) { o_s0 = s0; o_s1 = s1; o_h = most; }
            }
            __syncwarp();
            // the lanes' counts are added up and go out; the counters are cleared for the next pair
            const size_t k = k_lo + r0;
#pragma unroll 1
            for (int b = b_lo + lane; b < b_hi; b += 32) {
                uint4* row = reinterpret_cast<uint4*>(win + b * kCols);
                uint32_t t = 0;
#pragma unroll
                for (int c = 0; c < kCols / 4; ++c) {
                    const int at = (c + b / (32 / kCols)) & (kCols / 4 - 1);
                    const uint4 x = row[at];
                    row[at] = make_uint4(0u, 0u, 0u, 0u);
                    t += x.x + x.y + x.z + x.w;
                }
                const bool first = b < W0;
                uint16_t* to = first ? rec.win[0] + k * W0 + b : rec.win[1] + k * W1 + (b - W0);
                to[0] = (uint16_t)t;
                if (pair > 1) to[first ? W0 : W1] = (uint16_t)(t >> 16);
            }
            __syncwarp();
        }
        if (lane < n_here) {
            const uint32_t k = k_lo + lane, nI = n_l - 1u, tau = (uint32_t)cc.tau;
            uint32_t m = 0, M = 0, sumX = 0, maxX = 0;
            const uint32_t sum0 = on0 ? o_s0 : nI * tau, sum1 = on1 ? o_s1 : nI * tau;
            const uint32_t h2 = mix32(key_l + 2u * kHashTok);         // token 2's
            if (BOTH && cand && nI) {
                m = 1;
                if (to_dev) M = (uint32_t)gc.kappa * (l_l + 1u) + (uint32_t)gc.c0;
                else {
                    const uint32_t u = mix32(key_l);          // a server TTFT drawn from F by its knots
                    const uint32_t ki = u >> 24, fr = (u >> 8) & 0xFFFFu;
                    const int32_t* K = knots + g * kNKnots;
                    if (DBG_OK(ki + 1, kNKnots, DBG_K_PLAYOUT, DBG_KNOT))
                        M = (uint32_t)(K[ki] + (int32_t)(((int64_t)(K[ki + 1] - K[ki]) * (int64_t)fr) >> 16));
                }
                sumX = M + (to_dev ? sum1 - mad_hi(h2, mul1, base1) : sum0 - mad_hi(h2, mul0, base0));
                maxX = max(M, nI > 1u ? (to_dev ? mad_hi(o_h, mul1, base1) : mad_hi(o_h, mul0, base0)) : 0u);
            }
            const uint32_t most0 = mad_hi(max(o_h, h2), mul0, base0), most1 = mad_hi(max(o_h, h2), mul1, base1);
            rec.hand[k] = make_uint2(m, M);
            rec.sum[0][k] = sum0; rec.sum[1][k] = sum1; rec.sum[2][k] = sumX;
            rec.max[0][k] = nI ? (on0 ? most0 : tau) : 0u; rec.max[1][k] = nI ? (on1 ? most1 : tau) : 0u;
            rec.max[2][k] = maxX;
            // classes that differ in the pace alone: the same intervals, another pace beside them, and no hand-off either
            for (int c = 0; !BOTH && c < more.n; ++c) {
                const uint32_t pace = (uint32_t)more.tau[c];
                auto put = [&](uint32_t* at, uint32_t v) { *reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(at + k) + more.off[c]) = v; };
                *reinterpret_cast<uint2*>(reinterpret_cast<char*>(rec.hand + k) + more.off[c]) = make_uint2(0u, 0u);
                put(rec.sum[0], on0 ? sum0 : nI * pace); put(rec.sum[1], on1 ? sum1 : nI * pace); put(rec.sum[2], 0u);
                put(rec.max[0], nI ? (on0 ? most0 : pace) : 0u); put(rec.max[1], nI ? (on1 ? most1 : pace) : 0u); put(rec.max[2], 0u);
            }
        }
        __syncwarp();
        batch = gridDim.x * warps + __shfl_sync(FULL, drawn, 0);
    }
}

}  // namespace

DBG_TRANSLATION_UNIT()

cudaError_t launch_playout_free(const TraceDev& tr, const GroupConst* gc, const ClassConst& cc, const int32_t* knots, uint32_t k0, TimelineRec rec,
                                const FreeMore& more, uint32_t* ticket, const uint32_t* grp_n, bool beside, bool early, int sms, cudaStream_t st) {
    // as many warps to a block as the windows leave room for (wide jitter: up to 27 KB of counters a stream and warp)
    const size_t per_warp = (size_t)(cc.W[0] + cc.W[1]) * kCols * 4;
    const uint32_t warps = std::max<uint32_t>(1u, std::min<uint32_t>(kFreeWarps, (uint32_t)(100 * 1024 / per_warp)));
    const size_t smem = per_warp * warps;
    bool small = false;                                       // intervals below 32 ticks occur
    uint64_t n = 0;
    int play = P_BOTH;
    for (int g = 0; g < tr.n_groups; ++g) {
        small = small || cc.lo[g][0] < 32 || cc.lo[g][1] < 32;
        if (cc.kind[g] != G_FREE || !grp_n[g]) continue;
        const int here = (cc.even[g] & 1 ? 0 : 1) | (cc.even[g] & 2 ? 0 : 2);
        play = !cc.pacing ? P_BOTH : here != P_BOTH && (n == 0 || here == play) ? here : P_GROUP;
        n += grp_n[g];
    }
    // Some three batches a warp, of an even number of requests: draws follow each other at 0.7 ns and a batch takes a microsecond to
    // begin with (100,000 requests in twos 36 us, in fours 21, in sevens 18; the other way round, eight warps' worth of long
    // outputs wait for the last batch).
    const uint32_t at_once = (uint32_t)sms * kFreeBlocks * kFreeWarps, size = (uint32_t)std::min<uint64_t>(kFreeBatch, std::max<uint64_t>(2, n / (at_once * 3ull) / 2 * 2));
    uint32_t batches = 0;
    for (int g = 0; g < tr.n_groups; ++g) if (cc.kind[g] == G_FREE) batches += (grp_n[g] + size - 1) / size;
    auto* kernel = play == P_BOTH ? (small ? k_playout_free<P_BOTH, true> : k_playout_free<P_BOTH, false>)
                 : play == P_SERVER ? (small ? k_playout_free<P_SERVER, true> : k_playout_free<P_SERVER, false>)
                 : play == P_DEVICE ? (small ? k_playout_free<P_DEVICE, true> : k_playout_free<P_DEVICE, false>)
                                    : (small ? k_playout_free<P_GROUP, true> : k_playout_free<P_GROUP, false>);
    cudaError_t e;
    if ((e = allow_smem((const void*)kernel, 227 * 1024))) return e;
    const uint32_t blocks = std::min<uint32_t>((batches + warps - 1) / warps, at_once / warps);
    return launch_after(kernel, blocks, warps * 32, smem, st, tr, gc, cc, knots, k0, rec, more, ticket, batches, size, beside, early);
}

}  // namespace disco
