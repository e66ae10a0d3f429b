// Decode play-out (Sec. 4.3) of the groups whose streams are delivered as they are generated (G_FREE): pacing is off, or
// every token takes at least tau, so that the reader always waits for it (d_j = g_j, TBT_j = x_j); a stream that cannot
// clamp beside it keeps the pace and is not played.  Every token's interval goes to a sum, a maximum and a window of
// histogram bins.
//
// Bound: integer issue (a hash, a range map and a bin per token and stream).  A warp plays a request, a lane every 32nd
// token.  Every lane counts in counters of its own, [bin][lane] in shared memory: no atomics and no bank conflicts, where
// 32 lanes would meet in the few bins of a stream; two requests share a counter's halves before the lanes' counts are
// added up (a lane a bin, four counters at a time, lane b starting with the (b mod 8)th four: again without conflicts) and
// written as rows of 16-bit counts.  The stream after a hand-off stores no window: it is the target's without token 2,
// which the reductions take away (x_stream in disco_internal.cuh).  200,000 requests of 200 tokens, two streams: 204 us
// with one window a warp and atomics, 146 us with all three windows stored.
#include <algorithm>

#include "disco_internal.cuh"

namespace disco {

namespace {

constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr int kFreeWarps = 8;
constexpr int kFreeBatch = 8;             // requests a warp takes at a time

// Where a stream's window of counters starts for this lane, and the bin in front of it.
struct Counters { uint32_t* at; int lo, W; };

// One interval of x ticks more.  SMALL: intervals below 32 ticks occur, which have bins of their own (bin_of_ticks).
template <bool SMALL>
__device__ __forceinline__ void count_in(const Counters& c, uint32_t x, uint32_t inc) {
    const int b = (SMALL ? bin_of_ticks(x) : (int)(__float_as_uint(__uint2float_rz(x)) >> 18) - ((127 + 4) << 5)) - c.lo;
    if (DBG_OK(b, c.W, DBG_K_PLAYOUT, DBG_WINDOW)) c.at[b * 32] += inc;
}

// BOTH: pacing is off, both streams are played and a hand-off may follow the first token.  Otherwise pacing is on, a
// stream or two clamp at every token and no buffer fills: each is played for itself.  (Kernels of their own: in one
// kernel for all cases the warps waited for instructions four cycles of every ten.)
template <bool BOTH, bool SMALL>
__global__ void __launch_bounds__(kFreeWarps * 32, 4)
k_playout_free(TraceDev tr, const GroupConst* __restrict__ gcs, const __grid_constant__ ClassConst cc,
               const int32_t* __restrict__ knots, uint32_t k0, TimelineRec rec, const __grid_constant__ FreeMore more, bool early) {
    extern __shared__ __align__(16) uint32_t s_win[];         // per warp: [W0 + W1][32] counters
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, warps = blockDim.x >> 5;
    grid_dependency_wait();
    if (early) let_next_start();
    const int W0 = cc.W[0], W1 = cc.W[1], WW = W0 + W1;
    uint32_t* win = s_win + wib * (WW * 32);
    for (int b = lane; b < WW * 32; b += 32) win[b] = 0;
    __syncwarp();
    for (uint32_t batch = blockIdx.x * warps + wib;; batch += gridDim.x * warps) {
        int g;
        uint32_t k_lo, n_here;
        if (!batch_of_kind(tr, cc, G_FREE, kFreeBatch, batch, g, k_lo, n_here)) break;
        const GroupConst& gc = gcs[g];
        const uint32_t mul0 = 2u * (uint32_t)gc.J_srv + 1u, mul1 = 2u * (uint32_t)gc.J_dev + 1u;
        const uint32_t base0 = (uint32_t)(gc.T_srv - gc.J_srv), base1 = (uint32_t)(gc.T_dev - gc.J_dev);   // x = base + ((h * mul) >> 32)
        const Counters ct0 = {win + lane, cc.lo[g][0], W0}, ct1 = {win + W0 * 32 + lane, cc.lo[g][1], W1};
        const bool on0 = BOTH || !(cc.even[g] & 1u), on1 = BOTH || !(cc.even[g] & 2u);
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
        // sums of the jitter u = (h * (2J + 1)) >> 32, its maxima from token 3 on, and token 2's
        uint32_t o_s0 = 0, o_s1 = 0, o_m0 = 0, o_m1 = 0, o_f0 = 0, o_f1 = 0;
        const int b_lo = on0 ? 0 : W0, b_hi = on1 ? WW : W0;      // the bins in use
        for (int r0 = 0; r0 < (int)n_here; r0 += 2) {
            const int pair = min(2, (int)n_here - r0);
#pragma unroll 1
            for (int half = 0; half < pair; ++half) {
                const int r = r0 + half;
                const uint32_t n = __shfl_sync(FULL, n_l, r), inc = half ? 65536u : 1u;
                uint32_t hin = __shfl_sync(FULL, key_l, r) + (2u + lane) * kHashTok;
                uint32_t s0 = 0, s1 = 0, m0 = 0, m1 = 0, f0 = 0, f1 = 0, j = 2u + lane;
                // one token: its interval in each stream that is played
                auto token = [&](uint32_t& u, uint32_t& v) {
                    const uint32_t h = mix32(hin);
                    hin += 32u * kHashTok;
                    if (BOTH || on0) { u = __umulhi(h, mul0); s0 += u; count_in<SMALL>(ct0, base0 + u, inc); }
                    if (BOTH || on1) { v = __umulhi(h, mul1); s1 += v; count_in<SMALL>(ct1, base1 + v, inc); }
                };
                if (j <= n) {
                    token(f0, f1);
                    if (lane != 0) { m0 = f0; m1 = f1; }          // (lane 0 had token 2)
#pragma unroll 2
                    for (j += 32u; j <= n; j += 32u) {
                        uint32_t u = 0, v = 0;
                        token(u, v);
                        if (BOTH || on0) m0 = max(m0, u);
                        if (BOTH || on1) m1 = max(m1, v);
                    }
                }
                if (BOTH || on0) { s0 = __reduce_add_sync(FULL, s0); m0 = __reduce_max_sync(FULL, m0); f0 = __shfl_sync(FULL, f0, 0); }
                if (BOTH || on1) { s1 = __reduce_add_sync(FULL, s1); m1 = __reduce_max_sync(FULL, m1); f1 = __shfl_sync(FULL, f1, 0); }
                if (lane == r) { o_s0 = s0; o_s1 = s1; o_m0 = m0; o_m1 = m1; o_f0 = f0; o_f1 = f1; }
            }
            __syncwarp();
            // the lanes' counts are added up and go out; the counters are cleared for the next pair
            const size_t k = k_lo + r0;
#pragma unroll 1
            for (int b = b_lo + lane; b < b_hi; b += 32) {
                uint4* row = reinterpret_cast<uint4*>(win + b * 32);
                uint32_t t = 0;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int at = (c + b) & 7;
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
            const uint32_t sum0 = on0 ? o_s0 + nI * base0 : nI * tau, sum1 = on1 ? o_s1 + nI * base1 : nI * tau;
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
                const uint32_t base = to_dev ? base1 : base0;
                sumX = M + (to_dev ? sum1 - o_f1 : sum0 - o_f0) - base;
                maxX = max(M, nI > 1u ? base + (to_dev ? o_m1 : o_m0) : 0u);
            }
            const uint32_t most0 = max(o_m0, o_f0) + base0, most1 = max(o_m1, o_f1) + base1;
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
    }
}

}  // namespace

DBG_TRANSLATION_UNIT()

cudaError_t launch_playout_free(const TraceDev& tr, const GroupConst* gc, const ClassConst& cc, const int32_t* knots, uint32_t k0, TimelineRec rec, const FreeMore& more, uint32_t batches, bool early, int sms,
                                cudaStream_t st) {
    // as many warps to a block as the windows leave room for (wide jitter: up to 114 KB of counters a stream and warp)
    const size_t per_warp = (size_t)(cc.W[0] + cc.W[1]) * 32 * 4;
    const uint32_t warps = std::max<uint32_t>(1u, std::min<uint32_t>(kFreeWarps, (uint32_t)(100 * 1024 / per_warp)));
    const size_t smem = per_warp * warps;
    bool small = false;                                       // intervals below 32 ticks occur
    for (int g = 0; g < tr.n_groups; ++g) small = small || cc.lo[g][0] < 32 || cc.lo[g][1] < 32;
    auto* kernel = cc.pacing ? (small ? k_playout_free<false, true> : k_playout_free<false, false>)
                                  : (small ? k_playout_free<true, true> : k_playout_free<true, false>);
    cudaError_t e;
    if ((e = allow_smem((const void*)kernel, 227 * 1024))) return e;
    // (batches counts 32 requests each; four blocks of eight warps fit a multiprocessor)
    const uint32_t blocks = std::min<uint32_t>((batches * (32 / kFreeBatch) + warps - 1) / warps, (uint32_t)sms * 4u * kFreeWarps / warps);
    return launch_after(kernel, blocks, warps * 32, smem, st, tr, gc, cc, knots, k0, rec, more, early);
}

}  // namespace disco
