// Decode play-out (Sec. 4.3) of the groups whose streams are delivered as they are generated (G_FREE): pacing is off, or
// every token takes at least tau, so that the reader always waits for it (d_j = g_j, TBT_j = x_j); a stream that cannot
// clamp beside it keeps the pace and is not played.  Every token's interval goes to a sum, a maximum and a window of
// histogram bins.
//
// Bound: integer issue (a hash, a range map and a bin per token and stream).  A warp plays a request, a lane every 32nd
// token; the windows are counted in shared memory of the warp's own (increments of one, which the hardware merges
// where lanes meet) and written once, as rows of 16-bit counts.  200,000 requests of 200 tokens, two streams:
// see the figure at launch_playout_free.
#include <algorithm>

#include "disco_internal.cuh"

namespace disco {

namespace {

constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr int kFreeWarps = 8;

struct FreeStream {                      // one stream of a group
    uint32_t mul;
    int32_t base;                        // x = base + ((h * mul) >> 32), base = T - J
    int lo, W;                           // its window of bins
    bool on;                             // played here (else it keeps the pace)
};

// One interval more in a window that starts at bin lo.
__device__ __forceinline__ void count_in(uint32_t* win, int lo, int W, uint32_t x, int32_t* err) {
    const int b = bin_of_ticks(x) - lo;
    if (b >= 0 && b < W) atomicAdd(&win[b], 1u); else atomicExch(&err[2], 1);
}

__global__ void __launch_bounds__(kFreeWarps * 32)
k_playout_free(TraceDev tr, const GroupConst* __restrict__ gcs, const ClassConst* __restrict__ ccp,
               const int32_t* __restrict__ knots, uint32_t k0, TimelineRec rec, int32_t* __restrict__ err) {
    extern __shared__ uint32_t s_win[];                       // [warps][W0 + W1]
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    grid_dependency_wait();
    const ClassConst& cc = *ccp;
    const int W0 = cc.W[0], W1 = cc.W[1], W2 = cc.W[2];
    uint32_t* win0 = s_win + wib * (W0 + W1);
    uint32_t* win1 = win0 + W0;
    for (int b = lane; b < W0 + W1; b += 32) win0[b] = 0;
    __syncwarp();
    const uint32_t tau = (uint32_t)cc.tau;
    for (uint32_t batch = blockIdx.x * kFreeWarps + wib;; batch += gridDim.x * kFreeWarps) {
        int g;
        uint32_t k_lo, n_here;
        if (!batch_of_kind(tr, cc, G_FREE, batch, g, k_lo, n_here)) break;
        const GroupConst& gc = gcs[g];
        FreeStream st[2];
        st[0].mul = 2u * (uint32_t)gc.J_srv + 1u; st[0].base = gc.T_srv - gc.J_srv; st[0].lo = cc.lo[g][0]; st[0].W = W0;
        st[1].mul = 2u * (uint32_t)gc.J_dev + 1u; st[1].base = gc.T_dev - gc.J_dev; st[1].lo = cc.lo[g][1]; st[1].W = W1;
        st[0].on = !(cc.even[g] & 1u); st[1].on = !(cc.even[g] & 2u);
        // without pacing the buffer is empty and the dearer winner hands over after its first token; with pacing such a
        // stream never fills a buffer
        const int cand = (cc.mig_any && !cc.pacing) ? gc.candidate : 0;
        const int tgt = cand == 1 ? 1 : 0;
        // ---- one request per lane: inputs, results
        uint32_t n_l = 1, l_l = 1, key_l = 0;
        if (lane < n_here) {
            const uint4 q = tr.req[k_lo + lane];
            n_l = q.y >> 16; l_l = q.y & 0xFFFFu;
            key_l = mix32(k0 + q.z * kHashReq);
        }
        uint32_t o_sum[3] = {0, 0, 0}, o_max[3] = {0, 0, 0}, o_m = 0, o_stall = 0;
        for (int r = 0; r < (int)n_here; ++r) {
            const uint32_t n = __shfl_sync(FULL, n_l, r), key = __shfl_sync(FULL, key_l, r), k = k_lo + r;
            uint32_t sum[2] = {0, 0}, most[2] = {0, 0}, first[2] = {0, 0}, most_later[2] = {0, 0};
            for (uint32_t j = 2 + lane; j <= n; j += 32) {
                const uint32_t h = mix32(key + j * kHashTok);
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    if (!st[s].on) continue;                  // (uniform over the batch)
                    const uint32_t x = (uint32_t)st[s].base + __umulhi(h, st[s].mul);
                    sum[s] += x;
                    if (j == 2) first[s] = x; else most_later[s] = max(most_later[s], x);
                    count_in(s ? win1 : win0, st[s].lo, st[s].W, x, err);
                }
            }
            __syncwarp();
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                if (!st[s].on) { sum[s] = (n - 1) * tau; most[s] = n > 1 ? tau : 0u; continue; }
                sum[s] = __reduce_add_sync(FULL, sum[s]);
                most_later[s] = __reduce_max_sync(FULL, most_later[s]);
                first[s] = __shfl_sync(FULL, first[s], 0);
                most[s] = max(first[s], most_later[s]);
            }
            uint32_t m = 0, M = 0, sumX = 0, maxX = 0;
            if (cand && n > 1) {                              // stream X: one token of the candidate, then the target
                m = 1;
                if (cand == 1) M = (uint32_t)gc.kappa * (__shfl_sync(FULL, l_l, r) + 1u) + (uint32_t)gc.c0;
                else {
                    const uint32_t u = mix32(key);            // a server TTFT drawn from F by its knots
                    const uint32_t ki = u >> 24, fr = (u >> 8) & 0xFFFFu;
                    const int32_t* K = knots + g * kNKnots;
                    if (DBG_OK(ki + 1, kNKnots, DBG_K_PLAYOUT, DBG_KNOT))
                        M = (uint32_t)(K[ki] + (int32_t)(((int64_t)(K[ki + 1] - K[ki]) * (int64_t)fr) >> 16));
                }
                sumX = M + (sum[tgt] - first[tgt]);
                maxX = max(M, most_later[tgt]);
                const int shift = cc.lo[g][2] - st[tgt].lo, skip = bin_of_ticks(first[tgt]) - st[tgt].lo;
                const uint32_t* wt = tgt ? win1 : win0;
                for (int b = lane; b < W2; b += 32) {
                    const int t = b + shift;
                    uint32_t v = (t >= 0 && t < st[tgt].W) ? wt[t] : 0u;
                    if (t == skip) --v;
                    rec.win[2][(size_t)k * W2 + b] = (uint16_t)v;
                }
                __syncwarp();
            }
            // the windows go out and are cleared for the next request
            if (st[0].on) for (int b = lane; b < W0; b += 32) { rec.win[0][(size_t)k * W0 + b] = (uint16_t)win0[b]; win0[b] = 0; }
            if (st[1].on) for (int b = lane; b < W1; b += 32) { rec.win[1][(size_t)k * W1 + b] = (uint16_t)win1[b]; win1[b] = 0; }
            __syncwarp();
            if (lane == r) {
                o_sum[0] = sum[0]; o_sum[1] = sum[1]; o_sum[2] = sumX; o_max[0] = most[0]; o_max[1] = most[1]; o_max[2] = maxX;
                o_m = m; o_stall = M;
            }
        }
        if (lane < n_here) {
            const uint32_t k = k_lo + lane;
            rec.hand[k] = make_uint2(o_m, o_stall);
#pragma unroll
            for (int s = 0; s < 3; ++s) { rec.sum[s][k] = o_sum[s]; rec.max[s][k] = o_max[s]; }
        }
        __syncwarp();
    }
}

}  // namespace

DBG_TRANSLATION_UNIT()

cudaError_t launch_playout_free(const TraceDev& tr, const GroupConst* gc, const ClassConst* cc, const ClassConst& host_cc,
                                const int32_t* knots, uint32_t k0, TimelineRec rec, int32_t* err, uint32_t batches, int sms,
                                cudaStream_t st) {
    const size_t smem = (size_t)kFreeWarps * (host_cc.W[0] + host_cc.W[1]) * 4;
    cudaError_t e;
    if (smem > 48 * 1024 &&
        (e = cudaFuncSetAttribute(k_playout_free, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    const uint32_t blocks = std::min<uint32_t>((batches + kFreeWarps - 1) / kFreeWarps, (uint32_t)sms * 32u);
    return launch_after(k_playout_free, blocks, kFreeWarps * 32, smem, st, tr, gc, cc, knots, k0, rec, err);
}

}  // namespace disco
