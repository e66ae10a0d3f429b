// Decode play-out (Sec. 4.3) of the groups whose streams cannot clamp (G_EXACT): both endpoints generate every token no
// slower than it is consumed (c_j = tau - x_j >= 0 for all j), so delivery is exactly tau-paced and
//  * every TBT of the streams S and D equals tau;
//  * the hand-off index m (buffer holds B tokens: d_{j-B+1} > g_j) is the first j whose prefix sum of c on the
//    candidate stream exceeds (B-1) tau;
//  * on stream X token m+1 waits for the hand-off latency M; it is `need` = M - e_m - tau late if that is positive,
//    and each later token of the target stream gains its c_j until the lag is made up.
// No token of the candidate after m and none of the target after the lag is made up can change a result, so none is
// drawn: a request costs the few tokens that fill the buffer.  Bound: integer issue.  k_playout_short: a thread per
// request; k_playout_fast: where the search may be long, a warp shares its lanes among four or eight requests by the
// tokens each may need.
#include <algorithm>

#include "disco_internal.cuh"

namespace disco {

namespace {

constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr int kFastWarps = 8;

struct LaneGroup {                       // constants of a lane's current request group
    uint32_t mulS, mulD;
    int32_t cS_base, cD_base, kappa, c0;
    int cand;
    const int32_t* K;
};

// Inclusive prefix sum over the lanes of a team (q = lane's position in its team); all 32 lanes call it.
__device__ __forceinline__ int32_t team_inclusive_sum(int32_t v, int q) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int32_t p = __shfl_up_sync(FULL, v, off);
        if (q >= off) v += p;
    }
    return v;
}

// Walks the lane's own tokens, adding c = base - ((h * mul) >> 32) to `run`, and stops at the first token where run
// exceeds `limit`.  Returns the number of tokens passed before that one.
__device__ __forceinline__ uint32_t walk(uint32_t key, uint32_t j0, int cnt, int32_t base, uint32_t mul, int32_t limit,
                                         int32_t& run) {
    uint32_t passed = 0;
    uint32_t hin = key + j0 * kHashTok;
    for (int t = 0; t < cnt; ++t) {
        run += base - (int32_t)__umulhi(mix32(hin), mul);
        hin += kHashTok;
        if (run > limit) break;
        ++passed;
    }
    return passed;
}


// rpw = requests per ticket (8, 16 or 32): small traces use small batches so that enough warps are in flight.
template <int PER>
__global__ void __launch_bounds__(kFastWarps * 32)
k_playout_fast(TraceDev tr, const GroupConst* __restrict__ gcs, const __grid_constant__ ClassConst cc,
               const int32_t* __restrict__ knots, uint32_t k0, TimelineRec rec, uint32_t* __restrict__ tickets, int rpw,
               uint32_t one, bool early) {
    const int lane = threadIdx.x & 31;
    grid_dependency_wait();
    if (early) let_next_start();
    const int32_t tau = cc.tau;                                   // pacing is on for every launch of this kernel
    const uint32_t B = (uint32_t)cc.B;
    const long long thr64 = (long long)(B ? B - 1 : 0) * tau;
    const int32_t thr = thr64 > 0x7FFFFFFFLL ? 0x7FFFFFFF : (int32_t)thr64;
    const bool mig_any = cc.mig_any != 0;

    LaneGroup G;
    int cur_g = -1;
    // Batches of rpw requests are handed out by a ticket counter (zero at launch), so a warp that drew short
    // requests takes more of them and the last batches are spread over the whole GPU.
    for (;;) {
        uint32_t ticket = 0;
        if (lane == 0) ticket = atomicAdd(tickets, 1u);
        const uint32_t batch0 = __shfl_sync(FULL, ticket, 0) * (uint32_t)rpw;
        if (batch0 >= tr.n) break;
        // ---- one request per lane: inputs
        const uint32_t kk = batch0 + lane;
        bool live = lane < rpw && kk < tr.n;
        uint32_t n_l = 1, l_l = 1, key_l = 0, nI_l = 0;          // nI_l: tokens to draw
        int g_l = 0;
        if (live) {
            const uint4 q = tr.req[kk];
            while (g_l + 1 < tr.n_groups && kk >= tr.grp_off[g_l + 1]) ++g_l;
            live = cc.kind[g_l] == G_EXACT;
            if (live) {
                n_l = q.y >> 16; l_l = q.y & 0xFFFFu;
                key_l = mix32(k0 + q.z * kHashReq);
                nI_l = min(n_l - 1, cc.search[g_l]);
            }
        }
        // ---- one request per lane: results (bits 0-15 m, 16-31 late tokens)
        uint32_t o_md = 0, o_stall = 0;

        for (int it = 0; it < rpw / PER; ++it) {
            // ---- share the lanes among the PER requests: one lane for each request that has intervals, the
            //      other lanes in proportion to the intervals (n - 1 each).  Any split that gives such a request
            //      a lane is valid; the rounding only moves load.  Every group of PER lanes holds the same
            //      PER values here, lane s of a group standing for request r0 + s.
            const int r0 = it * PER, s8 = lane & (PER - 1);
            const uint32_t nI_s = __shfl_sync(FULL, nI_l, r0 + s8);
            uint32_t inc = nI_s;
#pragma unroll
            for (int off = 1; off < PER; off <<= 1) {
                const uint32_t up = __shfl_up_sync(FULL, inc, off, PER);
                if (s8 >= off) inc += up;
            }
            const uint32_t tot = __shfl_sync(FULL, inc, PER - 1, PER);
            const uint32_t busy = __ballot_sync(FULL, nI_s != 0) & ((1u << PER) - 1u);   // requests with intervals
            const float per = __fdividef((float)(32 - __popc(busy)), (float)max(tot, 1u));
            // first lane of request s: requests with intervals before it, plus its share of the spare lanes
            const int start_s = __popc(busy & ((1u << s8) - 1u)) + __float2int_rn((float)(inc - nI_s) * per);
            const bool owner_s = lane < PER && nI_s != 0;
            const uint32_t starts = __reduce_or_sync(FULL, owner_s ? 1u << start_s : 0u);   // bit 0 is set unless tot == 0
            // request of the k-th team (teams in request order), four bits each
            const uint32_t team_req = __reduce_or_sync(FULL, owner_s ? (uint32_t)s8 << (4 * __popc(busy & ((1u << s8) - 1u))) : 0u);
            const uint32_t upto = starts & (0xFFFFFFFFu >> (31 - lane));           // team starts at or below this lane
            const uint32_t after = starts & ~(0xFFFFFFFFu >> (31 - lane));
            const int a = upto ? 31 - __clz(upto) : 0;
            const int a_next = after ? __ffs(after) - 1 : 32;
            const int lanes = a_next - a, q = lane - a;
            const uint32_t tmask = lanes == 32 ? FULL : (((1u << lanes) - 1u) << a);   // this team's lanes: teams may diverge
            const int r = r0 + (int)((team_req >> (4 * max(__popc(upto) - 1, 0))) & 7u);
            const uint32_t n = __shfl_sync(FULL, n_l, r), l = __shfl_sync(FULL, l_l, r);
            const uint32_t key = __shfl_sync(FULL, key_l, r);
            const int g = __shfl_sync(FULL, g_l, r);
            if (g != cur_g && DBG_OK(g, tr.n_groups, DBG_K_PLAYOUT_FAST, DBG_GROUP)) {
                cur_g = g;
                const GroupConst& gc = gcs[g];
                G.mulS = 2u * (uint32_t)gc.J_srv + 1u; G.mulD = 2u * (uint32_t)gc.J_dev + 1u;
                G.cS_base = tau - (gc.T_srv - gc.J_srv); G.cD_base = tau - (gc.T_dev - gc.J_dev);
                G.kappa = gc.kappa; G.c0 = gc.c0;
                G.cand = mig_any ? gc.candidate : 0;
                G.K = knots + g * kNKnots;
            }
            const uint32_t nI_r = __shfl_sync(FULL, nI_l, r);
            const uint32_t nI = tot ? nI_r : 0u;                       // tokens to draw, from token 2 on
            // tokens per lane, ceil(nI / lanes) or one more (lanes >= 1 here); all that matters is lanes * L >= nI
            uint32_t L = __float2uint_ru(__fdividef((float)nI, (float)lanes));
            if (L * (uint32_t)lanes < nI) ++L;
            const uint32_t lo = (uint32_t)q * L;
            const int cnt = lo >= nI ? 0 : (int)min(L, nI - lo);
            const uint32_t j0 = lo + 2;

            // ---- every token up to the longest search: hash draw and jitter of the endpoint that may hand over
            const int Lmax = (int)__reduce_max_sync(FULL, L);
            uint32_t hin = key + j0 * kHashTok;
            const uint32_t mulC = G.cand == 2 ? G.mulD : G.mulS, mulT = G.cand == 2 ? G.mulS : G.mulD;
            const int32_t cC_base = G.cand == 2 ? G.cD_base : G.cS_base, cT_base = G.cand == 2 ? G.cS_base : G.cD_base;
            uint32_t hC = 0;
#pragma unroll 4
            for (int t = 0; t < Lmax; ++t) {
                const uint32_t x = __umulhi(mix32(hin), mulC);
                hin += kHashTok;
                if (t < cnt) hC = x * one + hC;            // `one` = 1: a multiply-add, off the busy integer pipe
            }
            const int32_t sC = cnt * cC_base - (int32_t)hC;
            const bool go = nI != 0;
            // ---- hand-off index on the candidate stream
            const int cand = go ? G.cand : 0;
            const int32_t inC = team_inclusive_sum(sC, q);
            uint32_t m = 0;
            int32_t e_m = 0;
            if (cand && B == 0) m = 1;                                 // nothing to fill: hand off after token 1
            const uint32_t crossers = __ballot_sync(FULL, cand && B != 0 && inC > thr) & tmask;
            if (crossers) {                                            // team-uniform from here on
                const int owner = __ffs(crossers) - 1;                 // first lane whose run takes the sum past thr
                uint32_t j_found = 0;
                int32_t run = inC - sC;
                if (lane == owner) j_found = j0 + walk(key, j0, cnt, cC_base, mulC, thr, run);   // (the run's total exceeds thr)
                j_found = __shfl_sync(tmask, j_found, owner);
                e_m = __shfl_sync(tmask, run, owner);                  // clean stream: e_m = S_m
                m = j_found + 1 <= n ? j_found : 0u;                   // the hand-off needs a token left to generate
            }
            // ---- stream X
            uint32_t stall = 0, delayed = 0;
            int32_t need = 0;                                          // how late token m+1 is, if it stalls
            if (m) {                                                   // team-uniform
                uint32_t M;
                if (cand == 1) M = (uint32_t)G.kappa * (l + m) + (uint32_t)G.c0;       // device re-prefills prompt + m tokens
                else {
                    const uint32_t u = mix32(key);                     // a server TTFT drawn from F by its knots
                    const uint32_t ki = u >> 24, fr = (u >> 8) & 0xFFFFu;
                    M = 0;
                    if (DBG_OK(ki + 1, kNKnots, DBG_K_PLAYOUT_FAST, DBG_KNOT))
                        M = (uint32_t)(G.K[ki] + (int32_t)(((int64_t)(G.K[ki + 1] - G.K[ki]) * (int64_t)fr) >> 16));
                }
                const int32_t v = e_m + (tau - (int32_t)M);            // slot lag of token m+1, negated
                stall = (uint32_t)tau + (uint32_t)max(-v, 0);
                need = max(-v, 0);
            }
            {
                // tokens m+2.. stay late while the target's prefix sum of c (from token m+2) is below the lag.  The
                // team draws `lanes` tokens of the target stream a round until the sum gets there (c >= 0: the
                // late tokens are a prefix).  All 32 lanes run the rounds; teams that are done draw nothing.
                bool more = need > 0 && m + 2 <= n;
                uint32_t jb = m + 2, late = 0;
                int32_t carry = 0;
                while (__any_sync(FULL, more)) {
                    const uint32_t j = jb + (uint32_t)q;
                    const bool in = more && j <= n;
                    const int32_t c = in ? cT_base - (int32_t)__umulhi(mix32(key + j * kHashTok), mulT) : 0;
                    const int32_t R = carry + team_inclusive_sum(c, q);
                    late += __popc(__ballot_sync(FULL, in && R < need) & tmask);
                    const bool reached = (__ballot_sync(FULL, in && R >= need) & tmask) != 0;
                    carry = __shfl_sync(FULL, R, a + lanes - 1);
                    jb += (uint32_t)lanes;
                    more = more && !reached && jb <= n;
                }
                if (need > 0) delayed = 1u + late;
            }
            // ---- hand the results to the lanes that own the requests' slots
            const uint32_t packed = m | (delayed << 16);
            const uint32_t got_md = __shfl_sync(FULL, packed, start_s & 31), got_stall = __shfl_sync(FULL, stall, start_s & 31);
            if (lane / PER == it) {
                const bool has_lanes = nI_s != 0;                      // no lanes: a single-token request, all zeros
                o_md = has_lanes ? got_md : 0u;
                o_stall = has_lanes ? got_stall : 0u;
            }
        }
        __syncwarp();
        // ---- one request per lane: results out
        if (live && DBG_OK(kk, tr.n, DBG_K_PLAYOUT_FAST, DBG_REQUEST)) rec.hand[kk] = make_uint2(o_md, o_stall);
    }
}

// Buffers that fill within a few tokens (no group's search looks at more than kShortSearch of them).  A thread plays a
// request up to the hand-off: the lanes of a warp hold requests whose searches take about the same number of tokens;
// beyond some 64 tokens the longest of 32 requests would keep the others waiting.  The lag after a hand-off is another
// matter: a few requests in ten have one, and where the server takes over it is as widely spread as its TTFT.  Those
// requests are therefore collected in shared memory first.  A thread each, in full warps, draws the first tokens of a lag;
// what is left of the longer ones is made up by a warp each, 32 tokens at a time, so that the longest (thousands of
// tokens) does not hold the block for as many dependent steps.  A thread draws 32 tokens, or 256 where most of the block's
// requests have longer lags (prompts that take a device long to read: those lags are alike).  (Without the collection:
// 513 us for the 16 M requests of three server profiles and two devices, 43 us for 250,000 of them; with it 304 and 12, and
// 248 and 10 with the tokens that can neither fill the buffer nor make up the lag drawn without a test each; 4 M requests of long
// outputs on a slow device 97 us, now 60, most of it because the blocks with the longest lags come first.)  Of those 248 us the lags took
// 100, since a warp draws as long as the longest of its 32: put in order by their lengths first they take 50 (4 M in six groups 66 us ->
// 54).  That pays where they are lags behind a server's TTFT; a device's, 4 M requests in one group, take 60 us as they come and 64
// put in order.
constexpr uint32_t kShortSearch = 64;
constexpr int kShortThreads = 256;
constexpr int kShortPer = 4;             // requests a thread may play

struct ShortGroup {                      // a group under the class
    uint32_t mulC, mulT;                 // candidate's and target's jitter ranges
    int32_t cC, cT;                      // c = base - ((h * mul) >> 32)
    uint32_t kappa, c0;
    int cand;
    uint32_t end;                        // where the group's requests end
    int exact;                           // played here
    int32_t cT_mean;
    uint32_t sure;                       // tokens that cannot fill the buffer, whatever their jitter
    // so many tokens are late for sure, each making up cT at most (the quotient is rounded down by more than its error)
    __device__ uint32_t sure_late(int32_t need) const { return (uint32_t)(__fdividef((float)(need - 1), (float)max(cT, 1)) * 0.99999f); }
};

// The lags of a block are put in order by what they take at least, in 64 steps: a token each, and from 32 on eight.
constexpr int kLagLengths = 64;
__device__ __forceinline__ uint32_t lag_length(uint32_t tokens) { return tokens < 32u ? tokens : min(28u + tokens / 8u, (uint32_t)kLagLengths - 1u); }

// (h * mul) >> 32 of so many tokens behind hin, added up: no test a token, so that several are under way at once.
__device__ __forceinline__ uint32_t sum_jitter(uint32_t& hin, uint32_t count, uint32_t mul) {
    uint32_t sum = 0;
#pragma unroll 4
    for (uint32_t t = 0; t < count; ++t) { hin += kHashTok; sum = mad_hi(mix32(hin), mul, sum); }
    return sum;
}

// MANY: several classes, a row of blocks each (250,000 requests under five paces one after another 42 us; the last four together 23, and 8 for the first).
template <bool MANY>
__global__ void __launch_bounds__(kShortThreads)
k_playout_short(TraceDev tr, const GroupConst* __restrict__ gcs, const __grid_constant__ ClassConst given,
                const int32_t* __restrict__ knots, uint32_t k0, TimelineRec rec, int per, bool early, const __grid_constant__ ShortMany many) {
    const ClassConst& cc = MANY ? many.classes[many.cls[blockIdx.y]] : given;
    if (MANY) rec.hand = reinterpret_cast<uint2*>(reinterpret_cast<char*>(rec.hand) + many.slot[blockIdx.y] * many.rec_stride);
    __shared__ ShortGroup groups[kMaxGroups];
    __shared__ uint4 lag[kShortThreads * kShortPer];         // hash key, lag, output length | hand-off << 16, place | group << 16
    __shared__ uint16_t rest[kShortThreads * kShortPer];     // the lags by their lengths, then those that a thread has not made up
    __shared__ int of_length[kLagLengths];                   // how many, then where they start
    __shared__ int n_lag, n_long, n_rest;
    grid_dependency_wait();
    if (early) let_next_start();
    const int32_t tau = cc.tau;
    const uint32_t B = (uint32_t)cc.B;
    const long long thr64 = (long long)(B ? B - 1 : 0) * tau;
    const int32_t thr = thr64 > 0x7FFFFFFFLL ? 0x7FFFFFFF : (int32_t)thr64;
    if (threadIdx.x == 0) { n_lag = 0; n_long = 0; n_rest = 0; }
    if (threadIdx.x < kLagLengths) of_length[threadIdx.x] = 0;
    for (int g = threadIdx.x; g < tr.n_groups; g += kShortThreads) {
        const GroupConst& gc = gcs[g];
        ShortGroup G;
        G.cand = cc.mig_any ? gc.candidate : 0;
        const uint32_t mulS = 2u * (uint32_t)gc.J_srv + 1u, mulD = 2u * (uint32_t)gc.J_dev + 1u;
        const int32_t cS = tau - (gc.T_srv - gc.J_srv), cD = tau - (gc.T_dev - gc.J_dev);
        G.mulC = G.cand == 2 ? mulD : mulS; G.mulT = G.cand == 2 ? mulS : mulD;
        G.cC = G.cand == 2 ? cD : cS; G.cT = G.cand == 2 ? cS : cD;
        G.kappa = (uint32_t)gc.kappa; G.c0 = (uint32_t)gc.c0;
        G.end = tr.grp_off[g + 1];
        G.exact = cc.kind[g] == G_EXACT;
        G.cT_mean = G.cT - (int32_t)(G.mulT >> 1);
        G.sure = G.cC > 0 ? (uint32_t)(thr / G.cC) : (uint32_t)kMaxOutput;     // (a token adds at most cC)
        groups[g] = G;
    }
    __syncthreads();
    // (the last blocks first: lags of a device that reads slowly grow with the prompt, and the requests are stored by it)
    const uint32_t first = (gridDim.x - 1u - blockIdx.x) * (uint32_t)(kShortThreads * per);
    int g = 0;
    while (g + 1 < tr.n_groups && first >= groups[g].end) ++g;
    for (int k = 0; k < per; ++k) {
        const uint32_t kk = first + k * kShortThreads + threadIdx.x;
        if (kk >= tr.n) break;
        while (g + 1 < tr.n_groups && kk >= groups[g].end) ++g;
        const ShortGroup& G = groups[g];
        if (!G.exact) continue;
        const uint4 q = tr.req[kk];
        const uint32_t n = q.y >> 16, l = q.y & 0xFFFFu;
        uint32_t m = 0, stall = 0;
        if (G.cand != 0 && n > 1) {
            const uint32_t key = mix32(k0 + q.z * kHashReq);
            int32_t e_m = 0;
            if (B == 0) m = 1;                                         // nothing to fill: hand off after token 1
            else {
                uint32_t hin = key + kHashTok;
                const uint32_t sure = min(G.sure, n - 2u);
                e_m = (int32_t)(sure * (uint32_t)G.cC - sum_jitter(hin, sure, G.mulC));
                for (uint32_t j = 2 + sure; j < n; ++j) {              // (the hand-off needs a token left to generate)
                    hin += kHashTok;
                    e_m += G.cC - (int32_t)__umulhi(mix32(hin), G.mulC);
                    if (e_m > thr) { m = j; break; }
                }
            }
            if (m) {
                uint32_t M;
                if (G.cand == 1) M = G.kappa * (l + m) + G.c0;         // device re-prefills prompt + m tokens
                else {
                    const uint32_t u = mix32(key);                     // a server TTFT drawn from F by its knots
                    const uint32_t ki = u >> 24, fr = (u >> 8) & 0xFFFFu;
                    const int32_t* K = knots + g * kNKnots;
                    M = 0;
                    if (DBG_OK(ki + 1, kNKnots, DBG_K_PLAYOUT_FAST, DBG_KNOT))
                        M = (uint32_t)(K[ki] + (int32_t)(((int64_t)(K[ki + 1] - K[ki]) * (int64_t)fr) >> 16));
                }
                const int32_t need = -(e_m + (tau - (int32_t)M));      // how late token m+1 is
                stall = (uint32_t)tau + (uint32_t)max(need, 0);
                if (need > 0) {
                    if (n - m > 33u && (need >> 5) > G.cT_mean) atomicAdd(&n_long, 1);
                    const int at = atomicAdd(&n_lag, 1);
                    if (DBG_OK(at, kShortThreads * kShortPer, DBG_K_PLAYOUT_FAST, DBG_SLOT))
                        lag[at] = make_uint4(key, (uint32_t)need, n | m << 16, (uint32_t)(k * kShortThreads) + threadIdx.x | (uint32_t)g << 16);
                }
            }
        }
        rec.hand[kk] = make_uint2(m, stall);
    }
    __syncthreads();
    const uint32_t most = n_long > kShortThreads / 4 ? 256u : 32u;
    // ---- many lags as widely spread as the server's TTFT: by their lengths, the longest first, so that the lanes of a warp have about
    //      the same to draw (a device's are alike among neighbours)
    uint64_t mine = 0;                                         // the thread's lags, 16 bits each; in order of place unless they are sorted
#pragma unroll
    for (int k = 0; k < kShortPer; ++k) mine |= (uint64_t)(k * kShortThreads + threadIdx.x) << (16 * k);
    static_assert(kShortPer <= 4, "16 bits each");
    if (n_lag > kShortThreads / 2 && groups[lag[0].w >> 16].cand == 2) {
        uint32_t at[kShortPer];                                    // length | rank << 8
#pragma unroll
        for (int k = 0; k < kShortPer; ++k) {
            const int i = k * kShortThreads + threadIdx.x;
            if (i >= n_lag) break;
            const uint4 x = lag[i];
            const uint32_t length = lag_length(min((x.z & 0xFFFFu) - (x.z >> 16), groups[x.w >> 16].sure_late((int32_t)x.y)));
            at[k] = length | (uint32_t)atomicAdd(&of_length[length], 1) << 8;
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            static_assert(kLagLengths == 64, "two a lane");
            const int a = of_length[63 - 2 * threadIdx.x], b = of_length[62 - 2 * threadIdx.x];
            const int before = team_inclusive_sum(a + b, threadIdx.x) - a - b;
            of_length[63 - 2 * threadIdx.x] = before; of_length[62 - 2 * threadIdx.x] = before + a;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kShortPer; ++k) {
            const int i = k * kShortThreads + threadIdx.x;
            if (i >= n_lag) break;
            const int to = of_length[at[k] & 255u] + (int)(at[k] >> 8);
            if (DBG_OK(to, kShortThreads * kShortPer, DBG_K_PLAYOUT_FAST, DBG_SLOT)) rest[to] = (uint16_t)i;
        }
        __syncthreads();
        mine = 0;
#pragma unroll
        for (int k = 0; k < kShortPer; ++k) mine |= (uint64_t)rest[k * kShortThreads + threadIdx.x] << (16 * k);     // (those behind the last are not used)
        __syncthreads();
    }
    // ---- tokens m+2.. stay late while the target's sum of c from there on is below the lag (c >= 0: a prefix)
    for (int j0 = threadIdx.x; j0 < n_lag; j0 += kShortThreads, mine >>= 16) {
        const int i = (int)(mine & 0xFFFFu);
        const uint4 x = lag[i];
        const ShortGroup& G = groups[x.w >> 16];
        const int32_t need = (int32_t)x.y, cT = G.cT;
        const uint32_t n = x.z & 0xFFFFu, m = x.z >> 16, mulT = G.mulT, end = min(n, m + 1 + most);
        uint32_t j = m + 2, hin = x.x + (m + 1) * kHashTok;
        const uint32_t sure = min(end + 1u - j, G.sure_late(need));
        int32_t run = (int32_t)(sure * (uint32_t)cT - sum_jitter(hin, sure, mulT));
        j += sure;
        for (hin += kHashTok; j <= end; ++j, hin += kHashTok) {
            run += cT - (int32_t)__umulhi(mix32(hin), mulT);
            if (run >= need) break;
        }
        if (run < need && j <= n) { lag[i].y = (uint32_t)(need - run); rest[atomicAdd(&n_rest, 1)] = (uint16_t)i; continue; }
        rec.hand[first + (x.w & 0xFFFFu)].x = m | (j - m - 1) << 16;             // tokens m+1 .. j-1 are late
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < n_rest; i += kShortThreads / 32) {
        const uint4 x = lag[rest[i]];
        const ShortGroup& G = groups[x.w >> 16];
        const int32_t need = (int32_t)x.y, cT = G.cT;
        const uint32_t n = x.z & 0xFFFFu, m = x.z >> 16, mulT = G.mulT;
        int32_t run = 0;
        uint32_t jb = m + 2 + most;
        for (; jb <= n; jb += 32) {
            const uint32_t j = jb + lane;
            const int32_t c = j <= n ? cT - (int32_t)__umulhi(mix32(x.x + j * kHashTok), mulT) : 0;
            const int32_t all = __reduce_add_sync(FULL, c);
            if (run + all >= need) {
                const int32_t R = run + team_inclusive_sum(c, lane);
                jb += __popc(__ballot_sync(FULL, R < need && j <= n));
                break;
            }
            run += all;
        }
        if (lane == 0) rec.hand[first + (x.w & 0xFFFFu)].x = m | (min(jb, n + 1) - m - 1) << 16;
    }
}

}  // namespace

DBG_TRANSLATION_UNIT()

// four requests a thread (fuller warps of lags) once that leaves several blocks to every multiprocessor
static int short_per(uint32_t n, int sms) { return n >= (uint32_t)sms * 8u * kShortThreads * kShortPer ? kShortPer : 1; }

bool short_search(uint32_t search) { return search <= kShortSearch; }

cudaError_t launch_playout_many(const TraceDev& tr, const GroupConst* gc, const int32_t* knots, uint32_t k0, TimelineRec rec, const ShortMany& many, bool early, int sms,
                                cudaStream_t st) {
    const int per = short_per(tr.n, sms);
    const uint32_t per_block = (uint32_t)(kShortThreads * per);
    return launch_after(k_playout_short<true>, dim3((tr.n + per_block - 1) / per_block, many.count), kShortThreads, 0, st, tr, gc, ClassConst{}, knots, k0,
                        rec, per, early, many);
}

cudaError_t launch_playout_exact(const TraceDev& tr, const GroupConst* gc, const ClassConst& cc, const int32_t* knots,
                                 uint32_t k0, TimelineRec rec, uint32_t* ticket, uint32_t search, bool long_outputs, bool early, int sms,
                                 cudaStream_t st) {
    if (short_search(search)) {
        const int per = short_per(tr.n, sms);
        const uint32_t per_block = (uint32_t)(kShortThreads * per);
        return launch_after(k_playout_short<false>, (tr.n + per_block - 1) / per_block, kShortThreads, 0, st, tr, gc, cc, knots, k0, rec, per, early, ShortMany{});
    }
    // requests per ticket: small batches spread the end of the launch evenly; large traces amortise the ticket
    int rpw = 8;
    while (rpw < 32 && (uint64_t)tr.n / (2 * rpw) >= (uint64_t)sms * 48u * 4u) rpw *= 2;
    const uint32_t per_block = kFastWarps * (uint32_t)rpw;
    // requests per round: eight halve the cost of a round per request; with long outputs the token loop is
    // what counts, and four requests split the lanes more evenly
    cudaError_t e = cudaMemsetAsync(ticket, 0, 4, st);
    if (e) return e;
    auto* kernel = long_outputs ? k_playout_fast<4> : k_playout_fast<8>;
    // as many blocks as the GPU holds at once (at most six of these per SM); the ticket counter feeds them
    const uint32_t blocks = std::min<uint32_t>((tr.n + per_block - 1) / per_block, (uint32_t)sms * 6u);
    return launch_after(kernel, blocks, kFastWarps * 32, 0, st, tr, gc, cc, knots, k0, rec, ticket, rpw, 1u, early);
}

}  // namespace disco
