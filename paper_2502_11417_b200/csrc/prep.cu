// Policy preparation: Algorithms 1-3 for every (group, policy).
#include <algorithm>
#include <type_traits>

#include "load.cuh"
#include "scan.cuh"

namespace disco {

namespace {

constexpr uint32_t FULL = 0xFFFFFFFFu;

// ------------------------------------------------------------------------------------------------------
// Algorithms 1-3, one warp per (group, policy).  All fp64 steps use explicit round-to-nearest
// operations so that no multiply-add is contracted.  Bound: the latency of a dozen dependent loads.  (A thread per pair
// with fifteen probes a round took 10 us for one policy and 23 us where the lanes of a warp held groups of both kinds.)
// ------------------------------------------------------------------------------------------------------
__device__ int32_t inverse_cdf(const int32_t* sorted, uint32_t N, double q) {
    if (N == 0) return 0;
    double r = ceil(__dmul_rn(q, (double)N)) - 1.0;
    long long k = (long long)r;
    if (k < 0) k = 0;
    if (k > (long long)N - 1) k = (long long)N - 1;
    return DBG_OK(k, N, DBG_K_PREP, DBG_ELEMENT) ? sorted[k] : 0;
}

// Smallest x in [lo, hi) with pred(x), or hi if there is none; pred is false up to some point and true from
// there on.  The lanes probe 32 places a round: the search over the 4098 cumulative masses takes three rounds.
template <class F>
__device__ __forceinline__ int first_true(int lo, int hi, F pred) {
    const int lane = threadIdx.x & 31;
    while (hi > lo) {
        const int step = (hi - lo + 31) >> 5;                         // the last places of 32 pieces
        const int x = min(lo + (lane + 1) * step, hi) - 1;
        const uint32_t holds = __ballot_sync(FULL, pred(x));
        if (holds == 0u) return hi;
        const int k = __ffs(holds) - 1;                               // the answer lies in piece k
        hi = min(lo + (k + 1) * step, hi) - 1;                        // ... or is its last place
        lo += k * step;
        if (step == 1) return lo;
    }
    return lo;
}

//
// The policies and the other small tables come with the launch, as a parameter (up to kTablesInline bytes), or from the pinned
// memory the host laid them out in: a block reads its own policies, and all blocks bring a share of the tables to the device
// for the kernels behind, and write the chunks of requests out.  (A copy in front of this kernel stood between it and the play-out: 10 to 20 us from
// the play-out's end to this kernel's start, 1 to 6 of them the copy.  From pinned memory this kernel takes 10 us with 1,024
// policies, with a parameter 3 to 4.  Steps of 100,000 requests under 64 policies 154 -> 146 us, of 200,000 without pacing
// 207 -> 197, of 4 M long ones 354 -> 341.)  Nothing here depends on the play-out, and the play-out reads nothing that is written here, so the
// kernel runs beside it -- the load was waited for by the host, and a play-out lets this kernel start only behind its own
// wait for what came before -- and waits for it at its end, on behalf of the kernels behind both.
constexpr int kPrepThreads = 128, kPrepWarps = kPrepThreads / 32;

__device__ __forceinline__ void prep_pair(const PolicyIn& pi, const PolicyKind& pc, uint32_t p, int g, uint32_t P, const GroupConst* __restrict__ gc,
                                          const int64_t* __restrict__ cum_mass, const uint32_t* __restrict__ cnt,
                                          const int32_t* __restrict__ sorted, const uint32_t* __restrict__ grp_off,
                                          Prep* __restrict__ prep) {
    const int64_t* cum = cum_mass + (size_t)g * (kMaxPrompt + 2);     // cum[L] = sum_{l<L} l*cnt[l]
    const uint32_t* c = cnt + (size_t)g * (kMaxPrompt + 1);
    const uint32_t off = grp_off[g], N = grp_off[g + 1] - off;
    const int32_t* srt = sorted + off;
    const double b = (double)pi.budget, alpha = (double)pc.alpha;
    const double Total = (double)cum[kMaxPrompt + 1];

    Prep r;
    r.device_constrained = pc.mode == 1 ? 1 : pc.mode == 2 ? 0 : gc[g].auto_device_constrained;
    r.l_th = 0; r.l_star = 0; r.w_star = 0; r.w_tail = 0;
    r.theta = pi.theta;
    r.mig_on = (pc.flags & DISCO_FLAG_MIGRATION) ? 1 : 0;
    r.stochastic = (pc.flags & DISCO_FLAG_STOCHASTIC) ? 1 : 0;
    r.expected_len = pc.expected_len; r.route_thr = pi.route_thr; r.route_all = pi.budget >= 1.0f ? 1 : 0;
    r.beta_rule = 0;

    if (!r.device_constrained) {
        // Eq. 3: smallest L with device-only mass sum_{l<L} l cnt[l] >= (1-b) Total
        const double target = __dmul_rn(__dsub_rn(1.0, b), Total);
        r.l_th = first_true(0, kMaxPrompt + 1, [&](int L) {                                         // in [0, 4097]
            return DBG_OK(L, kMaxPrompt + 2, DBG_K_PREP, DBG_TABLE) ? (double)cum[L] >= target : true; });
    } else {
        // Algorithm 2, phase 1: tail protection
        const double q_tail = __dsub_rn(1.0, fmin(alpha, b));
        r.w_tail = inverse_cdf(srt, N, q_tail);
        if (pc.flags & DISCO_FLAG_BETA_RULE) {
            // Eq. 1-2 variant: the slope is found by k_prep_beta; until then every wait is w_tail
            r.beta_rule = 1;
            r.l_star = b <= alpha ? 0 : (int32_t)pc.l_immediate;
            r.w_star = r.w_tail + 1;
        } else if (b <= alpha) {
            r.l_star = 0; r.w_star = r.w_tail;
        } else {
            // phase 2: A input tokens may start the device at once; shortest prompts first
            const double A = __dmul_rn(__ddiv_rn(__dsub_rn(b, alpha), __dsub_rn(1.0, alpha)), Total);
            // first length whose cumulative mass exceeds A; 4097 = every class is funded
            const int lo = first_true(0, kMaxPrompt + 1, [&](int l) {
                return DBG_OK(l + 1, kMaxPrompt + 2, DBG_K_PREP, DBG_TABLE) ? (double)cum[l + 1] > A : true; });
            r.l_star = lo;
            if (lo <= kMaxPrompt && DBG_OK(lo, kMaxPrompt + 1, DBG_K_PREP, DBG_TABLE)) {
                const double f = __ddiv_rn(__dsub_rn(A, (double)cum[lo]), __dmul_rn((double)lo, (double)c[lo]));
                r.w_star = inverse_cdf(srt, N, __dmul_rn(__dsub_rn(1.0, alpha), __dsub_rn(1.0, f)));
            }
        }
    }
    if ((threadIdx.x & 31) == 0) prep[(size_t)g * P + p] = r;
}

template <int BYTES> struct Inline { uint4 v[BYTES / 16]; };
template <> struct Inline<0> { };

template <int BYTES>
__global__ void __launch_bounds__(kPrepThreads)
k_prep(uint32_t P, int G, const GroupConst* __restrict__ gc, const int64_t* __restrict__ cum_mass,
       const uint32_t* __restrict__ cnt, const int32_t* __restrict__ sorted, const uint32_t* __restrict__ grp_off,
       Prep* __restrict__ prep, const __grid_constant__ TablesIn in, uint4* __restrict__ clear, uint32_t clear_vecs,
       const __grid_constant__ Inline<BYTES> given) {
    constexpr uint32_t kVecs = sizeof(PolicyIn) / 16, kKindVecs = sizeof(PolicyKind) / 16, kNear = kPrepThreads / kKindVecs;
    static_assert(kChunkTables == 3, "three to write out");
    static_assert(sizeof(PolicyIn) % 16 == 0 && sizeof(PolicyKind) % 16 == 0 && kPrepWarps * kVecs <= kPrepThreads, "a vector a thread");
    __shared__ uint4 s_pol[kPrepWarps * kVecs], s_kind[kPrepThreads];     // the block's policies, and the first kinds
    __shared__ uint4 s_far[kPrepWarps * kKindVecs];                       // the warps' kinds that are not among these
    auto table = [&](uint32_t i) {
        if constexpr (BYTES != 0) return given.v[i];
        else return static_cast<const uint4*>(in.host)[i];
    };
    // pairs policy by policy, so that a block needs few of them
    const uint32_t pairs = P * (uint32_t)G, first = blockIdx.x * kPrepWarps, idx = first + (threadIdx.x >> 5), p0 = first / (uint32_t)G;
    const uint32_t mine = first < pairs ? (min(first + kPrepWarps, pairs) - 1u) / (uint32_t)G - p0 + 1u : 0u;
    const uint32_t at = blockIdx.x * kPrepThreads + threadIdx.x, all = gridDim.x * kPrepThreads, vec_at = in.skip + at;
    uint4 pol, kind, vec;
    const bool has_kind = mine != 0 && threadIdx.x < in.kinds * kKindVecs;
    if (threadIdx.x < mine * kVecs) pol = table(p0 * kVecs + threadIdx.x);
    if (has_kind) kind = table(P * kVecs + threadIdx.x);
    if (vec_at < in.vecs) vec = table(vec_at);
    // what the kernels behind this one must find zero
    for (uint32_t i = at; i < clear_vecs; i += all) clear[i] = make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x < mine * kVecs) s_pol[threadIdx.x] = pol;
    if (has_kind) s_kind[threadIdx.x] = kind;
    for (uint32_t i = vec_at; i < in.vecs; i += all) static_cast<uint4*>(in.device)[i] = i == vec_at ? vec : table(i);
    __syncthreads();
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, g = (int)(idx % (uint32_t)G);
    const uint32_t p = idx / (uint32_t)G;
    const bool own = idx < pairs && DBG_OK(g, G, DBG_K_PREP, DBG_GROUP) && DBG_OK(p - p0, kPrepWarps, DBG_K_PREP, DBG_POLICY) &&
                     DBG_OK(reinterpret_cast<const PolicyIn*>(s_pol)[p - p0].kind, in.kinds, DBG_K_PREP, DBG_TABLE);
    const PolicyKind* pk = nullptr;
    if (own) {
        const uint32_t k = reinterpret_cast<const PolicyIn*>(s_pol)[p - p0].kind;
        pk = reinterpret_cast<const PolicyKind*>(k < kNear ? s_kind + k * kKindVecs : s_far + wi * kKindVecs);
        if (k >= kNear && lane < (int)kKindVecs) s_far[wi * kKindVecs + lane] = table(P * kVecs + k * kKindVecs + lane);
        __syncwarp();
    }
    if constexpr (BYTES == 0) {
        // Behind the last of the block's reads: the host may write the memory anew, or give it back, once all blocks have been here.
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            if (atomicInc(in.left, gridDim.x - 1u) == gridDim.x - 1u) { __threadfence_system(); *in.read = in.turn; }
        }
    }
    if (own) prep_pair(reinterpret_cast<const PolicyIn*>(s_pol)[p - p0], *pk, p, g, P, gc, cum_mass, cnt, sorted, grp_off, prep);
    // (the last blocks first: the others have clearing and preparing to do)
    for (uint32_t i = (gridDim.x - 1u - blockIdx.x) * kPrepThreads + threadIdx.x; i < in.n_chunks[0] + in.n_chunks[1] + in.n_chunks[2]; i += all) {
        uint32_t k = i;
        int w = 0;
        while (w + 1 < kChunkTables && k >= in.n_chunks[w]) k -= in.n_chunks[w++];
        const uint32_t len = in.chunk_len[w];
        uint32_t x = 0;
        while (x + 1 < in.n_plan[w] && in.plan[w][x + 1].first <= k) ++x;
        const ChunkPlan& pl = in.plan[w][x];
        const uint32_t start = pl.start + (k - pl.first) * len;
        in.chunks[w][k] = Chunk{start, min(len, pl.end - start), pl.g, 0};
    }
    grid_dependency_wait();
}

// The largest whole x with (double)x <= limit (>= 0, and below what Sum holds): sums are compared as whole numbers, since
// converting every sum in every thread took most of a round of the search below (4,200 cycles a round with hardly a
// request to add up).
template <class Sum>
__device__ Sum last_within(double limit) {
    if (limit < 9007199254740992.0) return (long long)limit;          // below 2^53 every whole number is a double (rounded down)
    const long long bits = __double_as_longlong(limit), mantissa = (bits & 0xFFFFFFFFFFFFFll) | 1ll << 52;
    const int shift = (int)(bits >> 52) - 1023 - 52;                  // limit = mantissa 2^shift, half the doubles' distance 2^(shift - 1)
    const Sum last = ((Sum)mantissa << shift) + ((Sum)1 << (shift - 1));
    return (mantissa & 1) ? last - 1 : last;                          // (ties go to the even one)
}

// Eq. 1-2 variant of phase 2, one block per (group, policy): the smallest whole slope beta (ticks per prompt
// token) with  sum_l l cnt[l] #{S > w(l)} <= b Total N,  w(l) = 0 for l <= l_immediate, min(beta l, w_tail) above.
// The sum is exact: it is at most Total N <= 4,096 N^2, which 64 bits hold up to kBetaLargeN requests in the group, and 128
// (LARGE) beyond.  It does not grow with beta, so beta is found by search: three slopes a
// round, which cut the range to a quarter.  A thread keeps up to four of the prompt lengths that occur and, for each, the two positions in the
// sorted ticks that belong to the ends of the range, between which the positions of the slopes in between lie; the first
// and last positions come from the bins' starts in shared memory.  Bound: issue and latency of one block (rounds by bins of
// two barriers and up to a dozen products a thread, then two by ticks).  (300,000 requests in six groups under sixteen such policies: 437 us
// with a bisection whose every step searched all the ticks for every length, 82 with every length and products of 64 by 64 bits, 31 of
// them the rounds by bins, 60 with these kept short, 50 now that they part octaves.  Four blocks a pair gave 4 us with few pairs and lost 15 once the pairs outnumbered the
// multiprocessors; three searches in step gave nothing.)
constexpr int kBetaThreads = 1024;
constexpr int kBetaLens = kMaxPrompt / kBetaThreads;                  // prompt lengths a thread has
static_assert(kBetaLens * kBetaThreads == kMaxPrompt, "lengths 1 .. 4096");
constexpr uint64_t kBetaLargeN = 47453132;
static_assert(kMaxPrompt * kBetaLargeN < (1ull << 63) / kBetaLargeN && kMaxPrompt * (kBetaLargeN + 1) >= (1ull << 63) / (kBetaLargeN + 1), "the last N");

// SMALL: a group has fewer than 2^20 requests, so that a length's tokens fit in 32 bits.
constexpr uint64_t kBetaSmallN = 1u << 20;
static_assert(kMaxPrompt * kBetaSmallN <= 1ull << 32, "a length's tokens");
template <bool LARGE, bool SMALL>
__global__ void __launch_bounds__(kBetaThreads)
k_prep_beta(const PolicyIn* __restrict__ pol, const PolicyKind* __restrict__ kinds, uint32_t P, const int64_t* __restrict__ cum_mass,
            const uint32_t* __restrict__ cnt, const int32_t* __restrict__ sorted, const uint32_t* __restrict__ grp_off,
            const uint32_t* __restrict__ tick_start, const uint32_t* __restrict__ tick_cnt, const uint32_t* __restrict__ pairs,
            Prep* __restrict__ prep, bool early) {
    __shared__ uint32_t s_end[kTickBins];                             // ticks of the group up to the bin's last
    __shared__ uint16_t s_len[kMaxPrompt];                            // the lengths that requests have
    __shared__ uint32_t s_wtot[32];
    __shared__ long long part[8][32], total[6];
    using Mass = typename std::conditional<SMALL, uint32_t, unsigned long long>::type;
    using Sum = typename std::conditional<LARGE, __int128, long long>::type;
    grid_dependency_wait();
    if (early) let_next_start();
    const uint32_t pair = pairs[blockIdx.x], p = pair % P;
    const int g = (int)(pair / P);
    Prep& out = prep[(size_t)g * P + p];
    const Prep pr = out;
    const PolicyIn pc = pol[p];
    if (!pr.beta_rule || !pr.device_constrained || (double)pc.budget <= (double)kinds[pc.kind].alpha) return;   // block-uniform
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const uint32_t off = grp_off[g], N = grp_off[g + 1] - off;
    const int32_t* srt = sorted + off;
    const double Total = (double)cum_mass[(size_t)g * (kMaxPrompt + 2) + kMaxPrompt + 1];
    const Sum limit = last_within<Sum>(__dmul_rn(__dmul_rn((double)pc.budget, Total), (double)N));
    const uint32_t w_tail = (uint32_t)pr.w_tail, l_imm = (uint32_t)pr.l_star;
    for (int k = threadIdx.x; k < kTickBins; k += kBetaThreads)
        s_end[k] = tick_start[(size_t)g * kTickBins + k] + tick_cnt[(size_t)g * kTickBins + k] - off;
    // a thread's four lengths, and from then on every 1,024th of those that requests have: each of these costs a round as much, and the
    // long ones are few
    uint32_t lengths, own = 0;
    {
        uint32_t c[kBetaLens];
#pragma unroll
        for (int i = 0; i < kBetaLens; ++i) {
            c[i] = cnt[(size_t)g * (kMaxPrompt + 1) + 1 + threadIdx.x * kBetaLens + i];
            own += c[i] ? 1u : 0u;
        }
        uint32_t at = block_inclusive_scan(own, s_wtot, &lengths) - own;
#pragma unroll
        for (int i = 0; i < kBetaLens; ++i) if (c[i]) s_len[at++] = (uint16_t)(1 + threadIdx.x * kBetaLens + i);
    }
    __syncthreads();

    // ticks at or below w, known to be between lo and hi of them
    auto position = [&](uint32_t w, uint32_t lo, uint32_t hi) {
        if (lo < hi) {
            const int bin = tick_bin(w);
            if (bin > 0) lo = max(lo, s_end[bin - 1]);
            hi = min(hi, s_end[bin]);
        }
        while (lo < hi) {
            const uint32_t mid = LARGE ? lo + ((hi - lo) >> 1) : (lo + hi) >> 1;       // (their sum may pass 2^32)
            if (!DBG_OK(mid, N, DBG_K_PREP, DBG_ELEMENT)) break;
            if ((uint32_t)srt[mid] <= w) lo = mid + 1; else hi = mid;
        }
        return lo;
    };
    Mass tokens[kBetaLens];                                           // of the requests of the length (0: there is no such length)
    uint32_t len[kBetaLens], at_lo[kBetaLens], at_hi[kBetaLens];      // positions at the range's ends
#pragma unroll
    for (int i = 0; i < kBetaLens; ++i) {
        const uint32_t x = threadIdx.x + i * kBetaThreads;
        len[i] = x < lengths ? s_len[x] : 1u;
        tokens[i] = x < lengths ? (Mass)len[i] * cnt[(size_t)g * (kMaxPrompt + 1) + len[i]] : (Mass)0;
    }
    // the block's sums of the values, the same to all threads.  Over a warp the lanes halve what they add up at every step
    // (nine exchanges for six values, not thirty); a warp then adds up the warps' parts of one value for all.
    auto add_up = [&](auto& v) {
        constexpr int kValues = (int)(sizeof(v) / sizeof(v[0])), kHold = kValues <= 2 ? 2 : kValues <= 4 ? 4 : 8;
        long long x[kHold];
#pragma unroll
        for (int j = 0; j < kHold; ++j) x[j] = j < kValues ? v[j] : 0ll;
#pragma unroll
        for (int s = kHold / 2, o = 16; s > 0; s >>= 1, o >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int j = 0; j < s; ++j) x[j] = (up ? x[j + s] : x[j]) + __shfl_xor_sync(FULL, up ? x[j] : x[j + s], o);
        }
#pragma unroll
        for (int o = 16 / kHold; o > 0; o >>= 1) x[0] += __shfl_xor_sync(FULL, x[0], o);
        if (lane % (32 / kHold) == 0) part[lane / (32 / kHold)][wi] = x[0];
        __syncthreads();
        if (wi < kValues) {
            long long y = part[wi][lane];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) y += __shfl_xor_sync(FULL, y, o);
            if (lane == 0) total[wi] = y;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kValues; ++j) v[j] = total[j];
    };
    auto totals = [&](auto& v) {
        if constexpr (!LARGE) {
            add_up(v);
        } else {
            constexpr int kValues = (int)(sizeof(v) / sizeof(v[0]));
            long long low[kValues], high[kValues];                    // 48 bits, and those above (28 at most)
#pragma unroll
            for (int j = 0; j < kValues; ++j) { low[j] = (long long)(v[j] & 0xFFFFFFFFFFFFll); high[j] = (long long)(v[j] >> 48); }
            add_up(low);
            add_up(high);
#pragma unroll
            for (int j = 0; j < kValues; ++j) v[j] = ((Sum)high[j] << 48) + low[j];
        }
    };
    // (a slope is at most w_tail + 1)
    auto wait = [&](long long beta, uint32_t l) {
        const unsigned long long w = (unsigned long long)(uint32_t)beta * l;
        return l <= l_imm ? 0u : w < w_tail ? (uint32_t)w : w_tail;
    };
    auto mass = [&](Mass t, uint32_t requests) { return LARGE ? (Sum)t * (Sum)requests : (Sum)((unsigned long long)t * requests); };
    long long lo = 0, hi = (long long)w_tail + 1;                     // beyond hi every wait is w_tail
    // ---- first by whole bins: the ticks up to a bin's first and last bound the sum from both sides, which settles most of
    //      the range without a look at the ticks
    while (hi - lo > 1) {
        const long long d = hi - lo;
        long long m[3] = {lo + (d + 3) / 4, lo + (d + 1) / 2, lo + (3 * d + 3) / 4};
        if (hi > 8 * (lo + 1)) {
            // The bins part octaves: while the ends are octaves apart so are the slopes in between.  (w_tail is far above the slope that fits,
            // which even parts of the range approach by two bits a round; any three in between will do, to whatever digits.)
            const float at = (float)(lo + 1), by = sqrtf(sqrtf((float)hi / at));
            m[0] = min((long long)(at * by), hi - 1); m[1] = min((long long)(at * by * by), hi - 1); m[2] = min((long long)(at * by * by * by), hi - 1);
        }
        Sum v[6] = {0, 0, 0, 0, 0, 0};                                // at least, at most
#pragma unroll
        for (int i = 0; i < kBetaLens; ++i) {
            if (tokens[i] == 0) continue;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int bin = tick_bin(wait(m[j], len[i]));
                v[j] += mass(tokens[i], N - s_end[bin]);
                v[3 + j] += mass(tokens[i], N - (bin ? s_end[bin - 1] : 0u));
            }
        }
        totals(v);
        const long long old_lo = lo, old_hi = hi;
#pragma unroll
        for (int j = 2; j >= 0; --j) if (v[3 + j] <= limit && m[j] < hi) hi = m[j];      // certainly fits
#pragma unroll
        for (int j = 0; j < 3; ++j) if (v[j] > limit && m[j] > lo && m[j] < hi) lo = m[j];   // certainly does not
        if (lo == old_lo && hi == old_hi) break;
    }
    // ---- the positions at the ends of what is left
    {
        Sum v[2] = {0, 0};
#pragma unroll
        for (int i = 0; i < kBetaLens; ++i) {
            at_lo[i] = at_hi[i] = 0;
            if (tokens[i] == 0) continue;
            at_lo[i] = position(wait(lo, len[i]), 0u, N);
            at_hi[i] = len[i] <= l_imm ? at_lo[i] : position(wait(hi, len[i]), at_lo[i], N);
            v[0] += mass(tokens[i], N - at_lo[i]);
            v[1] += mass(tokens[i], N - at_hi[i]);
        }
        totals(v);
        if (lo == 0 && v[0] <= limit) hi = lo;                // (no waits at all fit)
        else if (v[1] > limit) lo = hi;                       // not even the longest waits fit
    }
    // the slope at lo is too small, that at hi fits
    while (hi - lo > 1) {
        const long long d = hi - lo;
        const long long m[3] = {lo + (d + 3) / 4, lo + (d + 1) / 2, lo + (3 * d + 3) / 4};     // (ascending, above lo, at most hi)
        uint32_t at[3][kBetaLens];
        Sum v[3] = {0, 0, 0};
#pragma unroll
        for (int i = 0; i < kBetaLens; ++i) {
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                at[j][i] = at_lo[i];
                if (at_lo[i] < at_hi[i]) at[j][i] = position(wait(m[j], len[i]), at_lo[i], at_hi[i]);
                v[j] += mass(tokens[i], N - at[j][i]);
            }
        }
        totals(v);
        const int fit = v[0] <= limit ? 0 : v[1] <= limit ? 1 : v[2] <= limit ? 2 : 3;   // first slope that fits
        const long long old_lo = lo;
        lo = fit == 0 ? old_lo : fit == 1 ? m[0] : fit == 2 ? m[1] : m[2];
        hi = fit == 0 ? m[0] : fit == 1 ? m[1] : fit == 2 ? m[2] : hi;
#pragma unroll
        for (int i = 0; i < kBetaLens; ++i) {
            if (fit < 3) at_hi[i] = fit == 0 ? at[0][i] : fit == 1 ? at[1][i] : at[2][i];
            if (fit > 0) at_lo[i] = fit == 1 ? at[0][i] : fit == 2 ? at[1][i] : at[2][i];
        }
    }
    if (threadIdx.x == 0) out.w_star = (int32_t)hi;
}

}  // namespace

DBG_TRANSLATION_UNIT()

cudaError_t launch_prep(uint32_t P, int G, const GroupConst* gc, const int64_t* cum_mass,
                        const uint32_t* cnt, const int32_t* sorted, const uint32_t* grp_off, Prep* prep, const TablesIn& tables,
                        void* clear, size_t clear_bytes, int sms, cudaStream_t st) {
    // a warp per pair, and blocks enough to clear at the speed of memory and to read the tables at once
    uint32_t vecs = (uint32_t)(clear_bytes / 16);
    const uint32_t moved = std::max((vecs + 4 * kPrepThreads - 1) / (4 * kPrepThreads), (tables.vecs - tables.skip + kPrepThreads - 1) / kPrepThreads);
    const uint32_t blocks = std::max((P * (uint32_t)G + kPrepWarps - 1) / kPrepWarps, std::min(moved, (uint32_t)sms * 8u));
    auto go = [&](auto* kernel, const void* given) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = blocks; cfg.blockDim = kPrepThreads; cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        TablesIn in = tables;
        uint4* at = (uint4*)clear;
        void* args[] = {&P, &G, &gc, &cum_mass, &cnt, &sorted, &grp_off, &prep, &in, &at, &vecs, const_cast<void*>(given)};
        return cudaLaunchKernelExC(&cfg, (const void*)kernel, args);
    };
    // (a launch copies the whole parameter: three sizes of it)
    const size_t bytes = (size_t)tables.vecs * 16;
    if (bytes <= 4096) return go(k_prep<4096>, tables.host);
    if (bytes <= 12288) return go(k_prep<12288>, tables.host);
    if (bytes <= kTablesInline) return go(k_prep<(int)kTablesInline>, tables.host);
    return go(k_prep<0>, tables.host);
}

cudaError_t launch_prep_beta(const PolicyIn* pol, const PolicyKind* kinds, uint32_t P, const int64_t* cum_mass, const uint32_t* cnt,
                             const int32_t* sorted, const uint32_t* grp_off, const uint32_t* tick_start,
                             const uint32_t* tick_cnt, const uint32_t* pairs, uint32_t n_pairs, uint64_t most, Prep* prep, bool early, cudaStream_t st) {
    auto* kernel = most > kBetaLargeN ? k_prep_beta<true, false> : most < kBetaSmallN ? k_prep_beta<false, true> : k_prep_beta<false, false>;
    return launch_after(kernel, n_pairs, kBetaThreads, 0, st, pol, kinds, P, cum_mass, cnt, sorted, grp_off, tick_start,
                        tick_cnt, pairs, prep, early);
}

}  // namespace disco
