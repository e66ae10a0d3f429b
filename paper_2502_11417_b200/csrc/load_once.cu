// Trace ingestion of small and middling traces, and the sort of as many ticks: the same results as k_load's (load.cu) by one
// kernel whose threads read their requests once and keep them.
//
// One block of 1024 threads per multiprocessor, all resident at once (a cooperative launch):
//   1. a thread reads up to four (ticks alone: eight) requests and counts them by (group, bin of ticks) and (group, prompt
//      length) in counters of the block's own, which gives each its rank in the block's part of its bucket; the block adds its
//      counters to the global ones, which gives the place of its part in each bucket;
//   2. behind a wait for all blocks every block adds all global counters up by itself: where the buckets start.  The requests go
//      to their places, the blocks write a share of the tables each;
//   3. behind another wait the blocks sort the ticks window by window.
// Further blocks, one a group, only wait for the counts and add up the input-token mass.  A single block (one group, up to 4,096
// requests) keeps its counters in shared memory throughout and waits for nobody.
//
// Bound: latency, some fifteen dependent steps, and from half a million requests on the scattered stores.  Against k_load, which
// reads the requests twice and waits three times (with the memset in front of it, kernels and gaps): 100,000 requests in one group
// 42 us -> 19, in six 56 -> 33; a million 64 -> 44 and 76 -> 55; 1,000 in one block 23 -> 17; 100,000 ticks 25 -> 15.  Where the
// threads cannot keep their requests (8,192 a block) k_load is left.  (Eight requests a thread spill 168 bytes, four 48.)
#include <algorithm>
#include <cstdlib>

#include "ingest.cuh"

namespace disco {

namespace {

// Waits until `want` blocks have arrived.  False, to all threads: the block has to leave.
template <bool ARRIVE>
__device__ __forceinline__ bool wait_for(LoadZero* z, uint32_t want) {
    __syncthreads();
    bool lost = false;
    if (threadIdx.x == 0) {
        if (ARRIVE) { __threadfence(); atomicAdd(&z->barrier, 1u); }
        lost = !await_blocks(z, want);
    }
    return !__syncthreads_or(lost);
}

template <int SRC, int FORM, int QUADS>
__global__ void __launch_bounds__(kThreads, 1)
k_load_once(const __grid_constant__ LoadArgs a) {
    constexpr bool kTrace = SRC == S_TRACE;
    constexpr int kItems = 4 * QUADS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_off[kMaxGroups + 1], s_win0[kMaxGroups + 1];       // where the groups' ticks and windows start
    __shared__ uint32_t s_base[33], s_wtot[32];
    __shared__ unsigned long long s_wide[32], s_win[2];
    __shared__ uint32_t s_sum[kPrivateGroups], s_max, s_item, s_bins[2];
    const int G = a.G, tid = threadIdx.x, lane = tid & 31;
    const uint32_t block = blockIdx.x, blocks = a.once.blocks;
    LoadZero* z = a.z;
    // counters of the ticks' bins, then of the prompt lengths, as in global memory
    const int T0 = G * kTickBins, K = T0 + (kTrace ? G * kLens : 0), shift = a.once.seg_shift, segs = (K >> shift) + 1;
    uint32_t *s = (uint32_t*)smem_raw, *all = a.tick_cnt;
    const bool alone = gridDim.x == 1;

    if (kTrace && block >= blocks) {                   // a group's input-token mass
        const int g = (int)(block - blocks);
        if (!wait_for<false>(z, blocks + ABSENT(a, 1u) + ABSENT(a, 4u)) || __ldcg(&z->err[0])) return;
        group_mass(a.cnt + (size_t)g * kLens, a.cum_mass + (size_t)g * (kLens + 1), s_wide);
    } else {
        // ---- 1. count
        const uint32_t i00 = block * a.once.per_block, i_end = min(a.n, i00 + a.once.per_block);
        const auto aligned = [](const void* p, uintptr_t k) { return ((uintptr_t)p & (k - 1)) == 0; };
        const bool wide = SRC == S_TICKS ? aligned(a.ticks, 16)
                                         : aligned(a.ttft, 16) && (!kTrace || (aligned(a.prompt, 16) && aligned(a.outlen, 16) && aligned(a.sp, 4) && aligned(a.dp, 4)));
        Raw raw[QUADS];
#pragma unroll
        for (int q = 0; q < QUADS; ++q) {
            const uint32_t i0 = i00 + (uint32_t)(q * kThreads + tid) * 4u;
            if (i0 < i_end) read_raw<SRC, FORM, true>(a, i0, wide, raw[q]);
        }
        for (int i = tid * 4; i < segs << shift; i += 4 * kThreads) *reinterpret_cast<uint4*>(s + i) = make_uint4(0u, 0u, 0u, 0u);
        // the words that the next load finds zero
        for (uint32_t i = block * kThreads + tid; i < a.once.clear_vecs; i += blocks * kThreads) a.once.clear[i] = make_uint4(0u, 0u, 0u, 0u);
        if (alone) for (int i = tid; i < (int)(sizeof(LoadZero) / 4); i += kThreads) ((uint32_t*)z)[i] = 0;
        if (SRC == S_TICKS) for (int g = tid; g <= G; g += kThreads) s_off[g] = a.off[g];
        if (kTrace && tid < G) s_sum[tid] = 0;
        if (tid == 0) { s_max = 0; s_bins[0] = 0xFFFFFFFFu; s_bins[1] = 0; }
        __syncthreads();
        uint32_t S[kItems], ln[kItems] = {}, kg[QUADS], pt[kItems], pl[kTrace ? kItems : 1];   // kg: groups, a byte each (255: none); pt, pl: ranks, then places
        uint32_t longest = 0;
#pragma unroll
        for (int q = 0; q < QUADS; ++q) {
            Item x[4];
            const uint32_t i0 = i00 + (uint32_t)(q * kThreads + tid) * 4u;
            if (i0 < i_end) to_items<SRC, FORM, true>(a, i0, raw[q], s_off, x);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = q * 4 + u;
                kg[q] = u ? kg[q] | 255u << (8 * u) : 255u;
                if (i0 >= i_end || !x[u].in || !DBG_OK(x[u].g, G, DBG_K_INGEST, DBG_GROUP) || !DBG_OK(x[u].l, kLens, DBG_K_INGEST, DBG_TABLE)) continue;
                const int tb = tick_bin(x[u].S);
                if (!DBG_OK(tb, kTickBins, DBG_K_INGEST, DBG_BIN)) continue;
                S[k] = x[u].S; kg[q] ^= (255u ^ x[u].g) << (8 * u);
                pt[k] = atomicAdd(&s[x[u].g * kTickBins + tb], 1u);
                if constexpr (kTrace) {
                    ln[k] = x[u].l | x[u].o << 16;
                    pl[k] = atomicAdd(&s[T0 + x[u].g * kLens + x[u].l], 1u);
                    longest = max(longest, x[u].o);
                }
            }
        }
        auto group = [&](int k) { return byte_of(kg[k / 4], k % 4); };
        auto tick_at = [&](int k) { return group(k) * kTickBins + (uint32_t)tick_bin(S[k]); };
        auto len_at = [&](int k) { return kTrace ? (uint32_t)T0 + group(k) * kLens + (ln[k] & 0xFFFFu) : 0u; };
        __syncthreads();
        // what the host wants to know of the lengths (32 bits hold a block's tokens); read behind the second wait
        auto totals = [&] {
            if constexpr (kTrace) {
                longest = __reduce_max_sync(FULL, longest);
                if (lane == 0 && longest) atomicMax(&s_max, longest);
                for (int g = 0; g < G; ++g) {
                    uint32_t v = 0;
#pragma unroll
                    for (int k = 0; k < kItems; ++k) v += (int)group(k) == g ? ln[k] >> 16 : 0u;
                    v = __reduce_add_sync(FULL, v);
                    if (lane == 0 && v) atomicAdd(&s_sum[g], v);
                }
                __syncthreads();
                if (tid < G && s_sum[tid]) atomicAdd((unsigned long long*)&z->grp_sum_n[tid], (unsigned long long)s_sum[tid]);
                if (tid == 0 && s_max) atomicMax(&z->max_n, s_max);
            }
        };
        if (!alone) {
            // (Neighbouring counters together: an addition by the first request of each bucket took 20 us instead of 4 for 500,000
            // requests in six groups, each a request of its own to L2.)
            constexpr int kJoin = 8;
#pragma unroll 1
            for (int i0 = tid; i0 < K; i0 += kJoin * kThreads) {
                uint32_t c[kJoin];
#pragma unroll
                for (int u = 0; u < kJoin; ++u) c[u] = i0 + u * kThreads < K ? s[i0 + u * kThreads] : 0u;
#pragma unroll
                for (int u = 0; u < kJoin; ++u) if (c[u]) c[u] = atomicAdd(&all[i0 + u * kThreads], c[u]);
#pragma unroll
                for (int u = 0; u < kJoin; ++u) if (i0 + u * kThreads < K) s[i0 + u * kThreads] = c[u];
            }
            __syncthreads();
            if (tid == 0) { __threadfence(); atomicAdd(&z->barrier, 1u); }
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                if (group(k) == 255u) continue;
                pt[k] += s[tick_at(k)];
                if constexpr (kTrace) pl[k] += s[len_at(k)];
            }
            LATE(a, block == blocks - 1u);
            totals();
            if (!wait_for<false>(z, blocks + ABSENT(a, 1u) + ABSENT(a, 4u))) return;
        } else if (kTrace) {
            totals();
            // cumulative input-token mass, while the counts are there
            static_assert(4 * kThreads == kMaxPrompt, "four lengths a thread");
            const uint32_t* c = s + T0 + 1 + tid * 4;
            unsigned long long mass = 0, total;
#pragma unroll
            for (int u = 0; u < 4; ++u) mass += (unsigned long long)(tid * 4 + 1 + u) * c[u];
            unsigned long long run = block_inclusive_scan(mass, s_wide, &total) - mass;
#pragma unroll
            for (int u = 0; u < 4; ++u) { a.cum_mass[tid * 4 + 1 + u] = (int64_t)run; run += (unsigned long long)(tid * 4 + 1 + u) * c[u]; }
            if (tid == 0) { a.cum_mass[0] = 0; a.cum_mass[kLens] = (int64_t)total; }
            __syncthreads();
        }

        // ---- 2. place
        const int32_t refused = __ldcg(&z->err[0]);
        // where every bucket starts: a warp adds a segment of the counters up, then the segments' totals
        {
            const int w = tid >> 5;
            uint32_t carry = 0;
            if (w < segs) {
                // (a few loads at a time: they do not move over the stores by themselves)
                constexpr int kAhead = 4;
#pragma unroll 1
                for (int j0 = 0; j0 < 1 << (shift - 7); j0 += kAhead) {
                    uint4 c[kAhead];
                    uint32_t run[kAhead];
#pragma unroll
                    for (int j = 0; j < kAhead; ++j) {
                        const int k = (w << shift) + (j0 + j) * 128 + lane * 4;
                        c[j] = make_uint4(0u, 0u, 0u, 0u);
                        if (k >= K || j0 + j >= 1 << (shift - 7)) continue;        // (what lies behind the last in its vector is zero)
                        c[j] = alone ? *reinterpret_cast<uint4*>(s + k) : __ldcg(reinterpret_cast<const uint4*>(all + k));
                    }
#pragma unroll
                    for (int j = 0; j < kAhead; ++j) run[j] = c[j].x + c[j].y + c[j].z + c[j].w;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
#pragma unroll
                        for (int j = 0; j < kAhead; ++j) {
                            const uint32_t up = __shfl_up_sync(FULL, run[j], off);
                            if (lane >= off) run[j] += up;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < kAhead; ++j) {
                        if (j0 + j >= 1 << (shift - 7)) break;
                        const int k = (w << shift) + (j0 + j) * 128 + lane * 4;
                        if (alone && k < K) *reinterpret_cast<uint4*>(all + k) = c[j];
                        const uint32_t at = carry + run[j] - (c[j].x + c[j].y + c[j].z + c[j].w);
                        carry += __shfl_sync(FULL, run[j], 31);
                        *reinterpret_cast<uint4*>(s + k) = make_uint4(at, at + c[j].x, at + c[j].x + c[j].y, at + c[j].x + c[j].y + c[j].z);
                    }
                }
            }
            if (lane == 0) s_wtot[w] = carry;
            __syncthreads();
            if (w == 0) {
                const uint32_t own = s_wtot[lane];
                uint32_t run = own;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const uint32_t up = __shfl_up_sync(FULL, run, off);
                    if (lane >= off) run += up;
                }
                s_base[lane] = run - own;
            }
            __syncthreads();
        }
        if (refused) {                                 // a rejected trace: nothing is placed
            if (SRC != S_TICKS && block == 0 && tid < 4 && a.readback) a.readback->err[tid] = __ldcg(&z->err[tid]);
            return;
        }
        auto start = [&](uint32_t k) { return s[k] + s_base[k >> shift]; };     // (of a length: behind the n ticks)
        if (SRC != S_TICKS) for (int g = tid; g <= G; g += kThreads) s_off[g] = g < G ? start(g * kTickBins) : a.n;
        __syncthreads();
        const uint32_t win_shift = a.once.win_shift, win_more = (1u << win_shift) - 1u;
        if (tid == 0) {
            uint32_t at = 0;
            for (int g = 0; g < G; ++g) { s_win0[g] = at; at += (s_off[g + 1] - s_off[g] + win_more) >> win_shift; }
            s_win0[G] = at;
        }
#pragma unroll
        for (int q = 0; q < QUADS; ++q) {
            const uint32_t i0 = i00 + (uint32_t)(q * kThreads + tid) * 4u;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = q * 4 + u;
                if (group(k) == 255u) continue;
                const uint32_t tp = pt[k] + start(tick_at(k));
                if (DBG_OK(tp, a.n, DBG_K_GATHER, DBG_ELEMENT)) a.binned[tp] = S[k];
                if constexpr (kTrace) {
                    pl[k] += start(len_at(k)) - a.n;
                    if (DBG_OK(pl[k], a.n, DBG_K_GATHER, DBG_REQUEST)) a.req[pl[k]] = make_uint4(S[k], ln[k], i0 + u, 0u);
                }
            }
            if constexpr (kTrace) {
                if (i0 + 4u <= i_end) *reinterpret_cast<uint4*>(a.inv + i0) = make_uint4(pl[q * 4], pl[q * 4 + 1], pl[q * 4 + 2], pl[q * 4 + 3]);
                else
#pragma unroll
                    for (int u = 0; u < 4; ++u) if (i0 + u < i_end) a.inv[i0 + u] = pl[q * 4 + u];
            }
        }
        __syncthreads();
        // the block's share of the tables, and its bins' windows
        {
            const int per = (K + (int)blocks - 1) / (int)blocks, k0 = min(K, (int)block * per), k1 = min(K, k0 + per);
            for (int k = k0 + tid; k < k1; k += kThreads) {
                const uint32_t at = start(k), end = start(k + 1);
                if (k >= T0) { a.len_end[k - T0] = end - a.n; continue; }
                a.tick_start[k] = at;
                if (at == end) continue;
                if (alone) { atomicMin(&s_bins[0], (uint32_t)k); atomicMax(&s_bins[1], (uint32_t)k); continue; }
                const int g = k / kTickBins;
                const uint32_t win = s_win0[g] + ((at - s_off[g]) >> win_shift);
                unsigned long long* to = a.once.windows + 2 * (size_t)win;
                if (!DBG_OK(win, kOnceWindows, DBG_K_TABLES, DBG_SLOT)) continue;
                atomicMax(to, (unsigned long long)(0xFFFFFFFFu - (uint32_t)k) << 32 | at);
                atomicMax(to + 1, (unsigned long long)((uint32_t)k + 1u) << 32 | end);
            }
        }
        if (kTrace && block == 0) {
            for (int g = tid; g < G; g += kThreads) {
                const uint32_t N = s_off[g + 1] - s_off[g];
                a.readback->ng[g] = N; a.readback->grp_off[g] = s_off[g];
                a.grp_off[g] = s_off[g];
                a.fin_totals[G + g] = N;                               // what the final reductions' totals refer to
                if (N == 0) a.readback->knot_max[g] = 0;
            }
            if (tid == 0) { a.grp_off[G] = s_off[G]; a.readback->grp_off[G] = s_off[G]; }
            for (int k = tid; k < G * kNKnots; k += kThreads)
                if (s_off[k / kNKnots + 1] == s_off[k / kNKnots]) a.knots[k] = 0;
        }
        if (!alone && !wait_for<true>(z, 2 * blocks + ABSENT(a, 2u) + ABSENT(a, 3u))) return;
        // A block announces itself at the first wait before it adds its share of these, and at the second behind it.  (The last
        // block has the fewest windows.)
        if (kTrace && block == blocks - 1u) {
            for (int g = tid; g < G; g += kThreads) {
                const uint64_t sum = __ldcg((const unsigned long long*)&z->grp_sum_n[g]);
                a.readback->grp_sum_n[g] = sum; a.fin_totals[g] = sum;
            }
            if (tid == 0) a.readback->max_n = __ldcg(&z->max_n);
        }

        // ---- 3. sort
        SortSmem& sm = *reinterpret_cast<SortSmem*>(smem_raw);
        const uint32_t n_win = alone ? min(a.n, 1u) : s_win0[G];
#pragma unroll 1
        for (uint32_t win = block; win < n_win; win += blocks) {
            __syncthreads();
            if (tid < 2) s_win[tid] = alone ? (unsigned long long)(tid ? s_bins[1] + 1u : 0xFFFFFFFFu - s_bins[0]) << 32 | (tid ? a.n : 0u)
                                            : __ldcg(a.once.windows + 2 * (size_t)win + tid);
            __syncthreads();
            if (s_win[1] == 0ull) continue;                            // (inside a large bin)
            const uint32_t first = 0xFFFFFFFFu - (uint32_t)(s_win[0] >> 32), last = (uint32_t)(s_win[1] >> 32) - 1u;
            const uint32_t k0 = (uint32_t)s_win[0], k1 = (uint32_t)s_win[1];
            const int g = (int)first / kTickBins;
            sort_bins(a, sm, g, (int)first - g * kTickBins, (int)last - g * kTickBins, k0, k1);
            if (kTrace) write_knots<kThreads>(a, g, k0, k1, s_off[g], s_off[g + 1] - s_off[g]);
        }
    }
    if (kTrace || (SRC == S_TTFT && a.readback)) {
        // the last block to come here reports the flags (where a block has left, none does: what the host put there stands)
        if (tid == 0) { __threadfence(); s_item = atomicAdd(&z->done, 1u); }
        __syncthreads();
        if (s_item == gridDim.x - 1 && tid < 4) a.readback->err[tid] = __ldcg(&z->err[tid]);
    }
}

template <int SRC, int FORM, int QUADS>
cudaError_t launch(const LoadArgs& a, uint32_t spare, cudaStream_t st) {
    const int K = a.G * (kTickBins + (SRC == S_TRACE ? kLens : 0));
    const size_t smem = std::max((size_t)((K >> a.once.seg_shift) + 1 << a.once.seg_shift) * 4, sizeof(SortSmem));
    auto* kernel = k_load_once<SRC, FORM, QUADS>;
    cudaError_t e = allow_smem((const void*)kernel, 220 * 1024);
    if (e) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = a.once.blocks + spare; cfg.blockDim = kThreads; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (cfg.gridDim.x > 1) {
        if (!a.once.zeroed && (e = cudaMemsetAsync(a.z, 0, a.zero_bytes, st))) return e;
        const char* win = (const char*)a.once.windows;
        if (!a.once.zeroed && (win < (char*)a.z || win >= (char*)a.z + a.zero_bytes) &&
            (e = cudaMemsetAsync(a.once.windows, 0, kOnceWindows * 16, st))) return e;
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
    }
#ifdef DISCO_DEBUG
    LoadArgs b = a;
    if (const char* wait = std::getenv("DISCO_DEBUG_ABSENT")) b.absent = (uint32_t)std::atoi(wait);
    return cudaLaunchKernelEx(&cfg, kernel, b);
#else
    return cudaLaunchKernelEx(&cfg, kernel, a);
#endif
}

template <int SRC>
cudaError_t plan_and_launch(const LoadArgs& args, int sms, cudaStream_t st) {
    LoadArgs a = args;
    constexpr bool kTrace = SRC == S_TRACE;
    const bool single = a.G == 1 && a.n <= kOnceAlone;
    const uint32_t spare = kTrace && !single ? (uint32_t)a.G : 0u;   // (once_trace has seen that there are as many)
    const uint32_t most = std::min((uint32_t)sms, kLoadBlocks) - spare;
    // a request a thread until the multiprocessors are full, and some blocks whatever the number of requests
    const uint32_t least = a.G > 1 ? 4u * (uint32_t)a.G : 2u;
    uint32_t blocks = single ? 1u : std::min(std::max((a.n + kThreads - 1) / kThreads, least), most);
    a.once.per_block = ((a.n + blocks - 1) / blocks + 3u) / 4u * 4u;
    a.once.blocks = blocks;
    // segments of the counters, at most 32 and whole 128s; windows of ticks, about one a block
    const int K = a.G * (kTickBins + (kTrace ? kLens : 0));
    a.once.seg_shift = 7;
    while ((K >> a.once.seg_shift) + 1 > 32) ++a.once.seg_shift;
    a.once.win_shift = 9;
    while (a.once.win_shift < 12 && (1u << a.once.win_shift) < a.n / blocks) ++a.once.win_shift;
    const bool two = a.once.per_block > 4u * kThreads;
    if (a.once.per_block > 8u * kThreads) return cudaErrorInvalidConfiguration;
    if constexpr (SRC == S_TRACE) {
        if (a.packed) return two ? launch<SRC, F_PACKED, 2>(a, spare, st) : launch<SRC, F_PACKED, 1>(a, spare, st);
        return two ? launch<SRC, F_COLUMNS, 2>(a, spare, st) : launch<SRC, F_COLUMNS, 1>(a, spare, st);
    } else {
        return two ? launch<SRC, F_COLUMNS, 2>(a, 0u, st) : launch<SRC, F_COLUMNS, 1>(a, 0u, st);
    }
}

}  // namespace

DBG_TRANSLATION_UNIT()

cudaError_t run_load_once(const LoadArgs& a, int sms, cudaStream_t st) { return plan_and_launch<S_TRACE>(a, sms, st); }
cudaError_t run_sort_ticks_once(const LoadArgs& a, int sms, cudaStream_t st) { return plan_and_launch<S_TICKS>(a, sms, st); }
cudaError_t run_sort_ttft_once(const LoadArgs& a, int sms, cudaStream_t st) { return plan_and_launch<S_TTFT>(a, sms, st); }

}  // namespace disco
