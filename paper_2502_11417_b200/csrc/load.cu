// Trace ingestion on the device in one kernel, for the traces that load_once.cu and load_large.cu do not take (1.2 to 2.2 million
// requests, to 3.0 million where columns are read in place from page-locked memory, more than seven groups, beyond 2^24 requests, or without room for load_large.cu's buckets), and the sort of as many
// ticks: tick conversion and validation, per-group prompt-length histogram, internal request order (by group, then by prompt
// length), sort of the server-TTFT ticks (the empirical F of Algorithm 1), cumulative input-token mass (Eq. 3) and the quantile
// knots of F.
//
// One block of 1024 threads per multiprocessor, all resident at once (a cooperative launch), works in three passes with a
// wait for all blocks between them:
//   1. count: every request is checked and counted by (group, prompt length) and by (group, bin of its ticks), 128 bins an
//      octave, in counters of the block's own.  The block adds its counters to the global ones and keeps what was there
//      before: where its own requests of each bucket go within the bucket.
//   2. place: the blocks work out where the buckets start, each for its share of the counters (the blocks tell one another
//      their totals), then every block sends its requests to their places: one 16-byte record into the internal order and
//      the ticks into their bin.
//   3. sort: the bins in order, about 4,096 ticks at a time, are sorted in shared memory (all ticks of a window differ in
//      few low bits), each window by one block.  A bin of more than 8,192 ticks that spans at most 2^18 values is sorted by
//      counting them; a trace that has a denser and wider one goes to the radix sort (radix.cu) instead.
//
// Bound: latency up to some 10^5 requests, then scattered stores: the columns are read twice (once when they are in host memory:
// then the first pass leaves a copy), 20 bytes a request are written to scattered places, the ticks are read and written once
// more.  2 million requests in one group: 84 us, 3 million 120, a million in twenty groups 115.  From 2.2 million on load_large.cu is
// the faster one.  (The 64 registers that 1,024 threads leave spill 64 bytes.)
#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "ingest.cuh"

namespace disco {

namespace {

// Waits until every block of the grid has come here `times` times.  False, to all threads: the block has to leave.
__device__ __forceinline__ bool grid_barrier(LoadZero* z, uint32_t times, uint32_t absent) {
    __syncthreads();
    bool lost = false;
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&z->barrier, 1u);
        lost = !await_blocks(z, times * gridDim.x + absent);
    }
    return !__syncthreads_or(lost);
}

// Waits (boundedly, as above) for a word that another block writes once; 0 if it does not come.
__device__ __forceinline__ unsigned long long await_word(LoadZero* z, const unsigned long long* at) {
    unsigned long long v;
    uint32_t tries = 0;
    do {
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(at) : "memory");
    } while (v == 0ull && ++tries < kWaitTries);
    if (v == 0ull) give_up(z);
    return v;
}

// Four counters from k on (16-byte aligned), those from k1 on empty.
__device__ __forceinline__ uint4 four_counters(const uint32_t* cnt, int k, int k1) {
    if (k + 4 <= k1) return __ldcg(reinterpret_cast<const uint4*>(cnt + k));
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (k < k1) v.x = __ldcg(&cnt[k]);
    if (k + 1 < k1) v.y = __ldcg(&cnt[k + 1]);
    if (k + 2 < k1) v.z = __ldcg(&cnt[k + 2]);
    return v;
}

// A block's share of L counters: [k0, k1), whole vectors.
struct Share { int k0, k1; };
__device__ __forceinline__ Share share_of(int L) {
    const int per = ((L + (int)gridDim.x - 1) / (int)gridDim.x + 3) / 4 * 4;
    return Share{min(L, (int)blockIdx.x * per), min(L, ((int)blockIdx.x + 1) * per)};
}

// Exclusive prefix sums over the block's share, `carry` in front of it, four neighbouring counters a thread at a time.
// emit(k, counts, starts): the counters k .. k + 3.  first: this thread's counters of the first 4,096.
template <class E>
__device__ __forceinline__ void scan_share(const uint32_t* cnt, const Share& sh, const uint4& first, uint32_t carry, uint32_t* wtot, E emit) {
    for (int k0 = sh.k0; k0 < sh.k1; k0 += 4 * kThreads) {
        const int k = k0 + (int)threadIdx.x * 4;
        const uint4 c = k0 == sh.k0 ? first : four_counters(cnt, k, sh.k1);
        const uint32_t own = c.x + c.y + c.z + c.w;
        uint32_t total;
        const uint32_t at = carry + block_inclusive_scan(own, wtot, &total) - own;
        if (k < sh.k1) emit(k, c, make_uint4(at, at + c.x, at + c.x + c.y, at + c.x + c.y + c.z));
        carry += total;
        __syncthreads();
    }
}

template <int SRC, bool PRIV, int FORM>
__global__ void __launch_bounds__(kThreads, 1)
k_load(const __grid_constant__ LoadArgs a) {
    constexpr bool kTrace = SRC == S_TRACE;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_off[kMaxGroups + 1];        // group offsets in the internal order
    __shared__ unsigned long long s_wide[32];
    __shared__ uint32_t s_wtot[32];
    __shared__ unsigned long long s_sum[kMaxGroups];
    __shared__ uint32_t s_max, s_item, s_carry[2];
    const int G = a.G, tid = threadIdx.x, lane = tid & 31;
    LoadZero* z = a.z;
    uint32_t* s_tick = (uint32_t*)smem_raw;                            // [G][kTickBins]
    uint32_t* s_len = s_tick + G * kTickBins;                          // [G][kLens]
    uint32_t waits = 0;

    // the block's counters join the global ones; what it finds there is where its own requests go within the bucket
    auto join = [&](uint32_t* mine, uint32_t* all, int count) {
#pragma unroll 1
        for (int i0 = tid; i0 < count; i0 += 4 * kThreads) {
            uint32_t c[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) { const int i = i0 + u * kThreads; c[u] = i < count ? mine[i] : 0u; }
#pragma unroll
            for (int u = 0; u < 4; ++u) if (c[u]) c[u] = atomicAdd(&all[i0 + u * kThreads], c[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u) { const int i = i0 + u * kThreads; if (i < count) mine[i] = c[u]; }
        }
    };

    // ---- 1. count
    if (PRIV) for (int i = tid; i < (kTrace ? G * kLens : 0) + G * kTickBins; i += kThreads) s_tick[i] = 0;
    if (SRC == S_TICKS) for (int g = tid; g <= G; g += kThreads) s_off[g] = a.off[g];
    for (int g = tid; g < G; g += kThreads) s_sum[g] = 0;
    if (tid == 0) s_max = 0;
    __syncthreads();
    // a thread takes four neighbouring requests at a time, as vectors where the columns are aligned
    const auto aligned = [](const void* p, uintptr_t k) { return ((uintptr_t)p & (k - 1)) == 0; };
    const bool wide = SRC == S_TICKS ? aligned(a.ticks, 16)
                                     : aligned(a.ttft, 16) && (!kTrace || (aligned(a.prompt, 16) && aligned(a.outlen, 16) && aligned(a.sp, 4) && aligned(a.dp, 4)));
    const uint32_t stride = gridDim.x * kThreads * 4u, i_first = (blockIdx.x * kThreads + tid) * 4u;
    uint32_t i_next = i_first;                                         // (second pass)
    // Output tokens per group, of this thread's requests: below 2^32.  (Above 16,384 requests more than four blocks share a
    // trace, so that of 2^31 a thread has fewer than 2^19, of 8,192 tokens at most.)
    uint32_t tok[kPrivateGroups] = {};
    uint32_t longest = 0;
#pragma unroll 1
    for (uint32_t i0 = i_first; i0 < a.n; i0 += stride) {
        Item x[4];
        read_items<SRC, FORM, true>(a, i0, wide, s_off, x);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const Item& y = x[u];
            if (!y.in || !DBG_OK(y.g, G, DBG_K_INGEST, DBG_GROUP) || !DBG_OK(y.l, kLens, DBG_K_INGEST, DBG_TABLE)) continue;
            const int tb = tick_bin(y.S);
            if (!DBG_OK(tb, kTickBins, DBG_K_INGEST, DBG_BIN)) continue;
            if (PRIV) {
                if (kTrace) atomicAdd(&s_len[y.g * kLens + y.l], 1u);
                atomicAdd(&s_tick[y.g * kTickBins + tb], 1u);
            } else {
                if (kTrace) { atomicAdd(&a.cnt[(size_t)y.g * kLens + y.l], 1u); atomicAdd(&s_sum[y.g], (unsigned long long)y.o); }
                atomicAdd(&a.tick_cnt[(size_t)y.g * kTickBins + tb], 1u);
            }
            if (kTrace) {
                longest = max(longest, y.o);
                if (PRIV) {
#pragma unroll
                    for (int g = 0; g < kPrivateGroups; ++g) tok[g] += (int)y.g == g ? y.o : 0u;
                }
            }
        }
        if (FORM == F_STAGE) stage_items(a, i0, x);
    }
    if (kTrace) {
        longest = __reduce_max_sync(FULL, longest);
        if (lane == 0 && longest) atomicMax(&s_max, longest);
        if (PRIV) {
#pragma unroll
            for (int g = 0; g < kPrivateGroups; ++g) {
                if (g >= G) break;
                unsigned long long v = tok[g];
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
                if (lane == 0 && v) atomicAdd(&s_sum[g], v);
            }
        }
    }
    __syncthreads();
    if (kTrace) {
        for (int g = tid; g < G; g += kThreads) if (s_sum[g]) atomicAdd((unsigned long long*)&z->grp_sum_n[g], s_sum[g]);
        if (tid == 0 && s_max) atomicMax(&z->max_n, s_max);
    }
    if (PRIV) {
        if (kTrace) join(s_len, a.cnt, G * kLens);
        join(s_tick, a.tick_cnt, G * kTickBins);
    }
    ++waits;
    if (!grid_barrier(z, waits, ABSENT(a, waits))) return;

    // ---- 2. place
    if (__ldcg(&z->err[0])) {                          // a rejected trace: nothing is placed
        if (SRC != S_TICKS && blockIdx.x == 0 && tid < 4 && a.readback) a.readback->err[tid] = __ldcg(&z->err[tid]);
        return;
    }
    // where every bucket starts: the groups one after another, so one running sum over all groups' counters each
    const bool cursors = !PRIV || a.rounds > 1;                        // places are handed out by global cursors
    {
        bool lost = false;
        const Share st = share_of(G * kTickBins), sl = share_of(kTrace ? G * kLens : 0);
        const uint4 ft = four_counters(a.tick_cnt, st.k0 + tid * 4, st.k1);
        const uint4 fl = kTrace ? four_counters(a.cnt, sl.k0 + tid * 4, sl.k1) : make_uint4(0u, 0u, 0u, 0u);
        uint32_t sum[2] = {ft.x + ft.y + ft.z + ft.w, fl.x + fl.y + fl.z + fl.w};
        for (int k = st.k0 + (tid + kThreads) * 4; k < st.k1; k += 4 * kThreads) { const uint4 c = four_counters(a.tick_cnt, k, st.k1); sum[0] += c.x + c.y + c.z + c.w; }
        if (kTrace) for (int k = sl.k0 + (tid + kThreads) * 4; k < sl.k1; k += 4 * kThreads) { const uint4 c = four_counters(a.cnt, k, sl.k1); sum[1] += c.x + c.y + c.z + c.w; }
        if (tid < 2) s_carry[tid] = 0;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < (kTrace ? 2 : 1); ++j) {
            const uint32_t v = __reduce_add_sync(FULL, sum[j]);
            if (lane == 0 && v) atomicAdd(&s_carry[j], v);
        }
        __syncthreads();
        // a warp for each of the two sums: tells the other blocks, and adds up those in front
        const int j = tid >> 5;
        if (j < (kTrace ? 2 : 1)) {
            if (lane == 0)
                asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(&z->part[j][blockIdx.x]), "l"(((unsigned long long)s_carry[j] << 1) | 1ull) : "memory");
            uint32_t before = 0;
            for (uint32_t b = lane; b < blockIdx.x && !lost; b += 32) {
                const unsigned long long word = await_word(z, &z->part[j][b]);
                lost = word == 0ull;
                before += (uint32_t)(word >> 1);
            }
            if (ABSENT(a, 4u) && lane == 0) lost = await_word(z, &z->part[j][kLoadBlocks - 1]) == 0ull;
            before = __reduce_add_sync(FULL, before);
            if (lane == 0) s_carry[j] = before;
        }
        if (__syncthreads_or(lost)) return;                            // (some block's sum did not come)
        scan_share(a.tick_cnt, st, ft, s_carry[0], s_wtot, [&](int k, const uint4&, const uint4& start) {
            *reinterpret_cast<uint4*>(a.tick_start + k) = start;
            if (cursors) *reinterpret_cast<uint4*>(a.tick_at + k) = start;
        });
        if (kTrace)
            scan_share(a.cnt, sl, fl, s_carry[1], s_wtot, [&](int k, const uint4& c, const uint4& start) {
                const uint32_t cs[4] = {c.x, c.y, c.z, c.w}, at[4] = {start.x, start.y, start.z, start.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (k + u < sl.k1) a.len_end[k + u] = cursors ? at[u] : at[u] + cs[u];    // (a cursor ends up where its bucket does)
            });
    }
    ++waits;
    if (!grid_barrier(z, waits, ABSENT(a, waits))) return;
    if (SRC != S_TICKS) for (int g = tid; g <= G; g += kThreads) s_off[g] = g < G ? __ldcg(&a.tick_start[(size_t)g * kTickBins]) : a.n;
    __syncthreads();
    if (!cursors) {
        // The block's counters, places within the buckets so far, become places: a bucket starts where the one in front ends.
        // (All of them side by side: read one by one where they are needed, the few lines that most requests need keep L2
        // busy: 48 us instead of 8 for a million.)
#pragma unroll 4
        for (int k = tid * 4; k < G * kTickBins; k += 4 * kThreads) {
            const uint4 start = __ldcg(reinterpret_cast<const uint4*>(a.tick_start + k));
            uint4& mine = *reinterpret_cast<uint4*>(s_tick + k);
            mine = make_uint4(mine.x + start.x, mine.y + start.y, mine.z + start.z, mine.w + start.w);
        }
        if (kTrace)
#pragma unroll 8
            for (int k = tid + 1; k < G * kLens; k += kThreads) s_len[k] += __ldcg(&a.len_end[k - 1]);
    }
    // the windows' first and last bins
    {
        const Share st = share_of(G * kTickBins);
#pragma unroll 1
        for (int k = st.k0 + tid; k < st.k1; k += kThreads) {
            if (__ldcg(&a.tick_cnt[k]) == 0u) continue;
            const int g = k / kTickBins;
            uint32_t win = (__ldcg(&a.tick_start[k]) - s_off[g]) / kWindow;
            for (int h = 0; h < g; ++h) win += (s_off[h + 1] - s_off[h] + kWindow - 1) / kWindow;
            atomicMax(&a.windows[win].x, 0xFFFFFFFFu - (uint32_t)k);
            atomicMax(&a.windows[win].y, (uint32_t)k + 1u);
        }
    }
    if (kTrace && blockIdx.x == 0) {
        for (int g = tid; g < G; g += kThreads) {
            const uint32_t N = s_off[g + 1] - s_off[g];
            const uint64_t sum = __ldcg((const unsigned long long*)&z->grp_sum_n[g]);
            a.readback->ng[g] = N; a.readback->grp_sum_n[g] = sum; a.readback->grp_off[g] = s_off[g];
            a.grp_off[g] = s_off[g];
            a.fin_totals[g] = sum; a.fin_totals[G + g] = N;            // what the final reductions' totals refer to
            if (N == 0) a.readback->knot_max[g] = 0;
        }
        if (tid == 0) { a.grp_off[G] = s_off[G]; a.readback->grp_off[G] = s_off[G]; a.readback->max_n = __ldcg(&z->max_n); }
        for (int k = tid; k < G * kNKnots; k += kThreads)
            if (s_off[k / kNKnots + 1] == s_off[k / kNKnots]) a.knots[k] = 0;
    }
    __syncthreads();
    auto place = [&](uint32_t i_end) {
#pragma unroll 1
        for (; i_next < i_end; i_next += stride) {
            const uint32_t i0 = i_next;
            Item x[4];
            read_items<SRC, FORM, false>(a, i0, wide, s_off, x);
            uint32_t at[4] = {0, 0, 0, 0}, tp[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const Item& y = x[u];
                if (!y.in || !DBG_OK(y.g, G, DBG_K_GATHER, DBG_GROUP) || !DBG_OK(y.l, kLens, DBG_K_GATHER, DBG_TABLE)) { x[u].in = false; continue; }
                if (kTrace) { const uint32_t lb = y.g * kLens + y.l; at[u] = atomicAdd(PRIV ? &s_len[lb] : &a.len_end[lb], 1u); }
                const uint32_t tb = y.g * kTickBins + (uint32_t)tick_bin(y.S);
                tp[u] = atomicAdd(PRIV ? &s_tick[tb] : &a.tick_at[tb], 1u);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const Item& y = x[u];
                if (!y.in) continue;
                if (DBG_OK(tp[u], a.n, DBG_K_GATHER, DBG_ELEMENT)) a.binned[tp[u]] = y.S;
                if (kTrace && DBG_OK(at[u], a.n, DBG_K_GATHER, DBG_REQUEST)) a.req[at[u]] = make_uint4(y.S, y.l | y.o << 16, i0 + u, 0u);
            }
            if (kTrace) {
                if (i0 + 4u <= a.n) *reinterpret_cast<uint4*>(a.inv + i0) = make_uint4(at[0], at[1], at[2], at[3]);
                else for (uint32_t u = 0; i0 + u < a.n; ++u) a.inv[i0 + u] = at[u];
            }
        }
    };
    if (kTrace && PRIV && a.rounds > 1) {
        // a round of the trace at a time: its requests are counted once more, and the blocks take their shares of each bucket
        // and bin from the global cursors
        const uint32_t per_round = (a.n + a.rounds - 1) / a.rounds;
#pragma unroll 1
        for (uint32_t r = 0; r < a.rounds; ++r) {
            const uint32_t i_end = r + 1 == a.rounds ? a.n : (r + 1) * per_round;
            for (int i = tid; i < G * (kTickBins + kLens); i += kThreads) s_tick[i] = 0;
            __syncthreads();
#pragma unroll 1
            for (uint32_t i0 = i_next; i0 < i_end; i0 += stride) {
                Item x[4];
                read_items<SRC, FORM, false, true>(a, i0, wide, s_off, x);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (x[u].in && DBG_OK(x[u].g, G, DBG_K_GATHER, DBG_GROUP) && DBG_OK(x[u].l, kLens, DBG_K_GATHER, DBG_TABLE)) {
                        atomicAdd(&s_len[x[u].g * kLens + x[u].l], 1u);
                        atomicAdd(&s_tick[x[u].g * kTickBins + tick_bin(x[u].S)], 1u);
                    }
            }
            __syncthreads();
            join(s_len, a.len_end, G * kLens);
            join(s_tick, a.tick_at, G * kTickBins);
            __syncthreads();
            place(i_end);
            __syncthreads();
        }
    } else {
        place(a.n);
    }
    ++waits;
    if (!grid_barrier(z, waits, ABSENT(a, waits))) return;

    // ---- 3. sort
    SortSmem& sm = *reinterpret_cast<SortSmem*>(smem_raw);
    __shared__ uint32_t s_win[4][32];                 // of the block's next windows: first tick, end, first and last bin
    uint32_t n_win = 0;
    for (int g = 0; g < G; ++g) n_win += (s_off[g + 1] - s_off[g] + kWindow - 1) / kWindow;
#pragma unroll 1
    for (uint32_t j = 0;; ++j) {
        const uint32_t win = blockIdx.x + j * gridDim.x;
        if (win >= n_win) break;
        if ((j & 31u) == 0u) {
            __syncthreads();
            if (tid < 32) {
                const uint32_t mine = blockIdx.x + (j + tid) * gridDim.x;
                uint2 bins = make_uint2(0u, 0u);
                if (mine < n_win) bins = __ldcg(&a.windows[mine]);
                if (bins.y) {
                    const uint32_t first_bin = 0xFFFFFFFFu - bins.x, last_bin = bins.y - 1u;
                    s_win[0][tid] = __ldcg(&a.tick_start[first_bin]);
                    s_win[1][tid] = __ldcg(&a.tick_start[last_bin]) + __ldcg(&a.tick_cnt[last_bin]);
                    s_win[2][tid] = first_bin; s_win[3][tid] = last_bin;
                } else s_win[0][tid] = s_win[1][tid] = 0u;
            }
        }
        __syncthreads();
        const uint32_t k0 = s_win[0][j & 31u], k1 = s_win[1][j & 31u];
        if (k0 >= k1) continue;                                        // (inside a large bin)
        const int g = (int)s_win[2][j & 31u] / kTickBins, b0 = (int)s_win[2][j & 31u] - g * kTickBins, b1 = (int)s_win[3][j & 31u] - g * kTickBins;
        sort_bins(a, sm, g, b0, b1, k0, k1);
        if (kTrace) write_knots<kThreads>(a, g, k0, k1, s_off[g], s_off[g + 1] - s_off[g]);
    }
    if (kTrace) {
        for (int g = 0; g < G; ++g)                                    // (the last blocks have the fewest windows)
            if ((uint32_t)(G - 1 - g) % gridDim.x == gridDim.x - 1 - blockIdx.x)
                group_mass(a.cnt + (size_t)g * kLens, a.cum_mass + (size_t)g * (kLens + 1), s_wide);
    }
    if (kTrace || (SRC == S_TTFT && a.readback)) {
        // the last block to come here reports the flags (where a block has left, none does: what the host put there stands)
        if (tid == 0) { __threadfence(); s_item = atomicAdd(&z->done, 1u); }
        __syncthreads();
        if (s_item == gridDim.x - 1 && tid < 4) a.readback->err[tid] = __ldcg(&z->err[tid]);
    }
}

template <int SRC, int FORM>
cudaError_t launch_load(const LoadArgs& a, int sms, cudaStream_t st) {
    const bool priv = a.G <= (SRC == S_TRACE ? kPrivateGroups : kPrivateTickGroups);
    const size_t counters = priv ? (size_t)a.G * ((SRC == S_TRACE ? kLens : 0) + kTickBins) * 4 : 0;
    const size_t smem = std::max(counters, sizeof(SortSmem));
    static_assert(kTickBins % 4 == 0 && sizeof(LoadZero) % 16 == 0, "vector loads of the counters");
    auto* kernel = priv ? k_load<SRC, true, FORM> : k_load<SRC, false, FORM>;
    cudaError_t e = allow_smem((const void*)kernel, 220 * 1024);
    if (e) return e;
    // One group: four requests a thread until the multiprocessors are full.  Several: each has counters, a window and a table of
    // its own whatever the number of requests, so at least four blocks a group share that work (1,000 requests in twenty groups
    // 235 -> 54 us a load), and beyond, twice as many blocks as for one group.
    const uint32_t per_block = (a.G > 1 ? 2u : 4u) * kThreads, least = a.G > 1 ? 4u * (uint32_t)a.G : 1u;
    const uint32_t blocks = std::min(std::max((a.n + per_block - 1) / per_block, least), std::min((uint32_t)sms, kLoadBlocks));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = blocks; cfg.blockDim = kThreads; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if ((e = cudaMemsetAsync(a.z, 0, a.zero_bytes, st))) return e;
    if (((char*)a.windows < (char*)a.z || (char*)a.windows >= (char*)a.z + a.zero_bytes) &&
        (e = cudaMemsetAsync(a.windows, 0, sort_windows(a.n, a.G) * sizeof(uint2), st))) return e;
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
#ifdef DISCO_DEBUG
    LoadArgs b = a;
    if (const char* wait = std::getenv("DISCO_DEBUG_ABSENT")) b.absent = (uint32_t)std::atoi(wait);
    return cudaLaunchKernelEx(&cfg, kernel, b);
#else
    return cudaLaunchKernelEx(&cfg, kernel, a);
#endif
}

// The same tables from a length histogram and a sorted sample given by the caller (a whole trace's, of which
// the context holds a shard): one block of 1024 threads per group.
__global__ void __launch_bounds__(kThreads)
k_tables_imported(const uint32_t* __restrict__ cnt, int64_t* __restrict__ cum, const int32_t* __restrict__ F_sorted,
                  const uint32_t* __restrict__ F_off, int32_t* __restrict__ knots) {
    __shared__ unsigned long long wm[32];
    const int g = blockIdx.x;
    const uint32_t off = F_off[g], N = F_off[g + 1] - off;
    for (int k = threadIdx.x; k < kNKnots; k += blockDim.x) {
        const uint32_t at = N ? (uint32_t)(((uint64_t)k * (N - 1)) / 256u) : 0u;
        knots[g * kNKnots + k] = (N && DBG_OK(at, N, DBG_K_TABLES, DBG_ELEMENT)) ? F_sorted[off + at] : 0;
    }
    group_mass(cnt + (size_t)g * kLens, cum + (size_t)g * (kLens + 1), wm);
}

}  // namespace

DBG_TRANSLATION_UNIT()

cudaError_t run_load(const LoadArgs& a, int sms, cudaStream_t st) {
    if (a.packed) return launch_load<S_TRACE, F_PACKED>(a, sms, st);
    return a.st_ticks ? launch_load<S_TRACE, F_STAGE>(a, sms, st) : launch_load<S_TRACE, F_COLUMNS>(a, sms, st);
}
cudaError_t run_sort_ticks(const LoadArgs& a, int sms, cudaStream_t st) {
    return once_ticks(a.n, a.G, (uint32_t)sms) ? run_sort_ticks_once(a, sms, st) : launch_load<S_TICKS, F_COLUMNS>(a, sms, st);
}

cudaError_t run_sort_ttft(const LoadArgs& a, int sms, cudaStream_t st) {
    return once_ticks(a.n, a.G, (uint32_t)sms) ? run_sort_ttft_once(a, sms, st) : launch_load<S_TTFT, F_COLUMNS>(a, sms, st);
}

cudaError_t launch_tables_imported(int G, const uint32_t* cnt, int64_t* cum_mass, const int32_t* F_sorted,
                                   const uint32_t* F_off, int32_t* knots, cudaStream_t st) {
    k_tables_imported<<<G, kThreads, 0, st>>>(cnt, cum_mass, F_sorted, F_off, knots);
    return cudaGetLastError();
}

}  // namespace disco


// -----------------------------------------------------------------------------------------------------
// Sorting server TTFTs without allocating.  The scratch the sort needs (the ticks by bin, the bins' counters,
// and the radix sort's keys and counters, should it be needed) lives in a fixed array inside the library image
// instead of in cudaMalloc'd memory.  Every GPU that loads the library carries these bytes until the process
// exits, and every call on a GPU uses the same bytes.
// -----------------------------------------------------------------------------------------------------
namespace disco {
namespace {

constexpr uint32_t kNoAllocMaxN = DISCO_NOALLOC_MAX_N;
constexpr size_t kNaKeysBytes = (size_t)kNoAllocMaxN * sizeof(uint64_t);
constexpr size_t kNaCountsBytes = (256u * ((kNoAllocMaxN + 1023u) / 1024u) + 256u) * sizeof(uint32_t);   // as radix_sort_ticks sizes its grid, plus the digit totals
// words that must start at zero: the flags and the bins' counters; then the bins' starts and the offsets of the one group
// (they lie there twice: a call clears the half that the next one uses)
constexpr size_t kNaZeroOff = 2 * kNaKeysBytes + kNaCountsBytes;
constexpr size_t kNaZeroBytes = (sizeof(LoadZero) + kTickBins * 4 + kOnceWindows * 16 + 15) / 16 * 16;
static_assert(sort_windows(kNoAllocMaxN, 1) * 8 <= kOnceWindows * 16, "k_load's windows");
constexpr size_t kNaStartOff = kNaZeroOff + 2 * kNaZeroBytes;
constexpr size_t kNaOffOff = kNaStartOff + kTickBins * 4;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaOffOff + 256];

std::mutex g_na_mutex;
int g_na_sms[64] = {};                    // multiprocessors, per device ordinal
struct { bool zero[2]; int now; } g_na_half[64] = {};   // which halves are known to be zero, and which was used last
// Where the kernel reports its flags: a page of the library's own, page-locked by the first call, 64 bytes a device ordinal.  (A
// copy into pageable memory behind the kernel took 7 us of a call, the clearing in front of it 5: 100,000 values 35 us, now 27.)
alignas(4096) unsigned char g_na_report[4096];
bool g_na_unlockable = false;

}  // namespace
}  // namespace disco

extern "C" int disco_sort_ttft_ticks_noalloc(const float* server_ttft_s, uint32_t n, int32_t* sorted_ticks,
                                             void* stream) {
    using namespace disco;
    if (n > kNoAllocMaxN)
        return set_error(DISCO_EINVAL, "disco_sort_ttft_ticks_noalloc: n exceeds DISCO_NOALLOC_MAX_N (262144); "
                                       "use disco_load_trace for larger traces");
    if (n && (!server_ttft_s || !sorted_ticks)) return set_error(DISCO_EINVAL, "null array");
    if (n == 0) return 0;
    cudaStream_t st = (cudaStream_t)stream;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return set_error(DISCO_ECUDA, cudaGetErrorString(e));
    if (dev < 0 || dev >= 64) return set_error(DISCO_EINVAL, "device ordinal above 63");
    unsigned char* base;
    int sms, half;
    bool zeroed;
    int32_t* report = nullptr;
    void* report_dev = nullptr;
    {
        // In host code the array's name is only a handle; its address on the current device has to be asked for, and so has the
        // page's.  On every call: a reset of the device may move the one and takes the other away.
        std::lock_guard<std::mutex> lock(g_na_mutex);
        if ((e = cudaGetSymbolAddress((void**)&base, g_noalloc_scratch)) != cudaSuccess) return set_error(DISCO_ECUDA, cudaGetErrorString(e));
        if (!g_na_sms[dev]) {
            int count = 0;
            if ((e = cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess || count < 1)
                return set_error(DISCO_ECUDA, "cannot read the multiprocessor count of the current device");
            g_na_sms[dev] = count;
        }
        sms = g_na_sms[dev];
        unsigned char* page = g_na_report + 64 * dev;
        for (int locked = 0; !report && !g_na_unlockable; ++locked) {
            if (cudaHostGetDevicePointer(&report_dev, page, 0) == cudaSuccess) { report = (int32_t*)page; break; }
            cudaGetLastError();
            report_dev = nullptr;
            if (locked) break;
            if (cudaHostRegister(g_na_report, sizeof g_na_report, cudaHostRegisterPortable | cudaHostRegisterMapped) != cudaSuccess) {
                cudaGetLastError();
                g_na_unlockable = true;
            }
        }
        auto& h = g_na_half[dev];
        half = h.now ^= 1;
        zeroed = h.zero[half];
        h.zero[0] = h.zero[1] = false;    // (until the call has succeeded)
    }
#ifdef DISCO_DEBUG
    if (const char* few = std::getenv("DISCO_DEBUG_MULTIPROCESSORS")) sms = std::max(1, std::min(sms, std::atoi(few)));
#endif
    LoadArgs a = {};
    a.n = n; a.G = 1; a.ns = a.nd = 1;
    a.ttft = server_ttft_s;
    unsigned char *mine = base + kNaZeroOff + half * kNaZeroBytes, *next = base + kNaZeroOff + (half ^ 1) * kNaZeroBytes;
    a.z = (LoadZero*)mine; a.tick_cnt = (uint32_t*)(mine + sizeof(LoadZero));
    a.once.zeroed = zeroed; a.once.clear = (uint4*)next; a.once.clear_vecs = (uint32_t)(kNaZeroBytes / 16);
    a.readback = (LoadReadback*)report_dev;                          // (its flags alone)
    a.once.windows = (unsigned long long*)(a.tick_cnt + kTickBins);
    a.windows = (uint2*)a.once.windows;
    a.tick_start = (uint32_t*)(base + kNaStartOff);
    a.binned = (uint32_t*)base; a.sorted = sorted_ticks;
    a.zero_bytes = kNaZeroBytes;          // the array still holds the previous call's data: flags and counters must start at zero
    // Once a kernel has been queued the shared array is in use: every way out below, failures included, first
    // waits for the stream, so that a caller who retries cannot overlap kernels still writing the array.
    auto fail_after_launch = [&](cudaError_t err_code) {
        cudaStreamSynchronize(st);
        return set_error(DISCO_ECUDA, cudaGetErrorString(err_code));
    };
    int32_t h_err[4] = {0, 0, 0, 2};      // what stands where the blocks lose each other
    if (report) std::memcpy(report, h_err, sizeof h_err);
    if ((e = run_sort_ttft(a, sms, st)) != cudaSuccess) return fail_after_launch(e);
    if (!report && (e = cudaMemcpyAsync(h_err, a.z->err, sizeof h_err, cudaMemcpyDeviceToHost, st)) != cudaSuccess) return fail_after_launch(e);
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return set_error(DISCO_ECUDA, cudaGetErrorString(e));
    if (report) std::memcpy(h_err, report, sizeof h_err);
    if (h_err[3] != 2 && once_ticks(n, 1, (uint32_t)sms)) {          // (k_load clears its own half alone)
        std::lock_guard<std::mutex> lock(g_na_mutex);
        g_na_half[dev].zero[half ^ 1] = true;
    }
    if (int rc = check_debug_record()) return rc;
    if (h_err[0]) return set_error(DISCO_EINVAL, "server TTFT not finite, not positive or above 2000 s");
    if (h_err[3] == 2) return set_error(DISCO_ECUDA, "internal error: the blocks of the sort lost each other");
    if (h_err[3] == 1) {
        // a sample the bin-wise sort gives up on: radix sort, by way of the caller's output array
        uint64_t* keys_a = (uint64_t*)base;
        uint64_t* keys_b = (uint64_t*)(base + kNaKeysBytes);
        uint32_t* counts = (uint32_t*)(base + 2 * kNaKeysBytes);
        uint32_t* off = (uint32_t*)(base + kNaOffOff);
        const uint32_t h_off[2] = {0, n};
        if ((e = cudaMemcpyAsync(sorted_ticks, a.binned, (size_t)n * 4, cudaMemcpyDeviceToDevice, st)) != cudaSuccess ||
            (e = cudaMemcpyAsync(off, h_off, sizeof h_off, cudaMemcpyHostToDevice, st)) != cudaSuccess ||
            (e = radix_sort_ticks(sorted_ticks, off, 1, n, keys_a, keys_b, counts, sorted_ticks, sms, st)) != cudaSuccess)
            return fail_after_launch(e);
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return set_error(DISCO_ECUDA, cudaGetErrorString(e));
        if (int rc = check_debug_record()) return rc;
    }
    return 0;
}
