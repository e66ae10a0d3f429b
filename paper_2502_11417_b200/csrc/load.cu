// Trace ingestion on the device in one kernel: tick conversion and validation, per-group prompt-length histogram,
// internal request order (by group, then by prompt length), sort of the server-TTFT ticks (the empirical F of
// Algorithm 1), cumulative input-token mass (Eq. 3) and the quantile knots of F.
//
// One block of 1024 threads per multiprocessor, all resident at once (a cooperative launch), works in three passes with a
// wait for all blocks between them:
//   1. count: every request is checked and counted by (group, prompt length) and by (group, bin of its ticks), 128 bins an
//      octave, in counters of the block's own.  The block adds its counters to the global ones and keeps what was there
//      before: where its own requests of each bucket go within the bucket.
//   2. place: from the totals every block works out where the buckets start, then sends its requests to their places: one
//      16-byte record into the internal order and the ticks into their bin.
//   3. sort: the bins in order, about 4,096 ticks at a time, are sorted in shared memory (all ticks of a window differ in
//      few low bits), each window by one block.  A bin of more than 8,192 ticks that spans at most 2^18 values is sorted by
//      counting them; a trace that has a denser and wider one goes to the radix sort (radix.cu) instead.
//
// Bound: latency at 10^5 requests (one launch instead of eighteen), memory at 10^7: the columns are read twice (once when
// they are in host memory: then the first pass leaves a copy), 20 bytes a request are written to scattered places, the
// ticks are read and written once more.
#include "load.cuh"

#include <algorithm>
#include <mutex>

#include "scan.cuh"

namespace disco {

namespace {

constexpr int kThreads = 1024;
constexpr int kLens = kMaxPrompt + 1;
constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr uint32_t kWindow = 4096;        // a window starts with the first bin behind every 4,096th tick of its group
constexpr uint32_t kSortCap = 8192;       // ticks sorted at a time
constexpr uint32_t kCounters = 16384;     // values counted at a time
constexpr uint32_t kMaxRange = 1u << 18;  // values a dense bin may span
constexpr uint32_t kMaxCount = 1u << 24;  // ticks a dense bin may hold
constexpr int kPrivateGroups = 7;         // groups whose counters fit in shared memory (29 KB each)
constexpr int kPrivateTickGroups = 16;    // the same, counters of tick bins alone
constexpr int kUnroll = 4;                // requests a thread has in flight

enum Source { S_TRACE, S_TICKS, S_TTFT };

__device__ __forceinline__ int tick_bin(uint32_t t) {
    return t < 128u ? (int)t : (int)(__float_as_uint(__uint2float_rz(t)) >> 16) - ((127 + 7) << 7) + 128;
}
__device__ __forceinline__ uint32_t tick_bin_edge(int b) {     // smallest ticks of the bin (2^31 behind the last)
    return b < 128 ? (uint32_t)b : (uint32_t)(128 + (b & 127)) << ((b >> 7) - 1);
}

struct SortSmem {
    uint32_t a[kSortCap], b[kSortCap];                 // ticks of a window, twice; or kCounters counters
    uint16_t wcnt[kThreads / 32][256];                 // keys of each digit per warp; or the list of frequent values
    uint32_t dig[256];
    uint32_t wtot[32];
    uint32_t lo, hi, n_list;
    int bin0, bin1;
};
static_assert(kCounters == 2 * kSortCap, "the counters lie over the two key arrays");

// Waits until every block of the grid has come here `times` times.  The wait is bounded: a block that gives up sets the
// flag and goes on (the host refuses the results).
__device__ __forceinline__ void grid_barrier(LoadZero* z, uint32_t times) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&z->barrier, 1u);
        const uint32_t want = times * gridDim.x;
        uint32_t seen, tries = 0;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&z->barrier) : "memory");
        } while (seen < want && ++tries < (1u << 22));
        if (seen < want) atomicExch(&z->err[3], 2);
        __threadfence();
    }
    __syncthreads();
}

// A request of the trace (or a tick of a sample) as the two passes see it.
struct Item { uint32_t g, S, l, o; bool in; };

// First pass: reads and checks item i.
template <int SRC>
__device__ __forceinline__ Item check_item(const LoadArgs& a, uint32_t i, const uint32_t* s_off) {
    Item x = {0u, 0u, 1u, 1u, i < a.n};
    if (!x.in) return x;
    int bad = 0;
    if (SRC == S_TICKS) {
        while ((int)x.g + 1 < a.G && i >= s_off[x.g + 1]) ++x.g;
        const int32_t t = a.ticks[i];
        if (t < 0) bad = 3;
        x.S = (uint32_t)t;
    } else {
        const float t = a.ttft[i];
        uint32_t s = 0, d = 0;
        int32_t l = 1, o = 1;
        if (SRC == S_TRACE) { l = a.prompt[i]; o = a.outlen[i]; s = a.sp ? a.sp[i] : 0u; d = a.dp ? a.dp[i] : 0u; }
        if (l < 1 || l > kMaxPrompt) bad = 1;
        else if (o < 1 || o > kMaxOutput) bad = 2;
        else if (!(t > 0.0f) || !(t <= 2000.0f)) bad = 3;      // NaN fails both comparisons
        else if (SRC == S_TRACE && (s >= a.ns || d >= a.nd)) bad = 4;
        // ticks = nearest integer (ties to even) of the fp64 product, as a host llrint would give
        x.S = (uint32_t)__double2ll_rn(__dmul_rn((double)t, 1e6));
        x.g = s * a.nd + d; x.l = (uint32_t)l; x.o = (uint32_t)o;
        if (SRC == S_TTFT) x.g = 0;
    }
    if (bad) {
        if (atomicCAS(&a.z->err[0], 0, bad) == 0) a.z->err[1] = (int32_t)i;
        x.in = false;
    }
    return x;
}

// Second pass: the same item, known to be good.
template <int SRC, bool STAGE>
__device__ __forceinline__ Item read_item(const LoadArgs& a, uint32_t i, const uint32_t* s_off) {
    Item x = {0u, 0u, 1u, 1u, i < a.n};
    if (!x.in) return x;
    if (STAGE) {
        const uint32_t ln = a.st_ln[i];
        x.S = a.st_ticks[i]; x.l = ln & 0xFFFFu; x.o = ln >> 16; x.g = a.st_g[i];
    } else if (SRC == S_TICKS) {
        while ((int)x.g + 1 < a.G && i >= s_off[x.g + 1]) ++x.g;
        x.S = (uint32_t)a.ticks[i];
    } else {
        x.S = (uint32_t)__double2ll_rn(__dmul_rn((double)a.ttft[i], 1e6));
        if (SRC == S_TRACE) {
            x.l = (uint32_t)a.prompt[i]; x.o = (uint32_t)a.outlen[i];
            x.g = (a.sp ? a.sp[i] : 0u) * a.nd + (a.dp ? a.dp[i] : 0u);
        }
    }
    return x;
}

// Exclusive prefix sums of L <= 5 * kThreads counters, `base` added; emit(k, count, start).  All threads call.
template <class E>
__device__ __forceinline__ void scan_counts(const uint32_t* cnt, int L, uint32_t base, uint32_t* wtot, E emit) {
    constexpr int kPer = 5;
    const int k0 = (int)threadIdx.x * kPer;
    uint32_t c[kPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) { c[k] = k0 + k < L ? __ldcg(&cnt[k0 + k]) : 0u; sum += c[k]; }
    uint32_t run = base + block_inclusive_scan(sum, wtot, (uint32_t*)nullptr) - sum;
#pragma unroll
    for (int k = 0; k < kPer; ++k) { if (k0 + k < L) emit(k0 + k, c[k], run); run += c[k]; }
    __syncthreads();
}

// Cumulative input-token mass cum[L] = sum_{l<L} l cnt[l], L = 0 .. 4097.  All threads call.
__device__ __forceinline__ void group_mass(const uint32_t* cnt, int64_t* cum, unsigned long long* wm) {
    constexpr int kPer = 5;
    const int k0 = (int)threadIdx.x * kPer;
    uint32_t c[kPer];
    unsigned long long m = 0, total;
#pragma unroll
    for (int k = 0; k < kPer; ++k) { c[k] = k0 + k < kLens ? __ldcg(&cnt[k0 + k]) : 0u; m += (unsigned long long)(k0 + k) * c[k]; }
    unsigned long long run = block_inclusive_scan(m, wm, &total) - m;
#pragma unroll
    for (int k = 0; k < kPer; ++k) { if (k0 + k < kLens) cum[k0 + k] = (int64_t)run; run += (unsigned long long)(k0 + k) * c[k]; }
    if (threadIdx.x == 0) cum[kLens] = (int64_t)total;
    __syncthreads();
}

// Sorts `count` <= kSortCap ticks from src (all of them in [lo, lo + 2^bits)) into out: stable counting passes of at most
// eight bits in shared memory, a warp's 256 keys at a time with the ranks from ballots.
__device__ __forceinline__ void sort_window(SortSmem& sm, const uint32_t* src, uint32_t count, uint32_t lo, int bits, int32_t* out) {
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    if (bits == 0) {
        for (uint32_t i = tid; i < count; i += kThreads) out[i] = (int32_t)lo;
        return;
    }
    uint32_t *from = sm.a, *to = sm.b;
    for (uint32_t i = tid; i < count; i += kThreads) from[i] = __ldcg(&src[i]) - lo;
    const int passes = (bits + 7) / 8, d_bits = (bits + passes - 1) / passes, digits = 1 << d_bits;
    const int rounds = (int)((min(count, 256u) + 31u) / 32u), warps = (int)((count + 255u) / 256u);
    for (int p = 0; p < passes; ++p) {
        const int shift = p * d_bits;
        for (int i = tid; i < warps * 256; i += kThreads) (&sm.wcnt[0][0])[i] = 0;
        __syncthreads();
        uint32_t key[8], place[8];                    // place: digit | rank among the warp's equal digits so far << 8
        if (w < warps) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (j >= rounds) break;
                const uint32_t i = w * 256u + j * 32u + lane;
                const bool live = i < count;
                key[j] = live ? from[i] : 0u;
                const uint32_t d = (key[j] >> shift) & (uint32_t)(digits - 1);
                uint32_t peers = __ballot_sync(FULL, live);
                for (int b = 0; b < d_bits; ++b) {
                    const uint32_t bal = __ballot_sync(FULL, (d >> b) & 1u);
                    peers &= ((d >> b) & 1u) ? bal : ~bal;
                }
                const uint32_t below = __popc(peers & ((1u << lane) - 1u));
                uint32_t before = 0;
                if (live) before = sm.wcnt[w][d];
                __syncwarp();
                if (live && below == 0) sm.wcnt[w][d] = (uint16_t)(before + __popc(peers));
                __syncwarp();
                place[j] = d | (before + below) << 8;
            }
        }
        __syncthreads();
        // where each digit starts, and each warp's keys of it
        uint32_t total = 0;
        if (tid < digits) for (int k = 0; k < warps; ++k) { const uint32_t c = sm.wcnt[k][tid]; sm.wcnt[k][tid] = (uint16_t)total; total += c; }
        const uint32_t incl = block_inclusive_scan(tid < digits ? total : 0u, sm.wtot, (uint32_t*)nullptr);
        if (tid < digits) sm.dig[tid] = incl - total;
        __syncthreads();
        if (w < warps) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (j >= rounds) break;
                const uint32_t i = w * 256u + j * 32u + lane;
                if (i < count) {
                    const uint32_t d = place[j] & 255u, at = sm.dig[d] + sm.wcnt[w][d] + (place[j] >> 8);
                    if (DBG_OK(at, count, DBG_K_RADIX, DBG_ELEMENT)) to[at] = key[j];
                }
            }
        }
        __syncthreads();
        uint32_t* t = from; from = to; to = t;
    }
    for (uint32_t i = tid; i < count; i += kThreads) out[i] = (int32_t)(from[i] + lo);
}

// Sorts a dense bin by counting its values.  Returns false where that would take too long.
__device__ __forceinline__ bool sort_dense(SortSmem& sm, const uint32_t* src, uint32_t count, int32_t* out) {
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    if (tid == 0) { sm.lo = 0xFFFFFFFFu; sm.hi = 0u; }
    __syncthreads();
    uint32_t mn = 0xFFFFFFFFu, mx = 0u;
    for (uint32_t i = tid; i < count; i += kThreads) { const uint32_t t = __ldcg(&src[i]); mn = min(mn, t); mx = max(mx, t); }
    mn = __reduce_min_sync(FULL, mn); mx = __reduce_max_sync(FULL, mx);
    if (lane == 0) { atomicMin(&sm.lo, mn); atomicMax(&sm.hi, mx); }
    __syncthreads();
    const uint32_t lo = sm.lo, range = sm.hi - lo + 1u;
    if (range == 1u) {
        for (uint32_t i = tid; i < count; i += kThreads) out[i] = (int32_t)lo;
        return true;
    }
    if (range > kMaxRange || count > kMaxCount) return false;
    uint32_t* n_of = sm.a;                                            // kCounters of them
    uint16_t* list = &sm.wcnt[0][0];
    constexpr uint32_t kOften = 4096;                                 // such values are written by the whole block
    uint32_t done = 0;
    for (uint32_t r0 = 0; r0 < range; r0 += kCounters) {
        for (uint32_t i = tid; i < kCounters; i += kThreads) n_of[i] = 0;
        if (tid == 0) sm.n_list = 0;
        __syncthreads();
        for (uint32_t i = tid; i < count; i += kThreads) {
            const uint32_t v = __ldcg(&src[i]) - lo - r0;
            if (v < kCounters) atomicAdd(&n_of[v], 1u);
        }
        __syncthreads();
        // a thread's sixteen values, then where they start
        constexpr uint32_t kPer = kCounters / kThreads;
        uint32_t sum = 0, total;
        for (uint32_t k = 0; k < kPer; ++k) sum += n_of[tid * kPer + k];
        uint32_t run = done + block_inclusive_scan(sum, sm.wtot, &total) - sum;
        // a warp writes its threads' values one thread after another, 32 copies at a time
        for (int t = 0; t < 32; ++t) {
            uint32_t at = __shfl_sync(FULL, run, t);
            if (__shfl_sync(FULL, sum, t) == 0u) continue;
            for (uint32_t k = 0; k < kPer; ++k) {
                const uint32_t v = (uint32_t)(w * 32 + t) * kPer + k, c = n_of[v];
                if (c > kOften) {
                    if (lane == 0) { const uint32_t e = atomicAdd(&sm.n_list, 1u); if (DBG_OK(e, 8192, DBG_K_RADIX, DBG_SLOT)) list[e] = (uint16_t)v; }
                } else {
                    for (uint32_t j = lane; j < c; j += 32) out[at + j] = (int32_t)(lo + r0 + v);
                }
                at += c;
            }
        }
        __syncthreads();
        for (uint32_t e = 0; e < sm.n_list; ++e) {                    // (at most kMaxCount / kOften of them)
            const uint32_t v = list[e];
            // where it starts: the counters in front of it
            uint32_t part = 0;
            for (uint32_t k = tid; k < v; k += kThreads) part += n_of[k];
            uint32_t before;
            block_inclusive_scan(part, sm.wtot, &before);
            const uint32_t c = n_of[v];
            for (uint32_t j = tid; j < c; j += kThreads) out[done + before + j] = (int32_t)(lo + r0 + v);
            __syncthreads();
        }
        done += total;
        __syncthreads();
    }
    return true;
}

template <int SRC, bool PRIV, bool STAGE>
__global__ void __launch_bounds__(kThreads, 1)
k_load(const __grid_constant__ LoadArgs a) {
    constexpr bool kTrace = SRC == S_TRACE;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_off[kMaxGroups + 1];        // group offsets in the internal order
    __shared__ unsigned long long s_wide[32];
    __shared__ uint32_t s_wtot[32];
    __shared__ unsigned long long s_sum[kMaxGroups];
    __shared__ uint32_t s_max, s_item;
    const int G = a.G, tid = threadIdx.x, lane = tid & 31;
    LoadZero* z = a.z;
    uint32_t* s_len = (uint32_t*)smem_raw;                             // [G][kLens]
    uint32_t* s_tick = s_len + (kTrace ? G * kLens : 0);               // [G][kTickBins]
    uint32_t waits = 0;

    // ---- 1. count
    if (PRIV) for (int i = tid; i < (kTrace ? G * kLens : 0) + G * kTickBins; i += kThreads) s_len[i] = 0;
    if (SRC == S_TICKS) for (int g = tid; g <= G; g += kThreads) s_off[g] = a.off[g];
    for (int g = tid; g < G; g += kThreads) s_sum[g] = 0;
    if (tid == 0) s_max = 0;
    __syncthreads();
    const uint32_t stride = gridDim.x * kThreads, i_first = blockIdx.x * kThreads + tid;
    uint32_t tok[kPrivateGroups] = {};                                 // output tokens per group
    uint32_t longest = 0;
    for (uint32_t i0 = i_first; i0 < a.n; i0 += kUnroll * stride) {
        Item x[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const uint32_t i = i0 + u * stride;
            x[u] = check_item<SRC>(a, i, s_off);
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const Item& y = x[u];
            if (!y.in || !DBG_OK(y.g, G, DBG_K_INGEST, DBG_GROUP) || !DBG_OK(y.l, kLens, DBG_K_INGEST, DBG_TABLE)) continue;
            const int tb = tick_bin(y.S);
            if (!DBG_OK(tb, kTickBins, DBG_K_INGEST, DBG_BIN)) continue;
            if (STAGE) {
                const uint32_t i = i0 + u * stride;
                a.st_ticks[i] = y.S; a.st_ln[i] = y.l | y.o << 16; a.st_g[i] = (uint8_t)y.g;
            }
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
                    for (int g = 0; g < kPrivateGroups; ++g) tok[g] += (int)y.g == g ? y.o : 0u;    // (at most 2^21 requests a thread)
                }
            }
        }
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
    // the block's counters join the global ones; what it finds there is where its own requests go within the bucket
    if (PRIV) {
        auto join = [&](uint32_t* mine, uint32_t* all, int count) {
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
        if (kTrace) join(s_len, a.cnt, G * kLens);
        join(s_tick, a.tick_cnt, G * kTickBins);
    }
    grid_barrier(z, ++waits);

    // ---- 2. place
    const int32_t bad = __ldcg(&z->err[0]);
    // group sizes: the sum of their tick counts
    uint32_t base = 0;
    for (int g = 0; g < G; ++g) {
        if (SRC != S_TICKS && tid == 0) s_off[g] = base;
        const bool mine = (int)(blockIdx.x % (uint32_t)G) == g || gridDim.x < (uint32_t)G;    // the blocks that write the group's tables
        uint32_t in_group = 0;
        auto ticks_at = [&](int k, uint32_t c, uint32_t start) {
            const size_t at = (size_t)g * kTickBins + k;
            if (PRIV) s_tick[at] += start;
            if (mine) { a.tick_start[at] = start; if (!PRIV && blockIdx.x < (uint32_t)G) a.tick_at[at] = start; }
            if (k == kTickBins - 1) s_item = start + c - base;
        };
        scan_counts(a.tick_cnt + (size_t)g * kTickBins, kTickBins, base, s_wtot, ticks_at);
        in_group = s_item;
        if (kTrace) {
            scan_counts(a.cnt + (size_t)g * kLens, kLens, base, s_wtot, [&](int k, uint32_t c, uint32_t start) {
                const size_t at = (size_t)g * kLens + k;
                if (PRIV) { s_len[at] += start; if (mine) a.len_end[at] = start + c; }
                else if (mine && blockIdx.x < (uint32_t)G) a.len_end[at] = start;      // the cursor, which ends up there
            });
            if (mine) group_mass(a.cnt + (size_t)g * kLens, a.cum_mass + (size_t)g * (kLens + 1), s_wide);
        }
        base += in_group;
        __syncthreads();
    }
    if (SRC != S_TICKS && tid == 0) s_off[G] = base;
    __syncthreads();
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
    if (bad) {                                         // a rejected trace: nothing is placed
        if (kTrace && blockIdx.x == 0 && tid < 4) a.readback->err[tid] = __ldcg(&z->err[tid]);
        return;
    }
    if (!PRIV) grid_barrier(z, ++waits);               // the cursors are complete
    for (uint32_t i0 = i_first; i0 < a.n; i0 += kUnroll * stride) {
        Item x[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const uint32_t i = i0 + u * stride;
            x[u] = read_item<SRC, STAGE>(a, i, s_off);
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const Item& y = x[u];
            const uint32_t i = i0 + u * stride;
            if (!y.in || !DBG_OK(y.g, G, DBG_K_GATHER, DBG_GROUP) || !DBG_OK(y.l, kLens, DBG_K_GATHER, DBG_TABLE)) continue;
            const uint32_t tb = y.g * kTickBins + (uint32_t)tick_bin(y.S);
            const uint32_t tp = atomicAdd(PRIV ? &s_tick[tb] : &a.tick_at[tb], 1u);
            if (DBG_OK(tp, a.n, DBG_K_GATHER, DBG_ELEMENT)) a.binned[tp] = y.S;
            if (kTrace) {
                const uint32_t lb = y.g * kLens + y.l;
                const uint32_t at = atomicAdd(PRIV ? &s_len[lb] : &a.len_end[lb], 1u);
                if (!DBG_OK(at, a.n, DBG_K_GATHER, DBG_REQUEST)) continue;
                a.req[at] = make_uint4(y.S, y.l | y.o << 16, i, 0u);
                if (a.inv) a.inv[i] = at;
            }
        }
    }
    grid_barrier(z, ++waits);

    // ---- 3. sort
    SortSmem& sm = *reinterpret_cast<SortSmem*>(smem_raw);
    for (;;) {
        __syncthreads();
        if (tid == 0) s_item = atomicAdd(&z->ticket, 1u);
        __syncthreads();
        uint32_t win = s_item;
        int g = 0;
        for (; g < G; ++g) {
            const uint32_t here = (s_off[g + 1] - s_off[g] + kWindow - 1) / kWindow;
            if (win < here) break;
            win -= here;
        }
        if (g == G) break;
        const uint32_t first = s_off[g], N = s_off[g + 1] - first;
        const uint32_t* start = a.tick_start + (size_t)g * kTickBins;
        // the window's bins: those that hold ticks and start in [first + win * kWindow, ... + kWindow)
        if (tid == 0) { sm.bin0 = kTickBins; sm.bin1 = -1; }
        __syncthreads();
        const uint32_t x0 = first + win * kWindow, x1 = x0 + kWindow;
        const uint32_t* counts = a.tick_cnt + (size_t)g * kTickBins;
        int b_min = kTickBins, b_max = -1;
        for (int b = tid; b < kTickBins; b += kThreads) {
            const uint32_t s = __ldcg(&start[b]), c = __ldcg(&counts[b]);
            if (c && s >= x0 && s < x1) { b_min = min(b_min, b); b_max = max(b_max, b); }
        }
        if (b_max >= 0) { atomicMin(&sm.bin0, b_min); atomicMax(&sm.bin1, b_max); }
        __syncthreads();
        const int b0 = sm.bin0, b1 = sm.bin1;
        if (b1 < 0) continue;                                          // (inside a large bin)
        const uint32_t k0 = __ldcg(&start[b0]), k2 = __ldcg(&start[b1]), k1 = k2 + __ldcg(&counts[b1]);
        const uint32_t lo = tick_bin_edge(b0);
        auto bits_of = [](uint32_t range) { return range <= 1u ? 0 : 32 - __clz((int)(range - 1u)); };
        if (k1 - k0 <= kSortCap) {
            sort_window(sm, a.binned + k0, k1 - k0, lo, bits_of(tick_bin_edge(b1 + 1) - lo), a.sorted + k0);
        } else {                                                       // the last bin is a large one: the others first
            if (k2 > k0) {
                sort_window(sm, a.binned + k0, k2 - k0, lo, bits_of(tick_bin_edge(b1) - lo), a.sorted + k0);
                __syncthreads();
            }
            if (!sort_dense(sm, a.binned + k2, k1 - k2, a.sorted + k2) && tid == 0) atomicExch(&z->err[3], 1);
        }
        __syncthreads();
        if (kTrace) {
            // the knots K_g[k] = sorted_g[(k (N_g - 1)) / 256] that lie in the window
            for (int k = tid; k < kNKnots; k += kThreads) {
                const uint32_t at = first + (uint32_t)(((uint64_t)k * (N - 1)) / 256u);
                if (at >= k0 && at < k1) {
                    const int32_t v = __ldcg(&a.sorted[at]);
                    a.knots[g * kNKnots + k] = v;
                    if (k == kNKnots - 1) a.readback->knot_max[g] = v;
                }
            }
        }
    }
    if (kTrace) {
        // the last block to come here reports the flags
        if (tid == 0) { __threadfence(); s_item = atomicAdd(&z->pad, 1u); }
        __syncthreads();
        if (s_item == gridDim.x - 1 && tid < 4) a.readback->err[tid] = __ldcg(&z->err[tid]);
    }
}

template <int SRC, bool STAGE>
cudaError_t launch_load(const LoadArgs& a, int sms, cudaStream_t st) {
    const bool priv = a.G <= (SRC == S_TRACE ? kPrivateGroups : kPrivateTickGroups);
    const size_t counters = priv ? (size_t)a.G * ((SRC == S_TRACE ? kLens : 0) + kTickBins) * 4 : 0;
    const size_t smem = std::max(counters, sizeof(SortSmem));
    auto* kernel = priv ? k_load<SRC, true, STAGE> : k_load<SRC, false, STAGE>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
    if (e) return e;
    // a request a thread until the multiprocessors are full
    const uint32_t blocks = std::max<uint32_t>(1u, std::min<uint32_t>((a.n + kThreads - 1) / kThreads, (uint32_t)sms));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = blocks; cfg.blockDim = kThreads; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a);
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
    return a.st_ticks ? launch_load<S_TRACE, true>(a, sms, st) : launch_load<S_TRACE, false>(a, sms, st);
}
cudaError_t run_sort_ticks(const LoadArgs& a, int sms, cudaStream_t st) { return launch_load<S_TICKS, false>(a, sms, st); }
cudaError_t run_sort_ttft(const LoadArgs& a, int sms, cudaStream_t st) { return launch_load<S_TTFT, false>(a, sms, st); }

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
constexpr size_t kNaZeroOff = 2 * kNaKeysBytes + kNaCountsBytes;
constexpr size_t kNaZeroBytes = sizeof(LoadZero) + kTickBins * 4;
constexpr size_t kNaStartOff = kNaZeroOff + kNaZeroBytes;
constexpr size_t kNaOffOff = kNaStartOff + kTickBins * 4;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaOffOff + 256];

std::mutex g_na_mutex;
unsigned char* g_na_base[64] = {};        // device address of the scratch array, per device ordinal
int g_na_sms[64] = {};                    // multiprocessors, per device ordinal

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
    int sms;
    {
        // In host code the array's name is only a handle; its address on the current device has to be asked for.
        std::lock_guard<std::mutex> lock(g_na_mutex);
        if (!g_na_base[dev]) {
            int count = 0;
            if ((e = cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess || count < 1)
                return set_error(DISCO_ECUDA, "cannot read the multiprocessor count of the current device");
            e = cudaGetSymbolAddress((void**)&g_na_base[dev], g_noalloc_scratch);
            if (e != cudaSuccess) { g_na_base[dev] = nullptr; return set_error(DISCO_ECUDA, cudaGetErrorString(e)); }
            g_na_sms[dev] = count;
        }
        base = g_na_base[dev];
        sms = g_na_sms[dev];
    }
    LoadArgs a = {};
    a.n = n; a.G = 1; a.ns = a.nd = 1;
    a.ttft = server_ttft_s;
    a.z = (LoadZero*)(base + kNaZeroOff); a.tick_cnt = (uint32_t*)(base + kNaZeroOff + sizeof(LoadZero));
    a.tick_start = (uint32_t*)(base + kNaStartOff);
    a.binned = (uint32_t*)base; a.sorted = sorted_ticks;
    // the array still holds the previous call's data: flags and counters must start at zero
    if ((e = cudaMemsetAsync(a.z, 0, kNaZeroBytes, st)) != cudaSuccess) return set_error(DISCO_ECUDA, cudaGetErrorString(e));
    // Once a kernel has been queued the shared array is in use: every way out below, failures included, first
    // waits for the stream, so that a caller who retries cannot overlap kernels still writing the array.
    auto fail_after_launch = [&](cudaError_t err_code) {
        cudaStreamSynchronize(st);
        return set_error(DISCO_ECUDA, cudaGetErrorString(err_code));
    };
    if ((e = run_sort_ttft(a, sms, st)) != cudaSuccess) return fail_after_launch(e);
    int32_t h_err[4] = {0, 0, 0, 0};
    if ((e = cudaMemcpyAsync(h_err, a.z->err, sizeof h_err, cudaMemcpyDeviceToHost, st)) != cudaSuccess) return fail_after_launch(e);
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return set_error(DISCO_ECUDA, cudaGetErrorString(e));
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
