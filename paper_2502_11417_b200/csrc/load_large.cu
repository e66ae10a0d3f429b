// Trace ingestion of large traces: the same results as k_load's (load.cu), by six kernels that send the requests to their
// places in two steps.
//
// Sent straight to its place in the internal order, a record of 16 bytes meets a line that has left L2 before its neighbours
// come (the blocks' shares of all buckets are open at once), and memory reads and writes the line again: 16 M scattered
// stores take 93 us within 64 MB and 560 within 256.  Here a tile of 8,192 requests first takes places at the ends of some
// thousand buckets of neighbouring prompt lengths, and of neighbouring bins of ticks: only the buckets' last lines are open.
// Then a block puts one bucket's records in order, within the few hundred KB that the bucket takes.
//   k_count    checks the requests and counts them by (group, prompt length) and (group, bin of ticks);
//   k_plan     where every length's and bin's requests go, and which bucket they belong to;
//   k_records  tiles to buckets, by way of shared memory, so that the records of a bucket leave side by side;
//   k_ticks    the same for the ticks;
//   k_order    the records of a bucket by length;
//   k_sort     the ticks of a bucket ascending.
// Nothing waits for another block.  Records and ticks need nothing of each other: k_ticks begins where a block of k_records has ended, and
// so do k_order behind k_ticks and k_sort behind k_order, each of which waits for the kernel in front before it ends (a step of 4 M requests
// 297 -> 283 us, of 16 M in six groups 1,090 -> 1,057: the last tiles and buckets of a kernel leave most multiprocessors idle).
//
// Bound: memory and shared-memory atomics.  16 M requests in six groups: k_load 855 us, these, one after another, 550 (count 58, plan 13, records 149,
// ticks 109, order 105, sort 114; 527 as they overlap); 4 M in one group 213 and 138.  Below, k_load's scattered stores
// still meet their lines in L2, and it has one launch: steps with either, in one group, 1.5 M requests 177 us and 178, 2 M 199 and 199,
// 2.5 M 228 and 216, 3 M 261 and 231, 3.4 M 292 and 234; in six 205 and 208, 234 and 229, 268 and 261, 297 and 278, 338 and 290; from pageable
// arrays 2 M 738 and 737, 3.4 M 1,142 and 1,107.  From page-locked columns, which k_count reads, 2 M 767 and 808, 3 M 1,100 and 1,098, 3.4 M 1,244
// and 1,230.  Above 2^24 requests the tables
// of buckets do not fit in a block's shared memory, above seven groups the counters.
#include <algorithm>

#include "ingest.cuh"

namespace disco {

namespace {

constexpr int kPer = 8;                                // requests a thread has of a tile
constexpr uint32_t kTile = kThreads * kPer;
constexpr uint32_t kBigCap = 16384;                    // ticks sorted at a time
static_assert(2 * kTickShare <= kBigCap, "a share of ticks, and the last bin of a bucket");

__device__ __forceinline__ bool refused(const LoadArgs& a) { return __ldcg(&a.z->err[0]) != 0; }

__device__ __forceinline__ bool columns_aligned(const LoadArgs& a) {
    const auto aligned = [](const void* p, uintptr_t k) { return ((uintptr_t)p & (k - 1)) == 0; };
    return aligned(a.ttft, 16) && aligned(a.prompt, 16) && aligned(a.outlen, 16) && aligned(a.sp, 4) && aligned(a.dp, 4);
}

template <int FORM>
__global__ void __launch_bounds__(kThreads, 1)
k_count(const __grid_constant__ LoadArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned long long s_sum[kPrivateGroups];
    __shared__ uint32_t s_max, s_n[kPrivateGroups];
    const int G = a.G, tid = threadIdx.x, lane = tid & 31;
    uint32_t* s_tick = (uint32_t*)smem_raw;            // [G][kTickBins]
    uint32_t* s_len = s_tick + G * kTickBins;          // [G][kLens]
    for (int i = tid; i < G * (kLens + kTickBins); i += kThreads) s_tick[i] = 0;
    if (tid < G) { s_sum[tid] = 0; s_n[tid] = 0; }
    if (tid == 0) s_max = 0;
    __syncthreads();
    const bool wide = columns_aligned(a);
    const uint32_t stride = gridDim.x * kThreads * 4u;
    uint32_t tok[kPrivateGroups] = {}, longest = 0;    // (a thread has fewer than 2^19 requests of 8,192 tokens at most)
    uint32_t i0 = (blockIdx.x * kThreads + tid) * 4u;
    Raw ahead;                                         // read while the requests in front are counted
    if (i0 < a.n) read_raw<S_TRACE, FORM, true>(a, i0, wide, ahead);
#pragma unroll 1
    for (; i0 < a.n; i0 += stride) {
        const Raw r = ahead;
        if (i0 + stride < a.n) read_raw<S_TRACE, FORM, true>(a, i0 + stride, wide, ahead);
        Item x[4];
        to_items<S_TRACE, FORM, true>(a, i0, r, nullptr, x);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const Item& y = x[u];
            if (!y.in || !DBG_OK(y.g, G, DBG_K_INGEST, DBG_GROUP) || !DBG_OK(y.l, kLens, DBG_K_INGEST, DBG_TABLE)) continue;
            const int tb = tick_bin(y.S);
            if (!DBG_OK(tb, kTickBins, DBG_K_INGEST, DBG_BIN)) continue;
            atomicAdd(&s_len[y.g * kLens + y.l], 1u);
            atomicAdd(&s_tick[y.g * kTickBins + tb], 1u);
            longest = max(longest, y.o);
#pragma unroll
            for (int g = 0; g < kPrivateGroups; ++g) tok[g] += (int)y.g == g ? y.o : 0u;
        }
        if (FORM == F_STAGE) stage_items(a, i0, x);
    }
    longest = __reduce_max_sync(FULL, longest);
    if (lane == 0 && longest) atomicMax(&s_max, longest);
#pragma unroll
    for (int g = 0; g < kPrivateGroups; ++g) {
        if (g >= G) break;
        unsigned long long v = tok[g];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
        if (lane == 0 && v) atomicAdd(&s_sum[g], v);
    }
    __syncthreads();
    // requests per group, which the next kernel's blocks start from
#pragma unroll 4
    for (int i = tid; i < G * kTickBins; i += kThreads) {
        const uint32_t sum = __reduce_add_sync(FULL, s_tick[i]);
        if (lane == 0 && sum) atomicAdd(&s_n[i / kTickBins], sum);
    }
    __syncthreads();
    if (tid < G && s_n[tid]) atomicAdd(&a.z->grp_n[tid], s_n[tid]);
    static_assert(kTickBins % 32 == 0, "a warp's counters are of one group");
    if (tid < G && s_sum[tid]) atomicAdd((unsigned long long*)&a.z->grp_sum_n[tid], s_sum[tid]);
    if (tid == 0 && s_max) atomicMax(&a.z->max_n, s_max);
    for (int i = tid; i < G * kTickBins; i += kThreads) if (s_tick[i]) atomicAdd(&a.tick_cnt[i], s_tick[i]);
    for (int i = tid; i < G * kLens; i += kThreads) if (s_len[i]) atomicAdd(&a.cnt[i], s_len[i]);
}

// A block for each group's prompt lengths, and one for its bins of ticks.  A bucket starts with the first length behind every
// rec_share-th request of the group, or the first bin behind every tick_share-th tick; but a length or bin of more than that has
// a bucket to itself (these have odd numbers).  Bound: latency.
constexpr int kPlanBuckets = (int)std::max(kRecBuckets, kTickBuckets);
__global__ void __launch_bounds__(kThreads)
k_plan(const __grid_constant__ LoadArgs a) {
    extern __shared__ __align__(16) uint32_t s_first[];                // [kPlanBuckets] first member, then [kPlanBuckets] last
    __shared__ uint32_t s_n[kPrivateGroups], s_wtot[32];
    __shared__ unsigned long long s_wide[32];
    const int G = a.G, tid = threadIdx.x, g = (int)blockIdx.x >> 1;
    const bool ticks = blockIdx.x & 1;
    uint32_t* s_last = s_first + kPlanBuckets;
    // four neighbouring lengths or bins a thread (no request has length 0)
    const int first = ticks ? 0 : 1, count = ticks ? kTickBins : kMaxPrompt, width = ticks ? kTickBins : kLens;
    const uint32_t* cnt = (ticks ? a.tick_cnt : a.cnt) + (size_t)g * width;
    const int k0 = first + tid * 4;
    static_assert(4 * kThreads >= kMaxPrompt && 4 * kThreads >= kTickBins, "four to a thread");
    grid_dependency_wait();
    uint32_t c[4], own = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) { c[u] = tid * 4 + u < count ? __ldcg(&cnt[k0 + u]) : 0u; own += c[u]; }
    if (refused(a)) {
        if (blockIdx.x == 0 && tid < 4) a.readback->err[tid] = __ldcg(&a.z->err[tid]);
        return;
    }
    if (tid < G) s_n[tid] = __ldcg(&a.z->grp_n[tid]);
    for (int i = tid; i < kPlanBuckets; i += kThreads) { s_first[i] = 0xFFFFFFFFu; s_last[i] = 0; }
    __syncthreads();
    uint32_t off = 0, id0 = 0;                                         // requests and buckets of the groups in front
    const uint32_t share = ticks ? a.large.tick_share : a.large.rec_share;
    auto ids_of = [&](uint32_t n) { return (n + share - 1u) / share * 2u; };
    for (int h = 0; h < g; ++h) { off += s_n[h]; id0 += ids_of(s_n[h]); }
    const uint32_t ids = ids_of(s_n[g]);
    uint32_t at = block_inclusive_scan(own, s_wtot, (uint32_t*)nullptr) - own;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (tid * 4 + u >= count) break;
        const int k = k0 + u;
        const uint32_t id = at / share * 2u + (c[u] > share ? 1u : 0u);
        if (c[u] && DBG_OK(id, ids, DBG_K_TABLES, DBG_TABLE)) { atomicMin(&s_first[id], (uint32_t)k); atomicMax(&s_last[id], (uint32_t)k); }
        (ticks ? a.large.tick_bucket : a.large.rec_bucket)[(size_t)g * width + k] = (uint16_t)(id0 + id);
        if (ticks) a.tick_start[(size_t)g * kTickBins + k] = off + at;
        else a.len_end[(size_t)g * kLens + k] = off + at + c[u];
        at += c[u];
    }
    if (!ticks && tid == 0) a.len_end[(size_t)g * kLens] = off;
    __syncthreads();
    // where the buckets start, at their first member (written above by a thread of this block), and what they hold
    const uint32_t last_id = g == G - 1 ? (ticks ? a.large.n_tick : a.large.n_rec) - id0 : ids;        // (the last are buckets that no group has)
    for (uint32_t i = tid; i < last_id; i += kThreads) {
        const bool some = i < ids && s_first[i] <= s_last[i];
        const uint32_t m0 = (uint32_t)(g * width) + s_first[i], m1 = (uint32_t)(g * width) + s_last[i];
        if (ticks) {
            const uint32_t start = some ? a.tick_start[m0] : 0u;
            if (some) a.large.tick_at[id0 + i] = start;
            a.large.tick_jobs[id0 + i] = some ? make_uint4(start, a.tick_start[m1] + __ldcg(&a.tick_cnt[m1]), m0, m1) : make_uint4(0u, 0u, 0u, 0u);
        } else {
            if (some) a.large.rec_at[id0 + i] = a.len_end[m0 - 1];
            a.large.rec_members[id0 + i] = some ? make_uint2(m0, m1) : make_uint2(1u, 0u);
        }
    }
    if (ticks) return;
    // cumulative input-token mass cum[L] = sum_{l<L} l cnt[l], L = 0 .. 4097
    unsigned long long mass = 0, total;
#pragma unroll
    for (int u = 0; u < 4; ++u) mass += (unsigned long long)(k0 + u) * c[u];
    unsigned long long run = block_inclusive_scan(mass, s_wide, &total) - mass;
    int64_t* cum = a.cum_mass + (size_t)g * (kLens + 1);
#pragma unroll
    for (int u = 0; u < 4; ++u) { cum[k0 + u] = (int64_t)run; run += (unsigned long long)(k0 + u) * c[u]; }
    if (tid == 0) { cum[0] = 0; cum[kLens] = (int64_t)total; }
    static_assert(4 * kThreads == kMaxPrompt, "every length has a thread");
    const uint32_t N = s_n[g];
    if (tid == 0) {
        const uint64_t sum = __ldcg((const unsigned long long*)&a.z->grp_sum_n[g]);
        a.readback->ng[g] = N; a.readback->grp_sum_n[g] = sum; a.readback->grp_off[g] = off;
        a.grp_off[g] = off;
        a.fin_totals[g] = sum; a.fin_totals[G + g] = N;
        if (N == 0) a.readback->knot_max[g] = 0;
        if (g == G - 1) { a.grp_off[G] = off + N; a.readback->grp_off[G] = off + N; a.readback->max_n = __ldcg(&a.z->max_n); }
    }
    if (N == 0) for (int k = tid; k < kNKnots; k += kThreads) a.knots[g * kNKnots + k] = 0;
}

// Tiles to buckets.  (Straight from the registers, a store of 16 bytes a lane, the records took 366 us instead of 150 at 16 M;
// tiles of 4,096 ticks, two blocks to a multiprocessor, 141 instead of 111: half the ticks to a run; of 16,384, 110.)  A tile's requests are counted by bucket in shared memory, its shares of the buckets taken from global
// cursors, and what goes to one bucket is brought side by side in shared memory before it leaves.  The next tile is read while
// one leaves.
template <int FORM>
__device__ __forceinline__ void read_tile(const LoadArgs& a, uint32_t t0, uint32_t end, bool wide, Raw (&r)[kPer / 4]) {
#pragma unroll
    for (int q = 0; q < kPer / 4; ++q) {
        const uint32_t i0 = t0 + (uint32_t)(q * kThreads + (int)threadIdx.x) * 4u;
        if (i0 < end) read_raw<S_TRACE, FORM, false>(a, i0, wide, r[q]);
    }
}
// Ticks of a tile, whole vectors: as many to each block (4 M in one group 29.4 us -> 26.5, in six 31.3 -> 28.3, 16 M 112 -> 109; the same for
// records, whose kernel then spills more: 16 M 149 -> 156).
__device__ __forceinline__ uint32_t even_tile(uint32_t n) {
    const uint32_t tiles = gridDim.x * ((n - 1u) / (gridDim.x * kTile) + 1u);
    return ((n - 1u) / tiles + 4u) / 4u * 4u;
}

// Exclusive prefix sums over `count` counters, vectors of four (those behind the last are zero), and the tile's shares from the
// cursors: start[i] becomes the place in the tile's order, to[i] what to add to it for the place in the bucket.
__device__ __forceinline__ void take_shares(uint32_t* start, uint32_t* to, uint32_t count, uint32_t* cursors, uint32_t* wtot) {
    uint32_t carry = 0;
    for (uint32_t k0 = 0; k0 < count; k0 += 4 * kThreads) {
        const uint32_t k = k0 + threadIdx.x * 4u;
        uint4 c = make_uint4(0u, 0u, 0u, 0u), at = c;
        if (k < count) c = *reinterpret_cast<uint4*>(start + k);
        if (c.x) at.x = atomicAdd(&cursors[k], c.x);
        if (c.y) at.y = atomicAdd(&cursors[k + 1], c.y);
        if (c.z) at.z = atomicAdd(&cursors[k + 2], c.z);
        if (c.w) at.w = atomicAdd(&cursors[k + 3], c.w);
        const uint32_t own = c.x + c.y + c.z + c.w;
        uint32_t total;
        const uint32_t x = carry + block_inclusive_scan(own, wtot, &total) - own, y = x + c.x, z = y + c.y, w = z + c.z;
        if (k < count) {
            *reinterpret_cast<uint4*>(start + k) = make_uint4(x, y, z, w);
            *reinterpret_cast<uint4*>(to + k) = make_uint4(at.x - x, at.y - y, at.z - z, at.w - w);
        }
        carry += total;
        if (k0 + 4 * kThreads < count) __syncthreads();
    }
}
__host__ __device__ constexpr uint32_t whole_vectors(uint32_t n) { return (n + 3u) / 4u * 4u; }

template <int FORM>
__global__ void __launch_bounds__(kThreads, 1)
k_records(const __grid_constant__ LoadArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_wtot[32];
    const int G = a.G, tid = threadIdx.x;
    const uint32_t n_rec = whole_vectors(a.large.n_rec);
    uint4* s_req = (uint4*)smem_raw;                                   // [kTile] the tile's records, bucket by bucket
    uint32_t* s_start = (uint32_t*)(s_req + kTile);                    // [n_rec] counts, then places in s_req
    uint32_t* s_to = s_start + n_rec;                                  // [n_rec] place in the bucket less place in s_req
    uint16_t* s_of = (uint16_t*)(s_to + n_rec);                        // [G][kLens]
    grid_dependency_wait();
    let_next_start();
    if (refused(a)) return;
    for (int i = tid; i < G * kLens; i += kThreads) s_of[i] = a.large.rec_bucket[i];
    const bool wide = columns_aligned(a);
    uint32_t t0 = blockIdx.x * kTile;
    Raw raw[kPer / 4];
    if (t0 < a.n) read_tile<FORM>(a, t0, a.n, wide, raw);
#pragma unroll 1
    for (; t0 < a.n; t0 += gridDim.x * kTile) {
        for (uint32_t i = tid; i < n_rec; i += kThreads) s_start[i] = 0;
        __syncthreads();
        uint32_t S[kPer], ln[kPer], rec[kPer];                         // rec: bucket | rank among the tile's in it << 16
#pragma unroll
        for (int q = 0; q < kPer / 4; ++q) {
            Item x[4];
            const uint32_t i0 = t0 + (uint32_t)(q * kThreads + tid) * 4u;
            to_items<S_TRACE, FORM, false>(a, i0, raw[q], nullptr, x);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = q * 4 + u;
                rec[k] = 0xFFFFFFFFu;
                if (!x[u].in || !DBG_OK(x[u].g, G, DBG_K_GATHER, DBG_GROUP) || !DBG_OK(x[u].l, kLens, DBG_K_GATHER, DBG_TABLE)) continue;
                S[k] = x[u].S; ln[k] = x[u].l | x[u].o << 16;
                const uint32_t r = s_of[x[u].g * kLens + x[u].l];
                if (DBG_OK(r, n_rec, DBG_K_GATHER, DBG_TABLE)) rec[k] = r | atomicAdd(&s_start[r], 1u) << 16;
            }
        }
        __syncthreads();
        take_shares(s_start, s_to, n_rec, a.large.rec_at, s_wtot);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            if (rec[k] == 0xFFFFFFFFu) continue;
            const uint32_t slot = s_start[rec[k] & 0xFFFFu] + (rec[k] >> 16), i = t0 + (uint32_t)(k / 4 * kThreads + tid) * 4u + k % 4;
            if (DBG_OK(slot, kTile, DBG_K_GATHER, DBG_SLOT)) s_req[slot] = make_uint4(S[k], ln[k], i, rec[k] & 0xFFFFu);
        }
        if (t0 + gridDim.x * kTile < a.n) read_tile<FORM>(a, t0 + gridDim.x * kTile, a.n, wide, raw);
        __syncthreads();
        const uint32_t here = min(kTile, a.n - t0);
#pragma unroll 2
        for (uint32_t slot = tid; slot < here; slot += kThreads) {
            const uint4 q = s_req[slot];
            if (!DBG_OK(q.w, n_rec, DBG_K_GATHER, DBG_TABLE)) continue;
            const uint32_t to = s_to[q.w] + slot;
            uint4* where = q.w & 1u ? a.req : a.large.parted;          // (a bucket of one length is in order)
            if (DBG_OK(to, a.n, DBG_K_GATHER, DBG_REQUEST)) where[to] = make_uint4(q.x, q.y, q.z, 0u);
        }
        __syncthreads();
    }
}

template <int FORM>
__global__ void __launch_bounds__(kThreads, 1)
k_ticks(const __grid_constant__ LoadArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_wtot[32];
    const int G = a.G, tid = threadIdx.x;
    const uint32_t n_tick = whole_vectors(a.large.n_tick);
    uint32_t* s_tick = (uint32_t*)smem_raw;                            // [kTile] the tile's ticks, bucket by bucket
    uint32_t* s_start = s_tick + kTile;                                // [n_tick] as above
    uint32_t* s_to = s_start + n_tick;
    uint16_t* s_in = (uint16_t*)(s_to + n_tick);                       // [kTile] the ticks' buckets
    uint16_t* s_of = s_in + kTile;                                     // [G][kTickBins]
    // (beside k_records, which began when k_plan was complete)
    if (refused(a)) { grid_dependency_wait(); return; }
    for (int i = tid; i < G * kTickBins; i += kThreads) s_of[i] = a.large.tick_bucket[i];
    const bool wide = columns_aligned(a);
    const uint32_t tile = even_tile(a.n), stride = gridDim.x * tile;
    uint32_t t0 = blockIdx.x * tile, end = min(a.n, t0 + tile);
    Raw raw[kPer / 4];
    if (t0 < a.n) read_tile<FORM>(a, t0, end, wide, raw);
#pragma unroll 1
    for (; t0 < a.n; t0 += stride, end = min(a.n, t0 + tile)) {
        // (with the last tile; k_order reads what k_records has written.  The first block has a tile.)
        if (t0 + stride >= a.n) { grid_dependency_wait(); let_next_start(); }
        for (uint32_t i = tid; i < n_tick; i += kThreads) s_start[i] = 0;
        __syncthreads();
        uint32_t S[kPer], tick[kPer];
#pragma unroll
        for (int q = 0; q < kPer / 4; ++q) {
            Item x[4];
            const uint32_t i0 = t0 + (uint32_t)(q * kThreads + tid) * 4u;
            to_items<S_TRACE, FORM, false>(a, i0, raw[q], nullptr, x);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = q * 4 + u;
                tick[k] = 0xFFFFFFFFu;
                if (i0 + u >= end || !DBG_OK(x[u].g, G, DBG_K_GATHER, DBG_GROUP)) continue;
                S[k] = x[u].S;
                const uint32_t t = s_of[x[u].g * kTickBins + tick_bin(x[u].S)];
                if (DBG_OK(t, n_tick, DBG_K_GATHER, DBG_TABLE)) tick[k] = t | atomicAdd(&s_start[t], 1u) << 16;
            }
        }
        if (t0 + stride < a.n) read_tile<FORM>(a, t0 + stride, min(a.n, t0 + stride + tile), wide, raw);
        __syncthreads();
        take_shares(s_start, s_to, n_tick, a.large.tick_at, s_wtot);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            if (tick[k] == 0xFFFFFFFFu) continue;
            const uint32_t slot = s_start[tick[k] & 0xFFFFu] + (tick[k] >> 16);
            if (DBG_OK(slot, kTile, DBG_K_GATHER, DBG_SLOT)) { s_tick[slot] = S[k]; s_in[slot] = (uint16_t)tick[k]; }
        }
        __syncthreads();
        const uint32_t here = end - t0;
#pragma unroll 4
        for (uint32_t slot = tid; slot < here; slot += kThreads) {
            const uint32_t to = s_to[s_in[slot]] + slot;
            if (DBG_OK(to, a.n, DBG_K_GATHER, DBG_ELEMENT)) a.binned[to] = s_tick[slot];
        }
        __syncthreads();
    }
}

// A block per bucket.
constexpr int kOrderThreads = 512;
__global__ void __launch_bounds__(kOrderThreads)
k_order(const __grid_constant__ LoadArgs a) {
    __shared__ uint32_t s_at[kLens];
    // (beside k_ticks, which let it begin when k_records was complete; and k_sort beside this one, when k_ticks is: the last block, for all)
    if (blockIdx.x == gridDim.x - 1) grid_dependency_wait();
    let_next_start();
    if (refused(a)) return;
    const uint2 members = __ldcg(&a.large.rec_members[blockIdx.x]);
    if (members.x > members.y) return;
    if (blockIdx.x & 1u) return;                                       // (one length: k_records has sent it to its place)
    // the lengths of the bucket: where their requests start (those of the length in front end there; no group has length 0)
    const uint32_t lens = members.y - members.x + 1u, l0 = members.x % kLens;
    if (!DBG_OK(lens - 1u, kLens, DBG_K_GATHER, DBG_TABLE)) return;
    for (uint32_t k = threadIdx.x; k < lens; k += kOrderThreads) s_at[k] = __ldcg(&a.len_end[members.x + k - 1u]);
    const uint32_t begin = __ldcg(&a.len_end[members.x - 1u]), end = __ldcg(&a.len_end[members.y]);
    __syncthreads();
    constexpr int kAhead = 4;
    for (uint32_t i0 = begin + threadIdx.x; i0 < end; i0 += kAhead * kOrderThreads) {
        uint4 q[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) if (i0 + k * kOrderThreads < end) q[k] = __ldcs(&a.large.parted[i0 + k * kOrderThreads]);
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            if (i0 + k * kOrderThreads >= end) break;
            const uint32_t at = (q[k].y & 0xFFFFu) - l0;
            if (!DBG_OK(at, lens, DBG_K_GATHER, DBG_TABLE)) continue;
            const uint32_t to = atomicAdd(&s_at[at], 1u);
            if (DBG_OK(to, a.n, DBG_K_GATHER, DBG_REQUEST)) a.req[to] = q[k];
        }
    }
}

// A block per pair of buckets (the ones of odd numbers are mostly empty), two of 512 threads to a multiprocessor: one sorts while
// the other waits (16 M ticks 114 us; one of 1,024 threads 167 where two of 512 took 122).  As sort_window in ingest.cuh, but that the cells are counted in halves
// of words, and that the ticks are read and counted again to be placed: a thread has too many to keep them, or their ranks (121 us with cell
// and rank in a word, 121 with the rank in half a one).  Blocks that stay and draw their pairs were held up behind dense ones: 16 M ticks of
// one group 138 us -> 217.
constexpr int kSortThreads = 512;
struct BigSort {
    uint32_t a[kBigCap + 2 * kSortPad];                // the ticks; or counters
    uint32_t cell[kBigCap / 2];                        // counts, then starts, then ends, two to a word
    uint32_t bin[kTickBins];                           // bin_cells()
    uint32_t mixed[kBigCap / 32];                      // a bit a cell: it holds different ticks
    uint32_t wtot[32], range[2], most;
};
static_assert(2 * (sizeof(BigSort) + 1024 + 16) <= 227 * 1024, "two blocks to a multiprocessor");

__device__ __forceinline__ uint32_t half_of(uint32_t c, uint32_t w) { return c & 1u ? w >> 16 : w & 0xFFFFu; }

// A bucket whose ticks lie in their cells (sm.cell: where each ends), where cells of different ticks reach further than kSortPad: mostly
// a clock coarser than a microsecond, whose ticks share a cell with their like alone and need no order among themselves.  (A load of
// 4 M requests by a millisecond's clock: 189 us, by a microsecond's 184; with a trace that has one such cell of 256 left to the
// radix sort 454, of 16 M 1,213 and now 565.  Called, not inlined: k_sort of 16 M microsecond ticks in six groups, which do not come
// here, 124.5 us and 125.8; sort_dense called as well 128.9.)
__device__ __noinline__ void sort_crowded(BigSort& sm, uint32_t count, int b0, int b1, uint32_t cells, int32_t* out) {
    const int tid = threadIdx.x;
    uint32_t* const a = sm.a + kSortPad;
    uint32_t bin;
    auto cell_of = [&](uint32_t t) { return tick_cell(sm.bin, b0, b1, cells, t, bin); };
    auto end_of = [&](uint32_t c) { return half_of(c, sm.cell[c >> 1]); };
    auto start_of = [&](uint32_t c) { return c ? end_of(c - 1u) : 0u; };
    for (uint32_t i = tid; i < kBigCap / 32; i += kSortThreads) sm.mixed[i] = 0;
    __syncthreads();
    for (uint32_t i = tid; i + 1u < count; i += kSortThreads) {
        const uint32_t v = a[i];
        if (a[i + 1u] == v) continue;
        const uint32_t c = cell_of(v);
        if (i + 1u < end_of(c)) atomicOr(&sm.mixed[c >> 5], 1u << (c & 31u));
    }
    __syncthreads();
    uint32_t full = 0;
    for (uint32_t i = tid; i < count; i += kSortThreads) {
        const uint32_t v = a[i], c = cell_of(v);
        if (!(sm.mixed[c >> 5] >> (c & 31u) & 1u)) { out[i] = (int32_t)v; continue; }
        const uint32_t from = start_of(c), to = end_of(c);
        if (to - from > 4u * kCellCap) { full = 1u; continue; }
        const uint32_t p = place_in_cell(a, i, v, from, to);
        if (DBG_OK(p, count, DBG_K_RADIX, DBG_ELEMENT)) out[p] = (int32_t)v;
    }
    if (!__syncthreads_or((int)full)) return;
    // Hundreds of ticks of a few neighbouring values in a cell: the whole bucket by a bitonic network, padded with the largest word
    // (a power of two is at most kBigCap).
    uint32_t whole = 2;
    while (whole < count) whole <<= 1;
    for (uint32_t i = count + tid; i < whole; i += kSortThreads) a[i] = 0xFFFFFFFFu;
    for (uint32_t size = 2; size <= whole; size <<= 1)
        for (uint32_t gap = size >> 1; gap > 0; gap >>= 1) {
            __syncthreads();
            for (uint32_t k = tid; k < whole / 2; k += kSortThreads) {
                const uint32_t i = (k & ~(gap - 1u)) << 1 | (k & (gap - 1u)), x = a[i], y = a[i + gap];
                if ((x > y) == ((i & size) == 0u)) { a[i] = y; a[i + gap] = x; }
            }
        }
    __syncthreads();
    for (uint32_t i = tid; i < count; i += kSortThreads) out[i] = (int32_t)a[i];
}

__device__ __forceinline__ void sort_bucket(BigSort& sm, const uint32_t* src, uint32_t count, const uint32_t* bin_start,
                                            const uint32_t* bin_count, int b0, int b1, uint32_t k0, int32_t* out) {
    const int tid = threadIdx.x;
    constexpr int kVecs = kBigCap / 2 / kSortThreads / 4;              // vectors of cells a thread has
    uint32_t* const a = sm.a + kSortPad;
    const uint32_t down = count <= kBigCap / 2 ? 0u : 1u, cells = 2u * count >> down, words = (cells + 1u) / 2u;
    for (uint32_t i = tid; i < (words + kVecs * 4u - 1u) / (kVecs * 4u) * (kVecs * 4u); i += kSortThreads) sm.cell[i] = 0;
    for (int b = b0 + tid; b <= b1; b += kSortThreads)
        sm.bin[b - b0] = bin_cells(__ldcg(&bin_start[b]) - k0, __ldcg(&bin_count[b]), b, down);         // (an empty bin's is not used)
    if (tid < (int)kSortPad) { sm.a[tid] = 0u; a[count + tid] = 0xFFFFFFFFu; }
    if (tid == 0) sm.most = 0;
    __syncthreads();
    constexpr int kAhead = 8;
    uint32_t most = 1;                                                 // ticks of a cell that may hold different ones
#pragma unroll 1
    for (uint32_t i0 = tid; i0 < count; i0 += kAhead * kSortThreads) {
        uint32_t key[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) if (i0 + k * kSortThreads < count) key[k] = __ldcg(&src[i0 + k * kSortThreads]);
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            if (i0 + k * kSortThreads >= count) continue;
            uint32_t bin;
            const uint32_t c = tick_cell(sm.bin, b0, b1, cells, key[k], bin), rank = half_of(c, atomicAdd(&sm.cell[c >> 1], c & 1u ? 65536u : 1u));
            if (!one_value(bin)) most = max(most, rank + 1u);
        }
    }
    most = __reduce_max_sync(FULL, most);
    if ((tid & 31) == 0) atomicMax(&sm.most, most);
    __syncthreads();
    most = sm.most;
    {
        // (in turns that keep eight lanes off one another's banks)
        uint4* cell4 = reinterpret_cast<uint4*>(sm.cell) + tid * kVecs;
        static_assert(kVecs == 4, "the turns");
        const int turn = (tid >> 1) & 3;
        const bool mine = tid * (kVecs * 4u) < words;                  // (those beyond are zero)
        uint4 v[kVecs];
        uint32_t sum[kVecs], own = 0;
        auto both = [](uint32_t w) { return (w & 0xFFFFu) + (w >> 16); };
#pragma unroll
        for (int k = 0; k < kVecs; ++k) {
            v[k] = mine ? cell4[(k + turn) & 3] : make_uint4(0u, 0u, 0u, 0u);
            sum[k] = both(v[k].x) + both(v[k].y) + both(v[k].z) + both(v[k].w);
            own += sum[k];
        }
        const uint32_t run = block_inclusive_scan(own, sm.wtot, (uint32_t*)nullptr) - own;
#pragma unroll
        for (int k = 0; k < kVecs; ++k) {
            uint32_t r = run;
#pragma unroll
            for (int j = 0; j < kVecs; ++j) r += ((j + turn) & 3) < ((k + turn) & 3) ? sum[j] : 0u;
            auto starts = [&](uint32_t w) { const uint32_t s = r | (r + (w & 0xFFFFu)) << 16; r += both(w); return s; };
            const uint32_t x = starts(v[k].x), y = starts(v[k].y), z = starts(v[k].z), w = starts(v[k].w);
            if (mine) cell4[(k + turn) & 3] = make_uint4(x, y, z, w);
        }
    }
    __syncthreads();
#pragma unroll 1
    for (uint32_t i0 = tid; i0 < count; i0 += kAhead * kSortThreads) {
        uint32_t key[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) if (i0 + k * kSortThreads < count) key[k] = __ldcg(&src[i0 + k * kSortThreads]);
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            if (i0 + k * kSortThreads >= count) continue;
            uint32_t bin;
            const uint32_t c = tick_cell(sm.bin, b0, b1, cells, key[k], bin), p = half_of(c, atomicAdd(&sm.cell[c >> 1], c & 1u ? 65536u : 1u));
            if (DBG_OK(p, count, DBG_K_RADIX, DBG_ELEMENT)) a[p] = key[k];
        }
    }
    __syncthreads();
    if (most <= kSortPad) {
        order_by_neighbours<kSortThreads>(a, count, (int)most - 1, out);
        return;
    }
    sort_crowded(sm, count, b0, b1, cells, out);
}

__global__ void __launch_bounds__(kSortThreads, 2)
k_sort(const __grid_constant__ LoadArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_item;
    BigSort& sm = *reinterpret_cast<BigSort*>(smem_raw);
    if (refused(a)) { grid_dependency_wait(); return; }                // (beside k_order)
#pragma unroll 1
    for (uint32_t bucket = blockIdx.x * 2u; bucket <= blockIdx.x * 2u + 1u; ++bucket) {
        const uint4 j = __ldcg(&a.large.tick_jobs[bucket]);            // ticks [x, y) of the bins z .. w, counted through the groups
        if (j.x >= j.y) continue;
        const int g = (int)j.z / kTickBins, b0 = (int)j.z - g * kTickBins, b1 = (int)j.w - g * kTickBins;
        const uint32_t k0 = j.x, k1 = j.y, edge = tick_bin_edge(b0);
        const uint32_t first = __ldcg(&a.grp_off[g]), N = __ldcg(&a.grp_off[g + 1]) - first;
        if (k1 - k0 <= kBigCap) {
            sort_bucket(sm, a.binned + k0, k1 - k0, a.tick_start + (size_t)g * kTickBins, a.tick_cnt + (size_t)g * kTickBins, b0, b1, k0, a.sorted + k0);
        } else if (!sort_dense<kSortThreads, kBigCap>(sm.a, sm.wtot, sm.range, a.binned + k0, k1 - k0, edge, tick_bin_edge(b1 + 1) - edge, a.sorted + k0) &&
                   threadIdx.x == 0) {
            atomicMax(&a.z->err[3], 1);                                // (the radix sort, then)
        }
        __syncthreads();
        write_knots<kSortThreads>(a, g, k0, k1, first, N);
    }
    // the last block to come here reports the flags
    if (threadIdx.x == 0) { __threadfence(); s_item = atomicAdd(&a.z->done, 1u); }
    __syncthreads();
    if (s_item != gridDim.x - 1) return;
    grid_dependency_wait();
    if (threadIdx.x < 4) a.readback->err[threadIdx.x] = __ldcg(&a.z->err[threadIdx.x]);
}

size_t records_smem(const LoadArgs& a) { return (size_t)kTile * 16 + (size_t)whole_vectors(a.large.n_rec) * 8 + (size_t)a.G * kLens * 2; }
size_t ticks_smem(const LoadArgs& a) { return (size_t)kTile * 6 + (size_t)whole_vectors(a.large.n_tick) * 8 + (size_t)a.G * kTickBins * 2; }
static_assert(kTile * 16 + kRecBuckets * 8 + kPrivateGroups * kLens * 2 <= 220 * 1024, "k_records' shared memory");

template <int FORM>
cudaError_t launch_large(const LoadArgs& a, int sms, cudaStream_t st) {
    cudaError_t e;
    if ((e = cudaMemsetAsync(a.z, 0, a.zero_bytes, st))) return e;
    const size_t counters = (size_t)a.G * (kLens + kTickBins) * 4, plan = (size_t)2 * kPlanBuckets * 4;
    if ((e = allow_smem((const void*)k_count<FORM>, 220 * 1024)) || (e = allow_smem((const void*)k_records<FORM>, 220 * 1024)) || (e = allow_smem((const void*)k_ticks<FORM>, 220 * 1024)) ||
        (e = allow_smem((const void*)k_plan, plan)) || (e = allow_smem((const void*)k_sort, sizeof(BigSort))))
        return e;
    k_count<FORM><<<sms, kThreads, counters, st>>>(a);
    if ((e = cudaGetLastError())) return e;
    if ((e = launch_after(k_plan, 2 * a.G, kThreads, plan, st, a))) return e;
    if ((e = launch_after(k_records<FORM>, sms, kThreads, records_smem(a), st, a))) return e;
    if ((e = launch_after(k_ticks<FORM>, sms, kThreads, ticks_smem(a), st, a))) return e;
    if ((e = launch_after(k_order, a.large.n_rec, kOrderThreads, 0, st, a))) return e;
    return launch_after(k_sort, a.large.n_tick / 2, kSortThreads, sizeof(BigSort), st, a);
}

}  // namespace

DBG_TRANSLATION_UNIT()

cudaError_t run_load_large(const LoadArgs& a, int sms, cudaStream_t st) {
    if (a.packed) return launch_large<F_PACKED>(a, sms, st);
    return a.st_ticks ? launch_large<F_STAGE>(a, sms, st) : launch_large<F_COLUMNS>(a, sms, st);
}

}  // namespace disco
