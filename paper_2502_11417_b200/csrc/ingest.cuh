// What the ingestion kernels share (load.cu, load_large.cu): reading and checking the trace, and the sort of a window of ticks
// in shared memory.
#pragma once

#include "load.cuh"
#include "pack.cuh"
#include "scan.cuh"

namespace disco {

namespace {

constexpr int kThreads = 1024;
constexpr int kLens = kMaxPrompt + 1;
constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr uint32_t kWindow = 4096;        // a window starts with the first bin behind every 4,096th tick of its group
constexpr uint32_t kSortCap = 8192;       // ticks sorted at a time
constexpr uint32_t kCounters = 2 * kSortCap;      // values counted at a time
constexpr uint32_t kMaxRange = 1u << 18;  // values a dense bin may span
constexpr uint32_t kMaxCount = 1u << 22;  // ticks a dense bin may hold
constexpr int kPrivateGroups = kLargeMaxGroups;   // groups whose counters fit in shared memory (29 KB each)
constexpr int kPrivateTickGroups = 16;    // the same, counters of tick bins alone
static_assert(kMaxTicks + (uint64_t)kLoadBlocks * kThreads * 4 <= 1ull << 32, "a step of the loops over the ticks");

enum Source { S_TRACE, S_TICKS, S_TTFT };
enum Form { F_COLUMNS, F_STAGE, F_PACKED };   // a trace's columns; the same, with a copy left for the second pass; packed

__device__ __forceinline__ uint32_t tick_bin_edge(int b) {     // smallest ticks of the bin (2^31 behind the last)
    return b < 128 ? (uint32_t)b : (uint32_t)(128 + (b & 127)) << ((b >> 7) - 1);
}

constexpr uint32_t kSortPad = 16;         // ticks that a place is compared with on either side, at most
struct SortSmem {
    uint32_t a[kSortCap + 2 * kSortPad], b[kSortCap];  // ticks of a window, twice; or kCounters counters
    uint16_t wcnt[kThreads / 32][256];                 // keys of each digit per warp (radix sort)
    uint32_t dig[256];
    uint32_t wtot[32];
    uint32_t range[2], most;
    uint32_t bin[kTickBins];                           // of a window's bins: first place | count << 16
};

// The waits between blocks are bounded.  Behind one that ran out, tables may hold what an earlier call left in them, and
// places taken from those could lie anywhere: a block that gives up sets the flag that makes the host refuse the results
// and kLost in the barriers' word, and leaves the kernel; so does every block that finds kLost where it waits.  A block
// that passes a barrier has seen every block arrive there, with its part of the work in front of it done.
constexpr uint32_t kWaitTries = 1u << 22;
constexpr uint32_t kLost = 1u << 31;              // (the word counts at most 256 blocks three times)
__device__ __forceinline__ void give_up(LoadZero* z) {
    atomicMax(&z->err[3], 2);
    atomicOr(&z->barrier, kLost);
}

// Waits until `want` blocks have arrived; false: the caller's block has to leave.
__device__ __forceinline__ bool await_blocks(LoadZero* z, uint32_t want) {
    uint32_t seen, tries = 0;
    do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&z->barrier) : "memory");
    } while (seen < want && ++tries < kWaitTries);                     // (with kLost it is above any count)
    if (seen < want) give_up(z);
    __threadfence();
    return seen >= want && !(seen & kLost);
}

// Checked build: a wait for one arrival that nobody makes (LoadArgs::absent).
#ifdef DISCO_DEBUG
#define ABSENT(a, wait) ((a).absent == (wait) ? 1u : 0u)
// A block that is some two milliseconds late with what it has to do next (LoadArgs::absent = 5).
#define LATE(a, block) do { if ((a).absent == 5u && (block)) for (const long long t0 = clock64(); clock64() - t0 < 4000000ll;) { } } while (0)
#else
#define ABSENT(a, wait) 0u
#define LATE(a, block) do { } while (0)
#endif

// Four neighbouring requests of the trace (or ticks of a sample) as the two passes see them.
struct Item { uint32_t g, S, l, o; bool in; };

// (LAST: read for the last time, so that the lines need not stay in L2)
template <class T4, bool LAST, class T>
__device__ __forceinline__ void load4(const T* p, uint32_t i0, uint32_t n, bool wide, T (&v)[4], T fill) {
    if (wide && i0 + 4u <= n) {
        const T4 x = LAST ? __ldcs(reinterpret_cast<const T4*>(p + i0)) : *reinterpret_cast<const T4*>(p + i0);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = i0 + u < n ? p[i0 + u] : fill;
    }
}

// Four neighbouring bytes as a word.
template <bool LAST>
__device__ __forceinline__ uint32_t load_bytes(const uint8_t* p, uint32_t i0, uint32_t n, bool wide) {
    if (wide && i0 + 4u <= n) return LAST ? __ldcs(reinterpret_cast<const uint32_t*>(p + i0)) : *reinterpret_cast<const uint32_t*>(p + i0);
    uint32_t v = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) if (i0 + u < n) v |= (uint32_t)p[i0 + u] << (8 * u);
    return v;
}
__device__ __forceinline__ uint32_t byte_of(uint32_t v, int u) { return (v >> (8 * u)) & 255u; }

// What a thread has read of the items i0 .. i0 + 3: TTFTs or ticks, lengths (both in l unless FORM is F_COLUMNS), profiles or
// groups.
struct Raw { uint32_t t[4], l[4], o[4], sp, dp; };

// Reads the items i0 .. i0 + 3.  wide: the columns are aligned for vector loads.  CHECK: the first pass.  AGAIN: for counting;
// they will be read once more.
template <int SRC, int FORM, bool CHECK, bool AGAIN = false>
__device__ __forceinline__ void read_raw(const LoadArgs& a, uint32_t i0, bool wide, Raw& r) {
    constexpr bool kLast = !CHECK && !AGAIN;
    r.sp = r.dp = 0u;
    if (FORM == F_STAGE && !CHECK) {
        load4<uint4, kLast>(a.st_ln, i0, a.n, true, r.l, 0u);
        load4<uint4, kLast>(a.st_ticks, i0, a.n, true, r.t, 0u);
        r.sp = load_bytes<kLast>(a.st_g, i0, a.n, true);
    } else if (SRC == S_TICKS) {
        load4<uint4, !CHECK>(reinterpret_cast<const uint32_t*>(a.ticks), i0, a.n, wide, r.t, 0u);
    } else if (FORM == F_PACKED) {
        // (chunks are whole vectors, and a vector lies in one chunk; what lies behind item n is not used)
        const char* c = a.packed + (size_t)(i0 / kPackChunk) * kPackBytes;
        const uint32_t k = i0 % kPackChunk;
        const uint4 ln = *reinterpret_cast<const uint4*>(c + (size_t)k * 4);
        const uint4 tt = *reinterpret_cast<const uint4*>(c + (size_t)kPackChunk * 4 + (size_t)k * 4);
        r.dp = *reinterpret_cast<const uint32_t*>(c + (size_t)kPackChunk * 8 + k);
        r.l[0] = ln.x; r.l[1] = ln.y; r.l[2] = ln.z; r.l[3] = ln.w;
        r.t[0] = tt.x; r.t[1] = tt.y; r.t[2] = tt.z; r.t[3] = tt.w;
    } else {
        load4<uint4, kLast>(reinterpret_cast<const uint32_t*>(a.ttft), i0, a.n, wide, r.t, 0x3F800000u);
        if (SRC == S_TRACE) {
            load4<uint4, kLast>(reinterpret_cast<const uint32_t*>(a.prompt), i0, a.n, wide, r.l, 1u);
            if (!AGAIN) load4<uint4, kLast>(reinterpret_cast<const uint32_t*>(a.outlen), i0, a.n, wide, r.o, 1u);
            if (a.sp) r.sp = load_bytes<kLast>(a.sp, i0, a.n, wide);
            if (a.dp) r.dp = load_bytes<kLast>(a.dp, i0, a.n, wide);
        }
    }
}

// The items as read, checked in the first pass.  s_off: where the groups start (of ticks stored group after group).
template <int SRC, int FORM, bool CHECK, bool AGAIN = false>
__device__ __forceinline__ void to_items(const LoadArgs& a, uint32_t i0, const Raw& r, const uint32_t* s_off, Item (&x)[4]) {
    uint32_t g = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        bool in = i0 + u < a.n;
        if (FORM == F_STAGE && !CHECK) {
            x[u] = Item{byte_of(r.sp, u), r.t[u], r.l[u] & 0xFFFFu, r.l[u] >> 16, in};
            continue;
        }
        if (SRC == S_TICKS) {
            while ((int)g + 1 < a.G && i0 + u >= s_off[g + 1]) ++g;
            if (CHECK && (int32_t)r.t[u] < 0) {
                if (atomicCAS(&a.z->err[0], 0, 3) == 0) a.z->err[1] = (int32_t)(i0 + u);
                in = false;
            }
            x[u] = Item{g, r.t[u], 1u, 1u, in};
            continue;
        }
        const float t = __uint_as_float(r.t[u]);
        const uint32_t sp = byte_of(r.sp, u), dp = byte_of(r.dp, u);
        int32_t l = 1, o = 1;
        if (FORM == F_PACKED) { l = (int32_t)(r.l[u] & 0xFFFFu); o = (int32_t)(r.l[u] >> 16); }
        else if (SRC == S_TRACE) { l = (int32_t)r.l[u]; o = AGAIN ? 1 : (int32_t)r.o[u]; }
        if (CHECK && in) {
            int bad = 0;
            if (l < 1 || l > kMaxPrompt) bad = 1;
            else if (o < 1 || o > kMaxOutput) bad = 2;
            else if (!(t > 0.0f) || !(t <= 2000.0f)) bad = 3;      // NaN fails both comparisons
            else if (FORM == F_PACKED ? (int)dp >= a.G : SRC == S_TRACE && (sp >= a.ns || dp >= a.nd)) bad = 4;
            if (bad) {
                if (atomicCAS(&a.z->err[0], 0, bad) == 0) a.z->err[1] = (int32_t)(i0 + u);
                in = false;
            }
        }
        // ticks = nearest integer (ties to even) of the fp64 product, as a host llrint would give
        const uint32_t S = __double2uint_rn(__dmul_rn((double)t, 1e6));      // (2e9 at most)
        x[u] = Item{SRC == S_TRACE ? sp * a.nd + dp : 0u, S, (uint32_t)l, (uint32_t)o, in};
    }
}

template <int SRC, int FORM, bool CHECK, bool AGAIN = false>
__device__ __forceinline__ void read_items(const LoadArgs& a, uint32_t i0, bool wide, const uint32_t* s_off, Item (&x)[4]) {
    Raw r;
    read_raw<SRC, FORM, CHECK, AGAIN>(a, i0, wide, r);
    to_items<SRC, FORM, CHECK, AGAIN>(a, i0, r, s_off, x);
}

// Leaves the items for the second pass (the staging arrays hold whole vectors).
__device__ __forceinline__ void stage_items(const LoadArgs& a, uint32_t i0, const Item (&x)[4]) {
    *reinterpret_cast<uint4*>(a.st_ticks + i0) = make_uint4(x[0].S, x[1].S, x[2].S, x[3].S);
    *reinterpret_cast<uint4*>(a.st_ln + i0) = make_uint4(x[0].l | x[0].o << 16, x[1].l | x[1].o << 16, x[2].l | x[2].o << 16, x[3].l | x[3].o << 16);
    *reinterpret_cast<uchar4*>(a.st_g + i0) = make_uchar4((uint8_t)x[0].g, (uint8_t)x[1].g, (uint8_t)x[2].g, (uint8_t)x[3].g);
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

// Where a bin's ticks go: every bin has as many cells (`down` = 1), or twice as many, as ticks, evenly over its values.  A word a
// bin: its first cell, its cells << 14, and 1 << 31 if each of them holds one value (as many cells as values, or more).
__device__ __forceinline__ uint32_t bin_cells(uint32_t first, uint32_t count, int b, uint32_t down) {
    const uint32_t w = b < 128 ? 0u : (uint32_t)(b >> 7) - 1u, cells = count << 1 >> down;              // (a bin spans 2^w values)
    return (first << 1 >> down & 0x3FFFu) | cells << 14 | (1u << w <= cells ? 1u << 31 : 0u);
}
// The cell of a tick of the bins from b0 on, by the 16 bits of its float that follow the bin's; `bin`: its bin's word.
__device__ __forceinline__ uint32_t tick_cell(const uint32_t* bins, int b0, int b1, uint32_t cells, uint32_t t, uint32_t& bin) {
    const uint32_t f = __float_as_uint(__uint2float_rz(t));
    const int b = t < 128u ? (int)t : (int)(f >> 16) - ((127 + 7) << 7) + 128;
    bin = 0;
    if (!DBG_OK(b - b0, b1 - b0 + 1, DBG_K_RADIX, DBG_BIN)) return 0u;
    bin = bins[b - b0];
    const uint32_t c = mad_hi(f << 16, bin >> 14 & 0x7FFFu, bin & 0x3FFFu);
    return DBG_OK(c, cells, DBG_K_RADIX, DBG_BIN) ? c : 0u;
}
__device__ __forceinline__ bool one_value(uint32_t bin) { return (int32_t)bin < 0; }

// Ticks placed cell by cell into their order, found by comparing with neighbours as far as cells of different ticks reach
// (`reach` <= kSortPad; a tick moves up by those behind it that are smaller, and down by those in front that are larger).  A
// thread takes every THREADS-th place, so that neighbouring lanes look at the same few ticks and write side by side.
template <int THREADS>
__device__ __forceinline__ void order_by_neighbours(const uint32_t* a, uint32_t count, int reach, int32_t* out) {
#pragma unroll 2
    for (uint32_t i = threadIdx.x; i < count; i += THREADS) {
        const uint32_t v = a[i];
        uint32_t p = i;
#pragma unroll 2
        for (int d = 1; d <= reach; ++d) {
            p += a[i + d] < v ? 1u : 0u;
            p -= a[(int)i - d] > v ? 1u : 0u;
        }
        if (DBG_OK(p, count, DBG_K_RADIX, DBG_ELEMENT)) out[p] = (int32_t)v;
    }
}
// A tick's place where cells reach further: its cell is [from, to).
__device__ __forceinline__ uint32_t place_in_cell(const uint32_t* a, uint32_t i, uint32_t v, uint32_t from, uint32_t to) {
    uint32_t p = i;
    for (uint32_t y = from; y < to; ++y) { const uint32_t u = a[y]; p += y < i ? (u > v ? ~0u : 0u) : (u < v ? 1u : 0u); }
    return p;
}

// Sorts the `count` <= kSortCap ticks of the bins [b0, b1] of a group from src into out: every bin has cells in proportion to its
// ticks, evenly over its values, so that a cell holds a tick or two whatever the distribution; the ticks are counted by cell,
// placed, and compared with their neighbours as far as cells reach.  Returns false if more than kCellCap different ticks may
// share a cell (what it has written is to be written again).
// Bound: instruction issue.  (Of the 14 us of a window of 8,192 ticks cells put in order by insertion, a thread a cell, took 5.6,
// each tick compared with its cell's as long; with its neighbours 1.5.  A thread keeps its ticks, their cells and their ranks there: counted once
// more to be placed, and cells worked out from the ticks' places in their bins, k_load_once took 48 us for a million requests of one group,
// now 44, 35 and 33 for 100,000 of six.)
constexpr uint32_t kCellCap = 64;

__device__ __forceinline__ bool sort_window(SortSmem& sm, const uint32_t* src, uint32_t count, const uint32_t* bin_start,
                                            const uint32_t* bin_count, int b0, int b1, int32_t* out) {
    const int tid = threadIdx.x;
    constexpr int kKeep = kSortCap / kThreads, kVecs = kSortCap / kThreads / 4;     // ticks a thread keeps, vectors of cells it has
    uint32_t* cell = sm.b;                                             // counts, then starts
    uint32_t* const a = sm.a + kSortPad;
    // twice as many cells as ticks, or as many
    const uint32_t k0 = __ldcg(&bin_start[b0]), down = count <= kSortCap / 2 ? 0u : 1u, cells = 2u * count >> down;
    for (uint32_t i = tid; i < (cells + kVecs * 4u - 1u) / (kVecs * 4u) * (kVecs * 4u); i += kThreads) cell[i] = 0;
    for (int b = b0 + tid; b <= b1; b += kThreads) {
        const uint32_t c = __ldcg(&bin_count[b]);
        sm.bin[b - b0] = bin_cells(__ldcg(&bin_start[b]) - k0, c, b, down);           // (an empty bin's is not used)
    }
    if (tid < (int)kSortPad) { sm.a[tid] = 0u; a[count + tid] = 0xFFFFFFFFu; }
    if (tid == 0) sm.most = 0;
    uint32_t key[kKeep], at[kKeep];                                    // at: cell | rank among the cell's ticks << 14
#pragma unroll
    for (int k = 0; k < kKeep; ++k) {
        const uint32_t i = k * kThreads + tid;
        if (i < count) key[k] = __ldcg(&src[i]);
    }
    __syncthreads();
    auto cell_of = [&](uint32_t t, uint32_t& bin) { return tick_cell(sm.bin, b0, b1, cells, t, bin); };
    uint32_t most = 1;                                                 // ticks of a cell that may hold different ones
#pragma unroll
    for (int k = 0; k < kKeep; ++k) {
        if ((uint32_t)k * kThreads + tid >= count) break;
        uint32_t bin;
        const uint32_t c = cell_of(key[k], bin), rank = atomicAdd(&cell[c], 1u);
        if (!one_value(bin)) most = max(most, rank + 1u);
        at[k] = c | rank << 14;
    }
    most = __reduce_max_sync(FULL, most);
    if ((tid & 31) == 0) atomicMax(&sm.most, most);
    __syncthreads();
    most = sm.most;
    // the cells' starts; a thread's neighbouring cells as vectors, in turns that keep eight lanes off one another's banks
    {
        uint4* cell4 = reinterpret_cast<uint4*>(cell) + tid * kVecs;
        const int turn = (tid >> (kVecs == 2 ? 2 : 1)) & (kVecs - 1);
        const bool mine = tid * (kVecs * 4u) < cells;                  // (those beyond `cells` are zero)
        uint4 v[kVecs];
        uint32_t sum[kVecs], own = 0;
#pragma unroll
        for (int k = 0; k < kVecs; ++k) {
            v[k] = mine ? cell4[(k + turn) & (kVecs - 1)] : make_uint4(0u, 0u, 0u, 0u);
            sum[k] = v[k].x + v[k].y + v[k].z + v[k].w;
            own += sum[k];
        }
        const uint32_t run = block_inclusive_scan(own, sm.wtot, (uint32_t*)nullptr) - own;
#pragma unroll
        for (int k = 0; k < kVecs; ++k) {
            uint32_t r = run, t;
#pragma unroll
            for (int j = 0; j < kVecs; ++j) r += ((j + turn) & (kVecs - 1)) < ((k + turn) & (kVecs - 1)) ? sum[j] : 0u;
            t = v[k].x; v[k].x = r; r += t; t = v[k].y; v[k].y = r; r += t; t = v[k].z; v[k].z = r; r += t; v[k].w = r;
            if (mine) cell4[(k + turn) & (kVecs - 1)] = v[k];
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kKeep; ++k) {
        if ((uint32_t)k * kThreads + tid >= count) break;
        const uint32_t p = cell[at[k] & 0x3FFFu] + (at[k] >> 14);
        if (DBG_OK(p, count, DBG_K_RADIX, DBG_ELEMENT)) a[p] = key[k];
    }
    __syncthreads();
    if (most <= kSortPad) {
        order_by_neighbours<kThreads>(a, count, (int)most - 1, out);
        return true;
    }
    if (most > kCellCap) return false;
    for (uint32_t i = tid; i < count; i += kThreads) {
        uint32_t bin;
        const uint32_t v = a[i], c = cell_of(v, bin), from = cell[c], to = c + 1u < cells ? cell[c + 1u] : count;
        const uint32_t p = one_value(bin) ? i : place_in_cell(a, i, v, from, to);
        if (DBG_OK(p, count, DBG_K_RADIX, DBG_ELEMENT)) out[p] = (int32_t)v;
    }
    return true;
}

// The same whatever the ticks (all of them in [lo, lo + 2^bits)): stable counting passes of at most eight bits, a warp's share
// of the keys at a time with the ranks from ballots.  Four to six times slower.
__device__ __noinline__ void sort_window_radix(SortSmem& sm, const uint32_t* src, uint32_t count, uint32_t lo, int bits, int32_t* out) {
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    if (bits == 0) {
        for (uint32_t i = tid; i < count; i += kThreads) out[i] = (int32_t)lo;
        return;
    }
    uint32_t *from = sm.a, *to = sm.b;
    for (uint32_t i = tid; i < count; i += kThreads) from[i] = __ldcg(&src[i]) - lo;
    const int passes = (bits + 7) / 8, d_bits = (bits + passes - 1) / passes, digits = 1 << d_bits;
    constexpr uint32_t kShare = kSortCap / (kThreads / 32);                // keys of a warp
    constexpr int kRounds = kShare / 32;
    const int rounds = (int)((min(count, kShare) + 31u) / 32u), warps = (int)((count + kShare - 1u) / kShare);
    for (int p = 0; p < passes; ++p) {
        const int shift = p * d_bits;
        for (int i = tid; i < warps * 256; i += kThreads) (&sm.wcnt[0][0])[i] = 0;
        __syncthreads();
        uint32_t key[kRounds], place[kRounds];        // place: digit | rank among the warp's equal digits so far << 8
        if (w < warps) {
#pragma unroll
            for (int j = 0; j < kRounds; ++j) {
                if (j >= rounds) break;
                const uint32_t i = w * kShare + j * 32u + lane;
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
            for (int j = 0; j < kRounds; ++j) {
                if (j >= rounds) break;
                const uint32_t i = w * kShare + j * 32u + lane;
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

// Sorts a dense bin by counting its values, which all lie in [lo, lo + range).  Returns false where that would take too long.
// Bound: one block's latency.  (Loads of 4 M requests in one group: TTFTs by a 10 ms clock 264 us where every bin is counted, 180 with
// bins of one value written at once; all of them within 4 ms 1,074 with a search over all values for every place, 544 from the
// place before.)
// THREADS: the block's; at: shared memory for COUNTERS of them.
template <int THREADS, uint32_t COUNTERS>
__device__ __forceinline__ bool sort_dense(uint32_t* at, uint32_t* wtot, uint32_t (&lo_hi)[2], const uint32_t* src, uint32_t count,
                                           uint32_t lo, uint32_t range, int32_t* out) {
    const int tid = threadIdx.x;
    // One value, as a clock coarser than the bin is wide leaves it (its counter would be added to one by one): looked for where the
    // first ticks are equal.
    const uint32_t v0 = __ldcg(&src[0]);
    if (!__syncthreads_or((int)(__ldcg(&src[min((uint32_t)tid, count - 1u)]) != v0))) {
        uint32_t other = 0;
#pragma unroll 8
        for (uint32_t i = tid; i < count; i += THREADS) other |= __ldcg(&src[i]) ^ v0;
        if (!__syncthreads_or((int)(other != 0u))) {
            for (uint32_t i = tid; i < count; i += THREADS) out[i] = (int32_t)v0;
            return true;
        }
    }
    if (range > COUNTERS) {                                           // the values that occur may lie closer together
        if (tid == 0) { lo_hi[0] = 0xFFFFFFFFu; lo_hi[1] = 0u; }
        __syncthreads();
        uint32_t mn = 0xFFFFFFFFu, mx = 0u;
        for (uint32_t i = tid; i < count; i += THREADS) { const uint32_t t = __ldcg(&src[i]); mn = min(mn, t); mx = max(mx, t); }
        mn = __reduce_min_sync(FULL, mn); mx = __reduce_max_sync(FULL, mx);
        if ((tid & 31) == 0) { atomicMin(&lo_hi[0], mn); atomicMax(&lo_hi[1], mx); }
        __syncthreads();
        lo = lo_hi[0]; range = lo_hi[1] - lo + 1u;
    }
    if (range > kMaxRange || count > kMaxCount) return false;
    uint32_t done = 0;
    for (uint32_t r0 = 0; r0 < range; r0 += COUNTERS) {
        // a thread's neighbouring values, as few as the range needs
        const uint32_t here = min(range - r0, COUNTERS), per = (here + THREADS - 1) / THREADS;
        for (uint32_t i = tid; i < per * THREADS; i += THREADS) at[i] = 0;
        __syncthreads();
#pragma unroll 8
        for (uint32_t i = tid; i < count; i += THREADS) {
            const uint32_t v = __ldcg(&src[i]) - lo - r0;
            if (v < here) atomicAdd(&at[v], 1u);
        }
        __syncthreads();
        uint32_t sum = 0, total;
        for (uint32_t k = 0; k < per; ++k) sum += at[tid * per + k];
        uint32_t run = block_inclusive_scan(sum, wtot, &total) - sum;
        for (uint32_t k = 0; k < per; ++k) { const uint32_t c = at[tid * per + k]; at[tid * per + k] = run; run += c; }
        __syncthreads();
        // Equal ticks are the same: every place looks up its value, the last that starts at or in front of it.  The value of the thread's
        // next place is looked for among the next four where it lies there on the average.  (Looked for there always: k_sort of
        // 4 M microsecond ticks in one group, a hundred values further on, 35.4 us -> 41.)
        const int near = (unsigned long long)here * THREADS <= 4ull * total ? 4 : 0;
        uint32_t v = 0;
        for (uint32_t i = tid; i < total; i += THREADS) {
            int ahead = near;
            while (ahead > 0 && v + 1u < here && at[v + 1u] <= i) { ++v; --ahead; }
            if (ahead == 0)
                for (uint32_t n = here - v; n > 1u;) { const uint32_t half = n >> 1; if (at[v + half] <= i) v += half; n -= half; }
            if (DBG_OK(done + i, count, DBG_K_RADIX, DBG_ELEMENT)) out[done + i] = (int32_t)(lo + r0 + v);
        }
        done += total;
        __syncthreads();
    }
    return true;
}

// Writes the knots K_g[k] = sorted_g[(k (N_g - 1)) / 256] that lie in [k0, k1), sorted by this block; first, N: the group's.
template <int THREADS>
__device__ __forceinline__ void write_knots(const LoadArgs& a, int g, uint32_t k0, uint32_t k1, uint32_t first, uint32_t N) {
    for (int k = threadIdx.x; k < kNKnots; k += THREADS) {
        const uint32_t at = first + (uint32_t)(((uint64_t)k * (N - 1)) / 256u);
        if (at >= k0 && at < k1) {
            const int32_t v = __ldcg(&a.sorted[at]);
            a.knots[g * kNKnots + k] = v;
            if (k == kNKnots - 1) a.readback->knot_max[g] = v;
        }
    }
}

// Sorts the bins [b0, b1] of a group, whose ticks lie in [k0, k1); ends with a barrier.
__device__ __forceinline__ void sort_bins(const LoadArgs& a, SortSmem& sm, int g, int b0, int b1, uint32_t k0, uint32_t k1) {
    const uint32_t lo = tick_bin_edge(b0);
    auto bits_of = [](uint32_t range) { return range <= 1u ? 0 : 32 - __clz((int)(range - 1u)); };
    const uint32_t *starts = a.tick_start + (size_t)g * kTickBins, *counts = a.tick_cnt + (size_t)g * kTickBins;
    // up to kSortCap ticks; otherwise the last bin is a large one: the others first
    const bool large = k1 - k0 > kSortCap;
    const uint32_t to = large ? __ldcg(&starts[b1]) : k1;
    const int last = large ? b1 - 1 : b1;
    if (to > k0 && !sort_window(sm, a.binned + k0, to - k0, starts, counts, b0, last, a.sorted + k0)) {
        __syncthreads();
        sort_window_radix(sm, a.binned + k0, to - k0, lo, bits_of(tick_bin_edge(last + 1) - lo), a.sorted + k0);
    }
    if (large) {
        __syncthreads();
        const uint32_t edge = tick_bin_edge(b1);
        if (!sort_dense<kThreads, kCounters>(sm.a, sm.wtot, sm.range, a.binned + to, k1 - to, edge, tick_bin_edge(b1 + 1) - edge, a.sorted + to) &&
            threadIdx.x == 0)
            atomicMax(&a.z->err[3], 1);
    }
    __syncthreads();
}

}  // namespace

}  // namespace disco
