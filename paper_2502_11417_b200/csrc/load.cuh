// Trace ingestion and the sort of server-TTFT ticks (load.cu).
#pragma once

#include <algorithm>

#include "disco_internal.cuh"

namespace disco {

// Ticks fall into 3,200 bins a group: their value below 128, then 128 bins an octave up to 2^31.
constexpr int kTickBins = 128 + 24 * 128;
#ifdef __CUDACC__
__device__ __forceinline__ int tick_bin(uint32_t t) {
    return t < 128u ? (int)t : (int)(__float_as_uint(__uint2float_rz(t)) >> 16) - ((127 + 7) << 7) + 128;
}
#endif

struct LoadReadback {            // what the host needs after a load; pinned host memory, written by the kernel
    int32_t err[4];
    uint32_t max_n;
    uint32_t ng[kMaxGroups];
    uint32_t grp_off[kMaxGroups + 1];
    int32_t knot_max[kMaxGroups];
    uint64_t grp_sum_n[kMaxGroups];
};

// Words that a load or a sort must find zero, contiguous.
constexpr uint32_t kLoadBlocks = 256;     // blocks of the kernel, at most
// The ticks that the sorts take, at most.  They are counted in 32 bits by loops that step by up to 2^20 (256 blocks of 1,024
// threads with four each): an index below this, and one step on, does not wrap.
constexpr uint64_t kMaxTicks = (1ull << 32) - (1ull << 20);
struct LoadZero {
    unsigned long long part[2][kLoadBlocks];      // sums over the blocks' shares of the counters: sum << 1 | 1
    uint64_t grp_sum_n[kMaxGroups];       // output tokens per group
    uint32_t grp_n[kMaxGroups];           // requests per group (load_large.cu)
    uint32_t max_n;                       // longest output
    uint32_t barrier, done;
    uint32_t tables_left, free_ticket, pad[3];    // k_prep's and k_playout_free's, zero between their launches (no load touches them)
    int32_t err[4];                       // code, request index, window flag, sort flag (1: some bin needs the fallback, 2: a
                                          // wait between blocks ran out)
};

__host__ __device__ constexpr uint32_t sort_windows(uint32_t n, int G) { return n / 4096u + (uint32_t)G; }

// Large traces are placed in two steps, by way of buckets (load_large.cu).
constexpr uint32_t kLargeMaxN = 1u << 24;     // (beyond, the tables of buckets no longer fit in a block's shared memory)
constexpr uint32_t kLargeMinN = 2200000;    // (where it becomes the faster one: see load_large.cu)
constexpr uint32_t kLargeMinInPlace = 3000000;   // ... where columns are read in place, over the link
constexpr int kLargeMaxGroups = 7;            // groups whose counters fit there
constexpr uint32_t kTickShare = 8192;         // ticks to a bucket, at most
// Records to a bucket: 2,048, or as many as leave 1,024 buckets.  Ticks: so many that the multiprocessors sort equally many buckets.
inline uint32_t rec_share(uint32_t n) { return n / 1024u + 1u > 2048u ? n / 1024u + 1u : 2048u; }
inline uint32_t tick_share(uint32_t n, uint32_t sms) {
    const uint32_t most = kTickShare - 192u, blocks = 2u * sms, each = (n + blocks * most - 1u) / (blocks * most);
    const uint32_t share = (n + blocks * each - 1u) / (blocks * each) + 64u;                        // (the groups' last buckets are partly filled)
    return share < 2048u ? 2048u : share;
}
constexpr uint32_t kRecBuckets = 2 * (1024 + kLargeMaxGroups), kTickBuckets = 2 * (kLargeMaxN / 8000 + 512 + kLargeMaxGroups);
struct LargeLoad {
    uint4* parted;                        // [n] records bucket by bucket
    uint32_t rec_share, tick_share, n_rec, n_tick;    // requests or ticks to a bucket, numbers of buckets
    uint16_t *rec_bucket, *tick_bucket;   // [G][4097], [G][kTickBins]
    uint32_t *rec_at, *tick_at;           // cursors, [n_rec] and [n_tick]
    uint2* rec_members;                   // first and last length, counted through the groups (first > last: none)
    uint4* tick_jobs;                     // where the bucket's ticks start and end, first and last bin, counted through the groups (0, 0: none)
};

// Small and middling traces: a kernel whose threads read their requests once and keep them (load_once.cu).
constexpr uint32_t kOnceAlone = 4096;         // requests of one group that a single block takes
constexpr uint32_t kOnceWindows = 1024;       // windows of the sort, at most
struct OnceLoad {
    uint32_t blocks, per_block;           // blocks that read the trace, requests of each
    int seg_shift, win_shift;             // counters added up by a warp, ticks sorted at a time (their logarithms)
    unsigned long long* windows;          // [kOnceWindows][2]: complement of the first bin | where its ticks start, last bin + 1 | where they end
    uint4* clear;                         // words to set to zero on the way
    uint32_t clear_vecs;
    bool zeroed;                          // z and what lies behind it is zero already
};

struct LoadArgs {
    uint32_t n;
    int G;
    uint32_t ns, nd;
    // inputs in the caller's order: a trace's columns ...
    const int32_t *prompt, *outlen;
    const float* ttft;
    const uint8_t *sp, *dp;               // may be null
    // ... or packed (pack.cuh) ...
    const char* packed;
    // ... or ticks stored group after group (off[g] .. off[g + 1])
    const int32_t* ticks;
    const uint32_t* off;
    // where the kernel leaves a trace it reads from host memory, for its second pass (null: the columns are read twice)
    uint32_t *st_ticks, *st_ln;
    uint8_t* st_g;
    // Parts of the trace placed one after another (1: all at once), for traces whose records do not fit in L2: the blocks'
    // shares of all buckets are open at once, and what leaves L2 in parts is written twice.
    uint32_t rounds;
    LoadZero* z;
    size_t zero_bytes;                    // from z on: what must be zero (cleared by the launch where several blocks need it)
    uint32_t* cnt;                        // [G][4097] requests per prompt length (cleared)
    uint32_t* tick_cnt;                   // [G][kTickBins] (cleared)
    uint32_t* tick_start;                 // [G][kTickBins]
    uint32_t* tick_at;                    // [G][kTickBins] cursors, used when the groups' counters do not fit in shared memory
    uint2* windows;                       // [n / 4096 + G] of the sort: first and last bin (cleared)
    uint32_t* binned;                     // [n] ticks bin by bin
    // outputs
    uint4* req;                           // [n] internal order (by group, then by prompt length): see TraceDev
    uint32_t* inv;                        // [n] place of each of the caller's requests
    int32_t* sorted;                      // [n] ticks ascending within each group
    uint32_t* len_end;                    // [G][4097]
    int64_t* cum_mass;                    // [G][4098]
    uint32_t* grp_off;                    // [G + 1]
    int32_t* knots;                       // [G][257]
    uint64_t* fin_totals;                 // [2G]: output tokens per group, then requests per group
    LargeLoad large;
    OnceLoad once;
    LoadReadback* readback;               // its err holds 0, 0, 0, 2 (no report) before the launch
#ifdef DISCO_DEBUG
    uint32_t absent;                      // the wait that expects one arrival more than comes (from 1; 4: of the other blocks' sums);
                                          // 5: k_load_once's last block is late with its totals
#endif
};

cudaError_t run_load(const LoadArgs& a, int sms, cudaStream_t st);          // one kernel, after a memset
// The same for kLargeMinN to kLargeMaxN requests in at most kLargeMaxGroups groups: six kernels, after a memset.
cudaError_t run_load_large(const LoadArgs& a, int sms, cudaStream_t st);
// The same for as many requests as the threads can keep (eight each): one kernel, after a memset if `zeroed` is not
// set.
inline bool once_trace(uint32_t n, int G, uint32_t sms) {
    return G <= kLargeMaxGroups && sms > 2u * (uint32_t)G && n <= (std::min(sms, kLoadBlocks) - (uint32_t)G) * 8192u;
}
inline bool once_ticks(uint32_t n, int G, uint32_t sms) { return G <= 16 && n <= std::min(sms, kLoadBlocks) * 8192u; }
cudaError_t run_load_once(const LoadArgs& a, int sms, cudaStream_t st);
cudaError_t run_sort_ticks_once(const LoadArgs& a, int sms, cudaStream_t st);
cudaError_t run_sort_ttft_once(const LoadArgs& a, int sms, cudaStream_t st);
cudaError_t run_sort_ticks(const LoadArgs& a, int sms, cudaStream_t st);    // ticks, off, G, n -> sorted
cudaError_t run_sort_ttft(const LoadArgs& a, int sms, cudaStream_t st);     // ttft, n (one group) -> sorted

// The least-significant-digit radix sort, for samples that the kernels above give up on (err[3] = 1: more than 8,192 ticks
// in one bin, spread over more than 2^18 values).  keys_a, keys_b: n words each; counts: 256 * kRadixMaxBlocks + 256.
constexpr uint32_t kRadixMaxBlocks = 1024;
cudaError_t radix_sort_ticks(const int32_t* ticks, const uint32_t* off, int G, uint32_t total, uint64_t* keys_a, uint64_t* keys_b,
                             uint32_t* counts, int32_t* out, int sms, cudaStream_t st);
uint32_t radix_sort_launches(int G);

}  // namespace disco
