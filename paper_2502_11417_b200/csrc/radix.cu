// Stable least-significant-digit radix sort of (group, ticks), 8-bit digits: the fallback of the bin-wise sort in load.cu.
#include "load.cuh"

#include <algorithm>

#include "scan.cuh"

namespace disco {

namespace {

constexpr int kRadixThreads = 256;
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr uint32_t kWideBlocks = 4096;            // blocks of the kernels that take a key a thread, at most
// (a block's share of the keys is rounded up to whole rows of kRadixThreads, and its tiles reach 1,024 keys on)
static_assert(kMaxTicks + (uint64_t)(kRadixMaxBlocks + 8) * kRadixThreads <= 1ull << 32 &&
              kMaxTicks + (uint64_t)kWideBlocks * kRadixThreads <= 1ull << 32, "32-bit indices");

__global__ void k_radix_hist(const uint64_t* __restrict__ keys, uint32_t n, uint32_t per_block, int shift,
                             uint32_t* __restrict__ counts /* [256][gridDim.x] */) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t lo = min(n, blockIdx.x * per_block), hi = min(n, lo + per_block);
    for (uint32_t i = lo + threadIdx.x; i < hi; i += kRadixThreads)
        atomicAdd(&h[(uint32_t)(keys[i] >> shift) & 255u], 1u);
    __syncthreads();
    counts[threadIdx.x * gridDim.x + blockIdx.x] = h[threadIdx.x];
}

// One block per digit: exclusive scan of the digit's per-block counts, in place, and the digit's total.
__global__ void k_radix_rowscan(uint32_t* __restrict__ counts /* [256][blocks] */, uint32_t blocks,
                                uint32_t* __restrict__ totals /* [256] */) {
    __shared__ uint32_t wtot[32];
    uint32_t* row = counts + (size_t)blockIdx.x * blocks;
    const uint32_t per = (blocks + 127u) / 128u;
    const uint32_t lo = min(blocks, threadIdx.x * per), hi = min(blocks, lo + per);
    uint32_t s = 0;
    for (uint32_t i = lo; i < hi; ++i) s += row[i];
    uint32_t total;
    uint32_t run = block_inclusive_scan(s, wtot, &total) - s;
    for (uint32_t i = lo; i < hi; ++i) { const uint32_t c = row[i]; row[i] = run; run += c; }
    if (threadIdx.x == 0) totals[blockIdx.x] = total;
}

__global__ void k_radix_scatter(const uint64_t* __restrict__ keys_in, uint64_t* __restrict__ keys_out, uint32_t n,
                                uint32_t per_block, int shift, const uint32_t* __restrict__ offsets,
                                const uint32_t* __restrict__ totals) {
    __shared__ uint32_t run[256];                 // next output slot of each digit for this block
    __shared__ uint32_t wcnt[kRadixWarps][256];   // keys of each digit per warp in the current slab
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    {
        // offsets[d][b]: keys of digit d in earlier blocks (k_radix_rowscan); totals[d]: keys of digit d.
        // This block's first slot for digit d = keys of smaller digits + keys of d in earlier blocks.
        uint32_t* wtot = wcnt[0];                                    // scratch of the scan (32 words)
        const uint32_t total = totals[threadIdx.x], before = offsets[threadIdx.x * gridDim.x + blockIdx.x];
        const uint32_t incl = block_inclusive_scan(total, wtot, (uint32_t*)nullptr);
        run[threadIdx.x] = incl - total + before;
        __syncthreads();
    }
    const uint32_t lo = min(n, blockIdx.x * per_block), hi = min(n, lo + per_block);
    constexpr int kPer = 4;                                   // keys per thread and tile
    constexpr uint32_t kTile = kRadixThreads * kPer;          // a warp owns 128 consecutive keys of a tile
    for (uint32_t base = lo; base < hi; base += kTile) {
        for (int k = 0; k < kRadixWarps; ++k) wcnt[k][threadIdx.x] = 0;
        uint64_t key[kPer];
        uint32_t dig[kPer], peers[kPer];
        bool live[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const uint32_t i = base + w * (32 * kPer) + j * 32 + lane;
            live[j] = i < hi;
            key[j] = live[j] ? keys_in[i] : 0;
            dig[j] = (uint32_t)(key[j] >> shift) & 255u;
            // lanes holding the same digit, from eight ballots over the digit's bits
            uint32_t m = __ballot_sync(0xFFFFFFFFu, live[j]);
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const uint32_t bal = __ballot_sync(0xFFFFFFFFu, (dig[j] >> b) & 1u);
                m &= ((dig[j] >> b) & 1u) ? bal : ~bal;
            }
            peers[j] = m;
        }
        __syncthreads();
        // keys of each digit in each warp (a warp's row is its own: plain adds, rounds in order)
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            if (live[j] && (peers[j] & ((1u << lane) - 1u)) == 0) wcnt[w][dig[j]] += __popc(peers[j]);
            __syncwarp();
        }
        __syncthreads();
        {   // turn the counts into each warp's first slot per digit; advance the block's running slots
            uint32_t at = run[threadIdx.x];
            for (int k = 0; k < kRadixWarps; ++k) { const uint32_t c = wcnt[k][threadIdx.x]; wcnt[k][threadIdx.x] = at; at += c; }
            run[threadIdx.x] = at;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            if (live[j]) {
                const uint32_t pos = wcnt[w][dig[j]] + __popc(peers[j] & ((1u << lane) - 1u));
                if (DBG_OK(pos, n, DBG_K_RADIX, DBG_ELEMENT)) keys_out[pos] = key[j];
            }
            __syncwarp();
            if (live[j] && (peers[j] & ((1u << lane) - 1u)) == 0) wcnt[w][dig[j]] += __popc(peers[j]);
            __syncwarp();
        }
        __syncthreads();
    }
}


// Sort keys (group << 32 | ticks) for ticks stored group after group.
__global__ void k_keys_of_grouped_ticks(uint32_t total, const int32_t* __restrict__ ticks, const uint32_t* __restrict__ off,
                                        int G, uint64_t* __restrict__ keys) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        int g = 0;
        while (g + 1 < G && i >= off[g + 1]) ++g;
        keys[i] = ((uint64_t)(uint32_t)g << 32) | (uint32_t)max(ticks[i], 0);
    }
}

__global__ void k_low_words(uint32_t n, const uint64_t* __restrict__ keys, int32_t* __restrict__ out) {
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x)
        out[k] = (int32_t)(uint32_t)keys[k];
}

}  // namespace

DBG_TRANSLATION_UNIT()

uint32_t radix_sort_launches(int G) { return 2 + 3 * (G > 1 ? 5 : 4); }

cudaError_t radix_sort_ticks(const int32_t* ticks, const uint32_t* off, int G, uint32_t total, uint64_t* keys_a, uint64_t* keys_b,
                             uint32_t* counts, int32_t* out, int sms, cudaStream_t st) {
    if (total == 0) return cudaSuccess;
    const uint32_t wide = std::min<uint32_t>((total + 255u) / 256u, std::min((uint32_t)sms * 16u, kWideBlocks));
    k_keys_of_grouped_ticks<<<wide, 256, 0, st>>>(total, ticks, off, G, keys_a);
    uint32_t blocks = std::min<uint32_t>((total + 1023u) / 1024u, kRadixMaxBlocks);
    uint32_t per_block = (total + blocks - 1) / blocks;
    per_block = (per_block + kRadixThreads - 1) / kRadixThreads * kRadixThreads;
    uint32_t* totals = counts + (size_t)256u * blocks;
    const int passes = G > 1 ? 5 : 4;                   // the ticks' four bytes, then the group id
    for (int p = 0; p < passes; ++p) {
        k_radix_hist<<<blocks, kRadixThreads, 0, st>>>(keys_a, total, per_block, 8 * p, counts);
        k_radix_rowscan<<<256, 128, 0, st>>>(counts, blocks, totals);
        k_radix_scatter<<<blocks, kRadixThreads, 0, st>>>(keys_a, keys_b, total, per_block, 8 * p, counts, totals);
        std::swap(keys_a, keys_b);
    }
    k_low_words<<<wide, 256, 0, st>>>(total, keys_a, out);
    return cudaGetLastError();
}

}  // namespace disco
