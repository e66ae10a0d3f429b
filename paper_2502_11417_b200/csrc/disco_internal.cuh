// Internal declarations shared by the translation units of libdisco.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "disco.h"

namespace disco {

constexpr int kNBins = DISCO_NBINS;
constexpr int kMaxPrompt = DISCO_MAX_PROMPT;
constexpr int kMaxOutput = DISCO_MAX_OUTPUT;
constexpr int kNKnots = 257;
constexpr int kMaxGroups = 64;

// ---- per-group constants, ticks and costs (one per (server, device) profile pair) ----
struct GroupConst {
    int32_t T_srv, J_srv;        // server decode interval and jitter amplitude, ticks
    int32_t T_dev, J_dev;        // device decode interval and jitter amplitude
    int32_t kappa, c0;           // device TTFT = kappa * l + c0
    int32_t auto_device_constrained;   // Algorithm 1 evaluated on this group's costs
    int32_t candidate;           // 0 none, 1 a winning server may migrate (it is the dearer decoder), 2 a winning device may
    float delta_c;               // |c^d_s - lambda c^d_d|  (Eq. 5)
    float cps, cds, lcpd, lcdd;  // fp32 cost rates, device ones already in money
    double cps_d, cds_d, cpd_d, cdd_d, lambda_d;   // fp64 rates for the totals
};

// ---- per-policy constants derived on the host ----
struct PolicyConst {
    float budget, alpha, theta;
    uint32_t flags;
    int32_t tau, B;
    int32_t cls;                 // timeline class (policies with equal tau, B, pacing share play-outs)
    int32_t mode;                // 0 Algorithm 1 decides, 1 device-constrained, 2 server-constrained
    uint32_t expected_len;       // 0 = true remainder in the migration trigger
    uint32_t route_thr;          // stochastic routing: constrained endpoint iff hash < route_thr (or route_all)
    int32_t route_all;
    uint32_t l_immediate;        // Eq. 1's immediate-start threshold (beta rule)
};

// ---- the same for the preparation: what differs from policy to policy, and the rest, which most of them share (a thousand
//      policies then go with a launch, 28 KB at most, that took 57 KB) ----
struct PolicyIn { float budget, theta; uint32_t kind, route_thr; };
struct PolicyKind {
    float alpha;
    uint32_t flags;
    int32_t mode;
    uint32_t expected_len, l_immediate, pad[3];
};

// ---- what Algorithms 1-3 produce for one (group, policy) ----
struct Prep {
    int32_t device_constrained;
    int32_t l_th;
    int32_t l_star;
    int32_t w_star, w_tail;
    float theta;
    int32_t mig_on;
    int32_t stochastic;          // random routing instead of Algorithms 2-3
    uint32_t expected_len, route_thr;
    int32_t route_all;
    int32_t beta_rule;           // Eq. 1-2 variant: l_star holds the immediate-start threshold, w_star the slope beta
};

// ---- a timeline class: the parameters a play-out depends on besides the request ----
// How the streams of a group behave under a class, which decides the kernel that plays its requests:
//   G_EXACT    no interval of either stream can exceed tau: everything is delivered at the pace, but the token after a
//              hand-off.  Only the hand-off is played; sums, maxima and windows follow from the lengths.
//   G_FREE     a stream either cannot clamp, as above, or clamps at every token (or pacing is off): it is delivered as
//              it is generated, TBT = x_j.
//   G_GENERAL  anything else.
enum GroupKind { G_EXACT = 0, G_FREE = 1, G_GENERAL = 2 };
struct ClassConst {
    int32_t tau_eff;             // tau when pacing is on, else 0 (then delivery = generation)
    int32_t tau;                 // tau of the policies (for the "equals tau" fast count)
    int32_t B;
    int32_t pacing, mig_any;
    // dense windows of histogram bins that regular inter-token intervals can fall in
    int32_t W[3];                // bins per request for the server, device and migrated timelines
    int32_t lo[kMaxGroups][3];   // first bin of each window, per group
    int32_t ktau[kMaxGroups][3]; // index of bin(tau) inside the window, or -1
    // G_EXACT: tokens the search for the hand-off may have to look at.  Every token adds at least tau - (T + J) to the
    // delivery lag, so (B-1) tau is passed within that many.
    uint32_t search[kMaxGroups];
    uint8_t kind[kMaxGroups];    // GroupKind
    uint8_t even[kMaxGroups];    // bit s: every regular interval of stream s equals tau, and its windows are not stored
};

// Per-request summaries of the up to three distinct decode timelines of a class.
struct TimelineRec {
    uint2* hand;                 // [n]: hand-off index (0 = buffer never fills) | delayed tokens << 16, and the TBT of the
                                 // first token after the hand-off
    uint32_t *sum[3], *max[3];   // d_n - d_1 and the largest TBT, ticks ([n] each; not of G_EXACT groups)
    uint16_t* win[3];            // [n][W[c]] counts per window bin (not of streams that are even)
};

struct TraceDev {
    uint32_t n;
    int32_t n_groups;
    const uint4* req;            // internal order (by group, inside a group by prompt length): server TTFT ticks,
                                 // prompt length | output length << 16, caller's index, unused
    const uint32_t* inv;         // place of each of the caller's requests in the internal order
    const uint32_t* len_end;     // [G][4097]: where the group's requests of each prompt length end (the next length starts)
    const uint32_t* grp_off;     // [G+1]
};

struct Chunk { uint32_t start, len; int32_t g; int32_t pad; };

enum AccSlot { A_SERVER_ONLY = 0, A_DEVICE_ONLY, A_RACE, A_STARTED, A_DEVICE_WON, A_MIGR, A_TOK_DEVICE,
               A_PRE_SERVER, A_PRE_DEVICE, A_DELAYED, A_TTFT_SUM, A_TAU_CNT, kNAcc };

// ---- device helpers -------------------------------------------------------------------------------------

// Jitter hash: xorshift-multiply finaliser over a per-request key plus token counter.
__host__ __device__ __forceinline__ uint32_t mix32(uint32_t x) {
    x ^= x >> 16; x *= 0xA54FF53Bu;
    x ^= x >> 15; x *= 0x510E527Fu;
    x ^= x >> 16;
    return x;
}
constexpr uint32_t kHashSeed = 0x6A09E667u, kHashReq = 0xBB67AE85u, kHashTok = 0x3C6EF373u;

__host__ __device__ __forceinline__ uint32_t seed_key(uint64_t seed) {
    return mix32((uint32_t)seed ^ kHashSeed) ^ (uint32_t)(seed >> 32);
}

#ifdef __CUDACC__
// Histogram bin of a tick count: exact below 32, then 32 bins per octave.  The exponent and the five
// leading mantissa bits come from the float representation (round-toward-zero keeps them exact).
__device__ __forceinline__ int bin_of_ticks(uint32_t t) {
    if (t < 32u) return (int)t;
    int b = (int)(__float_as_uint(__uint2float_rz(t)) >> 18) - ((127 + 4) << 5);
    return min(b, kNBins - 1);
}
#endif

// Host-side bin (same partition of the axis, integer arithmetic).
inline int host_bin_of_ticks(int64_t t) {
    if (t < 0) t = 0;
    if (t < 32) return (int)t;
    int e = 63 - __builtin_clzll((unsigned long long)t);
    int64_t b = 32 * (int64_t)(e - 4) + ((t >> (e - 5)) & 31);
    return (int)(b < kNBins - 1 ? b : kNBins - 1);
}

// Lower edge of a bin, ticks.
inline int64_t host_bin_edge_ticks(int b) {
    return b < 32 ? (int64_t)b : (int64_t)(32 + (b & 31)) << ((b >> 5) - 1);
}

#ifdef __CUDACC__
// Launch that lets the grid be scheduled while its predecessor in the stream is still draining (programmatic
// stream serialisation).  grid_dependency_wait() returns once the predecessor has completed, its own waits included, and its writes are
// visible.  The rule: a kernel waits before it reads or writes global memory -- unless all that it touches (what it reads, what it
// writes and who else may write there) was complete before the blocks of its predecessor let it start; then at least one of its
// blocks waits before it ends, and before it lets a successor start that needs the predecessor's results.  So a kernel's completion
// always means that of all in front of it.  Who goes in front of its wait, and why it may, is said at each such kernel: k_prep, k_ticks, k_order,
// k_sort, k_grid, k_spread, k_playout_free.
template <class... KArgs, class... Args>
inline cudaError_t launch_after(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel of the stream start once every block of this one has come here (or ended); what it may do in front of
// its own wait is up to it.  To be called behind this kernel's wait, or where the successor touches nothing that a kernel in front of this
// one may still work on (k_order's other blocks, k_grid beside its predecessor).
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// add + ((h * mul) >> 32) in one instruction
__device__ __forceinline__ uint32_t mad_hi(uint32_t h, uint32_t mul, uint32_t add) {
    uint32_t x;
    asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(x) : "r"(h), "r"(mul), "r"(add));
    return x;
}

// The stream after a hand-off stores no window of its own where groups are played free without pacing: it is stream
// x_stream's (0 the server's, 1 the device's) without the interval in front of token 2, whose bin first_bin gives.  -1: it
// stores one, if it has any.
__device__ __forceinline__ int x_stream(const ClassConst& cc, const GroupConst& gc) {
    return cc.pacing ? -1 : (gc.candidate == 1 ? 1 : 0);
}
__device__ __forceinline__ int first_bin(const GroupConst& gc, int stream, uint32_t k0, uint32_t orig) {
    const uint32_t h = mix32(mix32(k0 + orig * kHashReq) + 2u * kHashTok);
    const int32_t T = stream ? gc.T_dev : gc.T_srv, J = stream ? gc.J_dev : gc.J_srv;
    return bin_of_ticks((uint32_t)(T - J) + __umulhi(h, 2u * (uint32_t)J + 1u));
}

// The batch-th batch of `size` requests among the groups of one kind: its group, first request and length.
__device__ __forceinline__ bool batch_of_kind(const TraceDev& tr, const ClassConst& cc, int kind, uint32_t size, uint32_t batch,
                                              int& g, uint32_t& k_lo, uint32_t& count) {
    for (g = 0; g < tr.n_groups; ++g) {
        if (cc.kind[g] != kind) continue;
        const uint32_t lo = tr.grp_off[g], len = tr.grp_off[g + 1] - lo, here = (len + size - 1u) / size;
        if (batch < here) { k_lo = lo + batch * size; count = min(size, len - batch * size); return true; }
        batch -= here;
    }
    return false;
}
#endif

// Lets a kernel use that much dynamic shared memory, once per kernel and device.
cudaError_t allow_smem(const void* kernel, size_t bytes);

// Records the calling thread's error message (read back by disco_last_error) and returns `code`.
int set_error(int code, const char* msg);

// ---- checked build (-DDISCO_DEBUG) -----------------------------------------------------------------------
// Every index a kernel derives from data or from its launch geometry -- request, policy, group, chunk, knot,
// histogram bin, window slot, staging slot, table entry -- goes through DBG_OK(index, bound, kernel, what) before
// the access.  An index outside [0, bound) is recorded (first one wins) and the access is skipped: nothing traps,
// the context stays usable, and the next call that synchronises returns DISCO_ECUDA naming kernel and index.
// In the ordinary build DBG_OK is the constant true and the checks vanish.
enum DbgKernel { DBG_K_INGEST = 1, DBG_K_RADIX, DBG_K_GATHER, DBG_K_TABLES, DBG_K_PREP, DBG_K_PLAYOUT_FAST, DBG_K_PLAYOUT,
                 DBG_K_PAIRS_ACC, DBG_K_GRID, DBG_K_PAIRS_ROWS, DBG_K_FINALIZE, DBG_K_SELECT, DBG_K_SELFTEST,
                 DBG_K_COUNT };
enum DbgWhat { DBG_REQUEST = 1, DBG_POLICY, DBG_GROUP, DBG_CHUNK, DBG_KNOT, DBG_BIN, DBG_WINDOW, DBG_SLOT, DBG_TABLE,
               DBG_COUNTER, DBG_ELEMENT, DBG_WHAT_COUNT };
#ifdef DISCO_DEBUG
#ifdef __CUDACC__
static __device__ int32_t dbg_word[4];          // one per translation unit: kernel, what, index, bound
__device__ __forceinline__ bool dbg_in(long long i, long long n, int kernel, int what) {
    if (i >= 0 && i < n) return true;
    if (atomicCAS(&dbg_word[0], 0, kernel) == 0) {
        dbg_word[1] = what;
        dbg_word[2] = (int32_t)(i < -2147483647LL ? -2147483647LL : (i > 2147483647LL ? 2147483647LL : i));
        dbg_word[3] = (int32_t)(n > 2147483647LL ? 2147483647LL : n);
    }
    return false;
}
#define DBG_OK(i, n, kernel, what) (::disco::dbg_in((long long)(i), (long long)(n), (kernel), (what)))
// Reads (and clears) this translation unit's record; registered with the host side once per unit that has kernels.
void dbg_register(cudaError_t (*reader)(int32_t*));
struct DbgRegistrar { explicit DbgRegistrar(cudaError_t (*r)(int32_t*)) { dbg_register(r); } };
#define DBG_TRANSLATION_UNIT()                                                                         \
    namespace {                                                                                        \
    cudaError_t dbg_read_unit(int32_t* out) {                                                          \
        cudaError_t e = cudaMemcpyFromSymbol(out, ::disco::dbg_word, 16);                              \
        if (e == cudaSuccess && out[0]) { const int32_t z[4] = {0, 0, 0, 0}; e = cudaMemcpyToSymbol(::disco::dbg_word, z, 16); } \
        return e;                                                                                      \
    }                                                                                                  \
    ::disco::DbgRegistrar dbg_registrar_unit(dbg_read_unit);                                           \
    }
#endif
#else
#define DBG_OK(i, n, kernel, what) true
#define DBG_TRANSLATION_UNIT()
#endif

// ---- launch wrappers (defined in the kernel translation units) -------------------------------------------
// The small tables of an evaluation on their way to the device with k_prep: as its parameter up to kTablesInline bytes, beyond
// it reads them in pinned host memory.
constexpr size_t kTablesInline = 28672;      // (a launch takes 32,764 bytes of parameters, the chunk plans 3,072)
struct ChunkPlan { uint32_t first, start, end; int32_t g; };     // a group's chunks: number of the first, requests [start, end)
enum { CHUNKS_RUNS, CHUNKS_PAIRS, CHUNKS_JOINED, kChunkTables };   // of the grid kernel run by run, of the pair kernel, of the grid kernel side by side
struct TablesIn {
    const void* host;            // the policies come first, then their kinds; room for kTablesInline bytes where they go as a parameter
    void* device;
    uint32_t vecs, skip;         // of 16 bytes; how many of them (policies and kinds) no kernel behind needs
    uint32_t kinds;
    // chunk tables that k_prep writes out, group by group
    ChunkPlan plan[kChunkTables][kMaxGroups];
    uint32_t n_plan[kChunkTables], chunk_len[kChunkTables], n_chunks[kChunkTables];
    Chunk* chunks[kChunkTables];
    // in pinned host memory only
    uint32_t* left;              // device word, zero; blocks that have read their share (zero again when all have)
    volatile uint32_t* read;     // pinned host word: set to `turn` once all have
    uint32_t turn;
};
cudaError_t launch_prep(uint32_t P, int G, const GroupConst* gc, const int64_t* cum_mass,
                        const uint32_t* cnt, const int32_t* sorted, const uint32_t* grp_off, Prep* prep, const TablesIn& tables,
                        void* clear, size_t clear_bytes /* a multiple of 16: set to zero on the way */, int sms, cudaStream_t st);
cudaError_t launch_prep_beta(const PolicyIn* pol, const PolicyKind* kinds, uint32_t P, const int64_t* cum_mass, const uint32_t* cnt,
                             const int32_t* sorted, const uint32_t* grp_off,
                             const uint32_t* tick_start, const uint32_t* tick_cnt /* [G][kTickBins], of the sorted ticks */,
                             const uint32_t* pairs /* [n_pairs]: g P + p */, uint32_t n_pairs,
                             uint64_t most /* ticks of a group, at most */, Prep* prep, bool early /* the grid kernel follows: it may start beside */,
                             cudaStream_t st);
// Further classes whose free streams are the same (api.cu): the play-out writes their summaries as well, so many bytes from its own.
constexpr int kFreeMore = 8;
struct FreeMore { int n; int32_t tau[kFreeMore]; ptrdiff_t off[kFreeMore]; };
// Plays every request under one class.  `kinds`: bit k set if some group with requests is of GroupKind k; `batches[k]`:
// batches of 32 requests of the groups of kind k.
cudaError_t launch_timeline(const TraceDev& tr, const GroupConst* gc, const ClassConst& cc, const int32_t* knots, uint32_t k0 /* hash key base: seed_key(seed) + first_index * kHashReq */,
                            TimelineRec rec, int32_t* err, uint32_t* ticket /* one word */, uint32_t kinds,
                            const uint32_t* batches, uint32_t search /* largest ClassConst::search of a group with requests */,
                            bool long_outputs /* mean output length of 512 tokens or more */,
                            cudaEvent_t mid /* recorded between the kernels of exact groups and the others, or null */,
                            const FreeMore& more, uint32_t* free_ticket /* one word, zero before and after */, const uint32_t* grp_n /* requests per group, on the host */,
                            bool beside /* the first kernel runs beside its predecessor (only one of streams that never wait for the reader) */, bool early /* the preparation follows: it may start beside the last kernel */,
                            int sms /* multiprocessors of the device */, cudaStream_t st);
uint32_t timeline_launches(uint32_t kinds);
// The exact groups of several classes whose searches are short, in one launch.
constexpr int kShortMany = 16;
struct ShortMany { const ClassConst* classes; size_t rec_stride; uint32_t count, cls[kShortMany], slot[kShortMany]; };
bool short_search(uint32_t search);
cudaError_t launch_playout_many(const TraceDev& tr, const GroupConst* gc, const int32_t* knots, uint32_t k0, TimelineRec rec /* of slot 0 */,
                                const ShortMany& many, bool early /* its successor runs beside it */, int sms, cudaStream_t st);

// Reductions over a grid of plain policies, budget by overhead (grid.cu).
constexpr int kGridRows = 8;     // overheads a slab may have
constexpr int kGridCols = 256;   // budgets a slab may have
struct Slab {
    int32_t K, T;                // distinct budgets (columns, ascending), distinct overheads (rows, ascending)
    uint32_t cols;               // index into the tables: policy whose preparation stands for each column, [K]
    uint32_t cells;              // index into the tables: policy of (column, row), [K][T], ~0 where there is none
    uint32_t expected_len;
    int32_t mig;                 // the policies migrate
    uint32_t policies;           // how many they are
    int32_t mixed;               // a column per policy, whose overheads lie between theta[0] and theta[1] (T = 1):
                                 // requests whose saving lies between the two are left to the pair kernel
    uint32_t cls, slot, win_slot;  // its class, where the class's records lie, and its windows (both in places of rec_stride bytes)
    int32_t bin_tau;             // the bin of the class's pace
    float theta[kGridRows];
    // 32- or 64-bit words in front of the slab's difference tables, see grid.cu
    uint64_t ttft, tbt, sums;
};
struct GridTables { uint32_t* ttft; void* tbt; unsigned long long* sums; };
struct LeftLists { uint32_t* list; uint32_t* count; };   // [slabs][n] places in the internal order, [slabs][G]
uint64_t grid_ttft_words(int K), grid_tbt_words(int K, int T), grid_sum_words(int K, int T, int G);
uint32_t grid_blocks_per_sm(int T);
bool grid_joins(uint32_t n, int groups /* that have requests */, int K, int T, bool inner /* a budget lies between 0 and 1 */);   // small traces under many policies: requests side by side
int grid_rows(int T);            // rows the kernel that takes such a slab is built for
cudaError_t launch_grid(const TraceDev& tr, const GroupConst* gc, const ClassConst* classes, const Prep* prep, uint32_t P,
                        const Slab* slabs, uint32_t n_slabs, int T /* most rows of a slab */, bool wide /* of all of them */,
                        const uint32_t* tab, const Chunk* chunks, uint32_t n_chunks, TimelineRec rec /* of slot 0 */, size_t rec_stride, GridTables gt,
                        LeftLists left /* of these slabs, or nulls: none is mixed */, uint32_t k0, uint32_t* ticket /* zero */,
                        uint64_t* work /* [4], added to */, bool beside /* runs beside its predecessor, whose own it has complete */,
                        bool early /* its successor runs beside it */,
                        bool waits /* Algorithm 2 decides in some group */, bool joined /* requests side by side, not run by run */, int sms, cudaStream_t st);
cudaError_t launch_spread(const TraceDev& tr, const GroupConst* gc, const Slab* slabs, uint32_t n_slabs, int T,
                          bool wide, const uint32_t* tab, GridTables gt, uint64_t* acc, uint64_t* hist_ttft,
                          uint64_t* hist_tbt, bool beside, bool early /* as above */, cudaStream_t st);
// Pair by pair: `n_list` policies under the chunks' requests, or (list not null) under the listed ones.
cudaError_t launch_pairs_acc(const TraceDev& tr, const GroupConst* gc, const ClassConst* cc, const Prep* prep, uint32_t P,
                             const uint32_t* pol_list, uint32_t n_list, const Chunk* chunks, uint32_t n_chunks,
                             const uint32_t* list /* [n] */, const uint32_t* list_count /* [G] */, TimelineRec rec,
                             uint64_t* acc, uint64_t* hist_ttft, uint64_t* hist_tbt, uint64_t* work, uint32_t k0,
                             bool extras /* some policy routes at random or waits by Eq. 1-2 */,
                             bool wide /* some window W of the class spans several bins */, cudaStream_t st);
// Fills tr.inv (a large trace's load leaves that to the evaluation that writes rows).
cudaError_t launch_inverse(const TraceDev& tr, uint32_t* inv, cudaStream_t st);
cudaError_t launch_pairs_rows(const TraceDev& tr, const GroupConst* gc, const ClassConst* cc, const Prep* prep, uint32_t P,
                              const uint32_t* pol_list, uint32_t n_list, TimelineRec rec, const disco_pair_out_t& out,
                              uint32_t k0, bool extras, cudaStream_t st);
cudaError_t launch_finalize(uint32_t P, int G, const GroupConst* gc, const uint64_t* acc, const uint64_t* hist_ttft,
                            const uint64_t* hist_tbt,
                            const uint64_t* fin_totals /* [2G]: output tokens per group, then requests per group */,
                            disco_policy_stats_t* stats /* [P] */,
                            disco_policy_stats_t* stats_host /* [P], pinned host memory, written by the kernel */,
                            const int32_t* err, int32_t* err_host /* pinned: a copy of err */, cudaStream_t st);
cudaError_t launch_select(const disco_policy_stats_t* stats, uint32_t P, double cost_cap, float tbt_slo_s,
                          int32_t* result /* [2]: status, index; may be pinned host memory */, cudaStream_t st);
// Cumulative token mass and knots from tables given by the caller (F_off[g] .. F_off[g+1] delimit group g's ticks).
cudaError_t launch_tables_imported(int G, const uint32_t* cnt, int64_t* cum_mass, const int32_t* F_sorted,
                                   const uint32_t* F_off, int32_t* knots, cudaStream_t st);
// Checked build: 0, or DISCO_ECUDA (error string set) if a kernel refused an index since the last call.  Always 0 in
// an ordinary build.  To be called after the stream has been synchronised.
int check_debug_record();
#ifdef DISCO_DEBUG
// Launches a kernel whose only access uses an index beyond its bound (refused by the check, never made).
cudaError_t run_debug_selftest(cudaStream_t st);
#endif
// Times the token loop's instruction mix on every multiprocessor; *token_steps_per_s receives the rate.
cudaError_t run_alu_peak(int sms, double* token_steps_per_s, cudaStream_t st);

}  // namespace disco
