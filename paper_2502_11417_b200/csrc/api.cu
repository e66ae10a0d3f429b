// Host side of the C ABI: argument checks, device memory, launch order.  No arithmetic of the method runs
// here apart from turning the handful of profile and policy parameters into ticks.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <new>
#include <numeric>
#include <string>
#include <vector>

#include "disco_internal.cuh"
#include "load.cuh"
#include "pack.cuh"

using namespace disco;

namespace {

thread_local std::string g_err;
std::atomic<uint64_t> g_launches{0};   // kernels launched by this library, all contexts

int fail(int code, const std::string& msg) { g_err = msg; return code; }
int fail_cuda(cudaError_t e, const char* what) {
    g_err = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? DISCO_ENOMEM : DISCO_ECUDA;
}
// Nothing throws across the C boundary.  (Messages that a string holds without allocating.)
#define DISCO_CATCH                                                          \
    catch (const std::bad_alloc&) { return fail(DISCO_ENOMEM, "out of memory"); } \
    catch (...) { return fail(DISCO_ECUDA, "host exception"); }
#define CU(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) return fail_cuda(e_, #call); } while (0)

// A growable device buffer.
struct DevBuf {
    void* p = nullptr;
    size_t cap = 0;
    cudaError_t reserve(size_t bytes) {
        if (bytes <= cap && p) return cudaSuccess;
        if (p) { cudaFree(p); p = nullptr; cap = 0; }
        if (bytes < 16) bytes = 16;
        cudaError_t e = cudaMalloc(&p, bytes);
        if (e == cudaSuccess) cap = bytes;
        return e;
    }
    void release() { if (p) cudaFree(p); p = nullptr; cap = 0; }
    template <class T> T* as() const { return (T*)p; }
};

// Places several arrays in one buffer, each on a 256-byte boundary.
struct Layout {
    size_t bytes = 0;
    size_t take(size_t n) { const size_t at = bytes; bytes += (n + 255) / 256 * 256; return at; }
};

int64_t ticks_of_seconds(float s) { return llrint((double)s * 1e6); }
int64_t ticks_of_rate(float per_s) { return llrint(1e6 / (double)per_s); }

using HostReadback = LoadReadback;   // pinned host mirror of the load's read-back block

}  // namespace

namespace disco {
int set_error(int code, const char* msg) {
    try { return fail(code, msg); } catch (...) { g_err.clear(); return code; }
}

cudaError_t allow_smem(const void* kernel, size_t bytes) {
    // (kernel, device, size) that have been allowed: a few dozen at most
    struct Allowed { const void* kernel; int device; size_t bytes; };
    static thread_local std::vector<Allowed> seen;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e) return e;
    for (const Allowed& x : seen) if (x.kernel == kernel && x.device == dev && x.bytes >= bytes) return cudaSuccess;
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes))) return e;
    try { seen.push_back({kernel, dev, bytes}); } catch (...) {}       // (asked for again, then)
    return cudaSuccess;
}

#ifdef DISCO_DEBUG
namespace {
std::vector<cudaError_t (*)(int32_t*)>& dbg_readers() { static std::vector<cudaError_t (*)(int32_t*)> v; return v; }
}  // namespace
void dbg_register(cudaError_t (*reader)(int32_t*)) { dbg_readers().push_back(reader); }
#endif
}  // namespace disco

namespace {
// Checked build: after a call has synchronised, asks every translation unit for an index its kernels refused.
// Returns 0, or DISCO_ECUDA with the kernel and the index in the error string.
int debug_check() {
#ifdef DISCO_DEBUG
    static const char* kernels[DBG_K_COUNT] = {"", "trace ingestion (counting)", "sort of the ticks", "trace ingestion (placing)", "group tables", "k_prep",
                                               "k_playout_fast", "k_playout", "k_pairs_acc", "k_grid", "k_pairs_rows",
                                               "k_finalize", "k_select", "self-test"};
    static const char* whats[DBG_WHAT_COUNT] = {"", "request", "policy", "group", "chunk", "knot", "histogram bin",
                                                "window slot", "staging slot", "table entry", "counter", "element"};
    for (auto reader : disco::dbg_readers()) {
        int32_t w[4] = {0, 0, 0, 0};
        const cudaError_t e = reader(w);
        if (e != cudaSuccess) return fail_cuda(e, "reading the checked build's record");
        if (w[0]) {
            const char* k = w[0] > 0 && w[0] < DBG_K_COUNT ? kernels[w[0]] : "?";
            const char* t = w[1] > 0 && w[1] < DBG_WHAT_COUNT ? whats[w[1]] : "?";
            return fail(DISCO_ECUDA, std::string("checked build: ") + k + " refused " + t + " index " + std::to_string(w[2]) +
                                         " (bound " + std::to_string(w[3]) + ")");
        }
    }
#endif
    return 0;
}
}  // namespace

struct disco_ctx {
    uint32_t n = 0, ns = 0, nd = 0;
    int G = 0;
    bool loaded = false;
    std::vector<GroupConst> gc;
    std::vector<GroupConst> gc_dev;   // what d_gc holds (a reload with the same profiles skips the copy)
    const void* gc_dev_at = nullptr;
    struct View { void* p = nullptr; template <class T> T* as() const { return (T*)p; } };
    // trace: one buffer for everything a load writes, and what a load needs in between
    DevBuf trace_mem, d_gc;
    View req, inv, sorted, len_end, tick_start, binned, zero, cum_mass, grp_off, knots;   // `zero`: what a load must clear
    View in_prompt, in_out, in_ttft, in_sp, in_dp;        // copies of host inputs
    View packed;                                          // ... or the same packed (pack.cuh)
    View st_ticks, st_ln, st_g;                           // ... or what the ingestion leaves when it reads host memory in place
    View fin_totals;                   // [2G] u64: output tokens and requests per group that the accumulators cover
    std::unique_ptr<Packer> packer;
    DevBuf keys_a, keys_b, radix_counts, sort_in;         // radix sort (fallback) and the sort of imported ticks
    uint64_t first_index = 0;          // index of request 0 in the whole trace (hash key base)
    int sms = 0;                       // multiprocessors of the context's device
    // F as Algorithms 1-3 read it: the trace's own sorted ticks, or a whole trace's given by the caller
    DevBuf F_sorted_imp, F_off_imp;
    const int32_t* F_sorted = nullptr;
    const uint32_t* F_off = nullptr;
    bool tables_imported = false;
    std::vector<uint64_t> F_n;         // requests per group behind F (the group's own count unless imported)
    bool fin_imported = false;         // fin_totals holds a caller's merged totals, not this trace's
    std::vector<uint64_t> fin_own;     // this trace's totals, to put back before the next evaluation
    LargeLoad large;                   // working memory of a large trace's load
    bool large_now = false;            // this trace is loaded by load_large.cu's kernels
    size_t trace_too_much = ~(size_t)0, rec_too_much = ~(size_t)0;   // bytes that trace_mem and rec_mem could not get, at least
    bool inv_there = false;            // `inv` has been written
    // What a load must clear lies twice in memory where load_once.cu's kernel loads the trace: it works in one half and clears the
    // other for the next load.  Where they lie (nowhere after any other load) and which of them is zero.
    struct Halves { void* at = nullptr; size_t cap = 0, bytes = 0; bool zero[2] = {false, false}; int now = 0; } halves;
    LoadZero* z = nullptr;
    uint32_t *cnt = nullptr, *tick_cnt = nullptr;
    uint2* windows = nullptr;
    int32_t* err = nullptr;
    size_t zero_bytes = 0;
    HostReadback* rb = nullptr;
    // evaluation
    uint32_t P = 0;
    bool evaluated = false, reduced = false;
    std::vector<PolicyConst> pol;
    DevBuf rec_mem;              // what the play-out writes
    DevBuf eval_mem;             // one buffer for everything else an evaluation writes
    View d_prep, d_accum, d_stats, d_tables, d_grid, d_left;
    View d_acc, d_hist_ttft, d_hist_tbt, d_work;          // regions of d_accum; d_work: the counters in front of d_grid
    View play_ticket, rec_hand, rec_u32[6], rec_win[3];      // regions of rec_mem
    std::vector<uint4> tables_host;   // the small host->device tables where they go with a launch
    void* stage = nullptr;       // pinned staging for the small host->device tables
    size_t stage_cap = 0;
    cudaEvent_t stage_free = nullptr;    // behind the copies that read it
    uint32_t stage_turn = 0;     // evaluations that have had their tables read there by a kernel, which puts their number into stage_read
    volatile uint32_t* stage_read = nullptr;   // in the pinned block of rb
    int32_t* sel_host = nullptr; // [2], in the pinned block of rb
    uint32_t* tab_host = nullptr;   // pinned copy of the group tables: [G][4097] length counts, then [G][257] knots
    int tab_host_groups = 0;        // groups it has room for
    bool tab_host_now = false;      // it holds the current tables
    void* stats_host = nullptr;  // pinned mirror of the statistics
    size_t stats_host_cap = 0;
    bool timing = false;         // record events around the play-out and pair kernels
    cudaEvent_t ev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    float ms[4] = {0.f, 0.f, 0.f, 0.f};   // clamp-free play-out, general play-out, pair reductions, pair rows
    bool timing_valid = false;

    ~disco_ctx() {
        DevBuf* all[] = {&trace_mem, &d_gc, &keys_a, &keys_b, &radix_counts, &sort_in, &F_sorted_imp, &F_off_imp, &rec_mem, &eval_mem};
        for (DevBuf* b : all) b->release();
        if (rb) cudaFreeHost(rb);
        if (stage) cudaFreeHost(stage);
        if (tab_host) cudaFreeHost(tab_host);
        if (stats_host) cudaFreeHost(stats_host);
        if (stage_free) cudaEventDestroy(stage_free);
        for (auto& e : ev) if (e) cudaEventDestroy(e);
    }
};

namespace {

int check_profiles(const disco_trace_desc_t* d, std::vector<GroupConst>* out) {
    if (!d->servers || !d->devices || d->n_servers == 0 || d->n_devices == 0 ||
        (uint64_t)d->n_servers * d->n_devices > kMaxGroups)
        return fail(DISCO_EINVAL, "profile tables: need at least one server and one device and at most 64 groups");
    out->clear();
    for (uint32_t s = 0; s < d->n_servers; ++s) {
        const disco_server_profile_t& sv = d->servers[s];
        if (!(sv.tbt_s > 0.0f) || !std::isfinite(sv.tbt_s) || !(sv.jitter >= 0.0f && sv.jitter <= 1.0f) ||
            !std::isfinite(sv.c_prefill) || !std::isfinite(sv.c_decode))
            return fail(DISCO_EINVAL, "server profile " + std::to_string(s) + " is invalid");
        for (uint32_t k = 0; k < d->n_devices; ++k) {
            const disco_device_profile_t& dv = d->devices[k];
            if (!(dv.prefill_tps > 0.0f) || !(dv.decode_tps > 0.0f) || !std::isfinite(dv.prefill_tps) ||
                !std::isfinite(dv.decode_tps) || !(dv.jitter >= 0.0f && dv.jitter <= 1.0f) ||
                !(dv.ttft_intercept_s >= 0.0f) || !std::isfinite(dv.ttft_intercept_s) ||
                !std::isfinite(dv.c_prefill) || !std::isfinite(dv.c_decode) || !std::isfinite(dv.lambda))
                return fail(DISCO_EINVAL, "device profile " + std::to_string(k) + " is invalid");
            const int64_t Ts = ticks_of_seconds(sv.tbt_s), Tdv = ticks_of_rate(dv.decode_tps);
            const int64_t Js = llrint((double)Ts * (double)sv.jitter), Jd = llrint((double)Tdv * (double)dv.jitter);
            const int64_t kappa = ticks_of_rate(dv.prefill_tps), c0 = ticks_of_seconds(dv.ttft_intercept_s);
            if (Ts + Js >= (1 << 30) || Tdv + Jd >= (1 << 30) || kappa * (kMaxPrompt + kMaxOutput) + c0 >= (1LL << 31))
                return fail(DISCO_EINVAL, "profile too slow: a token interval or device TTFT exceeds the 32-bit tick range");
            GroupConst g;
            std::memset(&g, 0, sizeof g);
            g.T_srv = (int32_t)Ts; g.J_srv = (int32_t)Js; g.T_dev = (int32_t)Tdv; g.J_dev = (int32_t)Jd;
            g.kappa = (int32_t)kappa; g.c0 = (int32_t)c0;
            const double cps = sv.c_prefill, cds = sv.c_decode, lam = dv.lambda;
            const double dcp = lam * (double)dv.c_prefill, dcd = lam * (double)dv.c_decode;
            g.auto_device_constrained = std::fmin(dcp, dcd) > std::fmax(cps, cds) ? 1 : 0;   // Algorithm 1
            g.candidate = cds > dcd ? 1 : (dcd > cds ? 2 : 0);
            g.delta_c = (float)std::fabs(cds - dcd);
            g.cps = (float)cps; g.cds = (float)cds; g.lcpd = (float)dcp; g.lcdd = (float)dcd;
            g.cps_d = cps; g.cds_d = cds; g.cpd_d = dv.c_prefill; g.cdd_d = dv.c_decode; g.lambda_d = lam;
            out->push_back(g);
        }
    }
    return 0;
}

// How a load's inputs reach the ingestion kernel.
enum Inputs { IN_DEVICE, IN_COPIED, IN_PLACE, IN_PACKED };

bool large_load(uint32_t n, int G, Inputs in) { return n >= (in == IN_PLACE ? kLargeMinInPlace : kLargeMinN) && n <= kLargeMaxN && G <= kLargeMaxGroups; }

cudaError_t reserve_trace(disco_ctx* c, uint32_t n, Inputs in, bool has_sp, bool has_dp) {
    const size_t N = n ? n : 1, N4 = N + 3;
    const int G = c->G;
    Layout lay;
    // one block for everything a load clears, first: the flags and sums, the two histograms, the windows of the sort
    const bool once = once_trace(n, G, (uint32_t)c->sms);
    const size_t tick_bytes = (size_t)G * kTickBins * 4, cnt_bytes = ((size_t)G * (kMaxPrompt + 1) * 4 + 15) / 16 * 16;
    c->zero_bytes = sizeof(LoadZero) + tick_bytes + cnt_bytes + (once ? (size_t)kOnceWindows * 16 : (size_t)sort_windows(n, G) * 8);
    const size_t o_zero[2] = {lay.take(c->zero_bytes), once ? lay.take(c->zero_bytes) : 0};
    const size_t o_req = lay.take(N * 16), o_sorted = lay.take(N * 4), o_binned = lay.take(N * 4), o_inv = lay.take(N * 4);
    const size_t o_ends = lay.take((size_t)G * (kMaxPrompt + 1) * 4), o_starts = lay.take(2 * tick_bytes);
    const size_t o_mass = lay.take((size_t)G * (kMaxPrompt + 2) * 8), o_off = lay.take((kMaxGroups + 1) * 4);
    const size_t o_knots = lay.take((size_t)G * kNKnots * 4), o_fin = lay.take((size_t)2 * kMaxGroups * 8);
    size_t o_in[5] = {0, 0, 0, 0, 0};
    if (in == IN_COPIED) {
        for (int k = 0; k < 3; ++k) o_in[k] = lay.take(N * 4);
        o_in[3] = lay.take(has_sp ? N : 0); o_in[4] = lay.take(has_dp ? N : 0);
    } else if (in == IN_PLACE) {
        o_in[0] = lay.take(N4 * 4); o_in[1] = lay.take(N4 * 4); o_in[2] = lay.take(N4);      // (whole vectors of four)
    } else if (in == IN_PACKED) {
        o_in[0] = lay.take(n > kPackInPlace ? packed_bytes(n) : 0);
    }
    const size_t without = lay.bytes;
    const bool large = large_load(n, G, in);
    LargeLoad& lg = c->large;
    std::memset(&lg, 0, sizeof lg);
    if (large) {
        lg.rec_share = rec_share(n); lg.tick_share = tick_share(n, (uint32_t)c->sms);
        lg.n_rec = 2 * (n / lg.rec_share + G); lg.n_tick = 2 * (n / lg.tick_share + G);
    }
    const size_t o_parted = lay.take(large ? N * 16 : 0), o_rec_of = lay.take(large ? (size_t)G * (kMaxPrompt + 1) * 2 : 0);
    const size_t o_tick_of = lay.take(large ? (size_t)G * kTickBins * 2 : 0), o_at = lay.take(large ? ((size_t)lg.n_rec + lg.n_tick + 4) * 4 : 0);
    const size_t o_members = lay.take(large ? (size_t)lg.n_rec * 8 + (size_t)lg.n_tick * 16 : 0);
    disco_ctx::Halves& hv = c->halves;
    // (a large load works without its buckets, by k_load, where there is no room for them: 16 bytes a request)
    c->large_now = large && lay.bytes < c->trace_too_much;
    cudaError_t e = c->trace_mem.reserve(c->large_now ? lay.bytes : without);
    if (e == cudaErrorMemoryAllocation && c->large_now) {
        cudaGetLastError();
        c->large_now = false;
        c->trace_too_much = lay.bytes;
        e = c->trace_mem.reserve(without);
    }
    if (e) { hv = disco_ctx::Halves(); return e; }                   // (a later buffer may lie where the one that was given back did)
    char* base = (char*)c->trace_mem.p;
    if (!once || hv.at != base || hv.cap != c->trace_mem.cap || hv.bytes != c->zero_bytes) {
        hv = disco_ctx::Halves();
        if (once) { hv.at = base; hv.cap = c->trace_mem.cap; hv.bytes = c->zero_bytes; }
    }
    if (once) hv.now ^= 1;
    lg.parted = (uint4*)(base + o_parted);
    lg.rec_bucket = (uint16_t*)(base + o_rec_of); lg.tick_bucket = (uint16_t*)(base + o_tick_of);
    lg.rec_at = (uint32_t*)(base + o_at); lg.tick_at = lg.rec_at + lg.n_rec;
    lg.rec_members = (uint2*)(base + o_members); lg.tick_jobs = (uint4*)(lg.rec_members + lg.n_rec);     // (an even number)
    c->req.p = base + o_req; c->sorted.p = base + o_sorted; c->binned.p = base + o_binned; c->inv.p = base + o_inv;
    c->zero.p = base + o_zero[hv.now]; c->len_end.p = base + o_ends; c->tick_start.p = base + o_starts; c->cum_mass.p = base + o_mass;
    c->grp_off.p = base + o_off; c->knots.p = base + o_knots; c->fin_totals.p = base + o_fin;
    c->in_prompt.p = c->st_ticks.p = c->packed.p = base + o_in[0];
    c->in_out.p = c->st_ln.p = base + o_in[1];
    c->in_ttft.p = c->st_g.p = base + o_in[2];
    c->in_sp.p = base + o_in[3]; c->in_dp.p = base + o_in[4];
    c->z = (LoadZero*)c->zero.p;
    c->tick_cnt = (uint32_t*)(c->z + 1);
    c->cnt = (uint32_t*)((char*)c->tick_cnt + tick_bytes);
    c->windows = (uint2*)((char*)c->cnt + cnt_bytes);
    c->err = c->z->err;
    return c->d_gc.reserve((size_t)kMaxGroups * sizeof(GroupConst));
}

// The pinned copy of the group tables; fetch_knots brings the knots alone (copies queued on the stream).
constexpr size_t kLengths = kMaxPrompt + 1;
int32_t* host_knots(disco_ctx* c, int g) { return (int32_t*)c->tab_host + c->G * kLengths + (size_t)g * kNKnots; }
int reserve_tab_host(disco_ctx* c) {
    if (c->tab_host_groups >= c->G) return 0;
    if (c->tab_host) cudaFreeHost(c->tab_host);
    c->tab_host = nullptr; c->tab_host_groups = 0;
    CU(cudaMallocHost((void**)&c->tab_host, (size_t)c->G * (kLengths + kNKnots) * 4));
    c->tab_host_groups = c->G;
    return 0;
}
int fetch_knots(disco_ctx* c, cudaStream_t st) {
    if (int rc = reserve_tab_host(c)) return rc;
    CU(cudaMemcpyAsync(host_knots(c, 0), c->knots.p, (size_t)c->G * kNKnots * 4, cudaMemcpyDeviceToHost, st));
    return 0;
}

// Pinned staging of at least that many bytes, once the copies or the kernel of an earlier call no longer read it.
int reserve_stage(disco_ctx* c, size_t bytes, cudaStream_t st) {
    if (c->stage_free) CU(cudaEventSynchronize(c->stage_free));
    else CU(cudaEventCreateWithFlags(&c->stage_free, cudaEventDisableTiming));
    // Two evaluations in a row: the first one's kernel puts its number into stage_read.  (An event behind that kernel would hold the
    // next one up.)  The stream is asked as well, since what the earlier evaluation launched lies in front of this one: nothing
    // else on the device is waited for.
    while (*c->stage_read != c->stage_turn) {
        const cudaError_t e = cudaStreamQuery(st);
        if (e == cudaErrorNotReady) { cudaGetLastError(); continue; }
        CU(e);
        if (*c->stage_read == c->stage_turn) break;
        CU(cudaDeviceSynchronize());                                 // (it lay on another stream, against the rules)
        *c->stage_read = c->stage_turn;
    }
    if (bytes > c->stage_cap) {
        if (c->stage) cudaFreeHost(c->stage);
        c->stage = nullptr; c->stage_cap = 0;
        CU(cudaMallocHost(&c->stage, bytes));
        c->stage_cap = bytes;
    }
    return 0;
}

// The fallback sort: ticks stored group after group (off: [G + 1], device memory) ascending within each group into out.
int radix_sort(disco_ctx* c, const int32_t* ticks, const uint32_t* off, uint32_t total, int32_t* out, cudaStream_t st) {
    cudaError_t e;
    if ((e = c->keys_a.reserve((size_t)total * 8)) != cudaSuccess || (e = c->keys_b.reserve((size_t)total * 8)) != cudaSuccess ||
        (e = c->radix_counts.reserve(((size_t)256 * kRadixMaxBlocks + 256) * 4)) != cudaSuccess)
        return fail_cuda(e, "device allocation for the radix sort");
    if ((e = radix_sort_ticks(ticks, off, c->G, total, c->keys_a.as<uint64_t>(), c->keys_b.as<uint64_t>(),
                              c->radix_counts.as<uint32_t>(), out, c->sms, st)) != cudaSuccess) return fail_cuda(e, "radix sort");
    g_launches += radix_sort_launches(c->G);
    return 0;
}

}  // namespace

namespace disco {
int check_debug_record() { return debug_check(); }
}  // namespace disco

extern "C" {

const char* disco_last_error(void) { return g_err.c_str(); }

void disco_free_trace(disco_ctx_t* ctx) { delete ctx; }

int disco_load_trace(disco_ctx_t** pctx, const disco_trace_desc_t* d, void* stream) try {
    if (!pctx || !d) return fail(DISCO_EINVAL, "null argument");
    if (d->n >= (1ull << 31)) return fail(DISCO_EINVAL, "too many requests");
    if (d->n && (!d->prompt_len || !d->output_len || !d->server_ttft_s)) return fail(DISCO_EINVAL, "null trace array");
    if (d->arrays_on_device > 2) return fail(DISCO_EINVAL, "arrays_on_device must be 0, 1 or 2");
    if (d->first_index + d->n > (1ull << 32)) return fail(DISCO_EINVAL, "first_index + n exceeds 2^32");
    std::vector<GroupConst> gc;
    if (int rc = check_profiles(d, &gc)) return rc;
    cudaStream_t st = (cudaStream_t)stream;

    disco_ctx* c = *pctx;
    const bool fresh = c == nullptr;
    if (fresh) {
        c = new (std::nothrow) disco_ctx;
        if (!c) return fail(DISCO_ENOMEM, "out of host memory");
    }
    std::unique_ptr<disco_ctx> own(fresh ? c : nullptr);              // (until the load has succeeded)
    auto bail = [&](int rc) { c->loaded = false; return rc; };
    c->loaded = c->evaluated = c->reduced = false;
    c->n = (uint32_t)d->n; c->ns = d->n_servers; c->nd = d->n_devices; c->G = (int)gc.size(); c->gc = gc;
    c->first_index = d->first_index;
    c->tables_imported = c->tab_host_now = false;
    c->fin_imported = false;
    if (!c->sms) {
        int dev = 0;
        cudaError_t e0 = cudaGetDevice(&dev);
        if (e0 == cudaSuccess) e0 = cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev);
        if (e0 != cudaSuccess || c->sms < 1) return bail(fail_cuda(e0, "multiprocessor count of the current device"));
    }
    const uint32_t n = c->n;
    cudaError_t e;
    // Host arrays that are page-locked and mapped (cudaHostAlloc, cudaHostRegister, a pinned tensor) are read by
    // the ingestion kernel in place (it reads every element exactly once): no staging copies.  Pageable arrays are
    // packed and copied by several threads, which must not meet device memory.
    const void* in_place[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    Inputs in = d->arrays_on_device == 1 ? IN_DEVICE : (d->arrays_on_device == 2 || n == 0) ? IN_COPIED : IN_PLACE;
    if (in == IN_PLACE) {
        const void* host[5] = {d->prompt_len, d->output_len, d->server_ttft_s, d->server_profile, d->device_profile};
        for (int k = 0; k < 5; ++k) {
            if (!host[k]) continue;
            cudaPointerAttributes attr;
            if (cudaPointerGetAttributes(&attr, host[k]) != cudaSuccess) { cudaGetLastError(); in = IN_PACKED; continue; }
            if (attr.type == cudaMemoryTypeDevice)
                return bail(fail(DISCO_EINVAL, "a trace array is device memory, but arrays_on_device says host memory"));
            if (attr.type != cudaMemoryTypeHost || !attr.devicePointer) in = IN_PACKED;
            else in_place[k] = attr.devicePointer;
        }
    }
    if (!c->rb && (e = cudaMallocHost((void**)&c->rb, sizeof(HostReadback) + 256)) != cudaSuccess)    // (the selection's pair behind it)
        return bail(fail_cuda(e, "cudaMallocHost"));
    c->sel_host = (int32_t*)((char*)c->rb + (sizeof(HostReadback) + 15) / 16 * 16);
    if (!c->stage_read) {
        c->stage_read = (uint32_t*)(c->sel_host + 4);
        *c->stage_read = c->stage_turn;
    }
    if ((e = reserve_trace(c, n, in, d->server_profile != nullptr, d->device_profile != nullptr)) != cudaSuccess)
        return bail(fail_cuda(e, "device allocation for the trace"));

    LoadArgs a;
    std::memset(&a, 0, sizeof a);
    a.n = n; a.G = c->G; a.ns = c->ns; a.nd = c->nd;
    if (in == IN_COPIED && n) {
#define H2D(dst, src, bytes) if ((e = cudaMemcpyAsync(c->dst.p, src, bytes, cudaMemcpyHostToDevice, st)) != cudaSuccess) return bail(fail_cuda(e, "host to device copy"))
        H2D(in_prompt, d->prompt_len, (size_t)n * 4); H2D(in_out, d->output_len, (size_t)n * 4);
        H2D(in_ttft, d->server_ttft_s, (size_t)n * 4);
        if (d->server_profile) H2D(in_sp, d->server_profile, (size_t)n);
        if (d->device_profile) H2D(in_dp, d->device_profile, (size_t)n);
#undef H2D
        a.prompt = c->in_prompt.as<int32_t>(); a.outlen = c->in_out.as<int32_t>(); a.ttft = c->in_ttft.as<float>();
        a.sp = d->server_profile ? c->in_sp.as<uint8_t>() : nullptr;
        a.dp = d->device_profile ? c->in_dp.as<uint8_t>() : nullptr;
    } else if (in == IN_PACKED) {
        if (!c->packer) c->packer.reset(new (std::nothrow) Packer);
        if (!c->packer) return bail(fail(DISCO_ENOMEM, "out of host memory"));
        // The CPU reads the columns now, and work on the stream may still write them: page-locked or managed ones by copies and
        // kernels, any by host functions.  (Asked first: to wait for an idle stream takes 3 us.)
        if ((e = cudaStreamQuery(st)) == cudaErrorNotReady) { cudaGetLastError(); e = cudaStreamSynchronize(st); }
        if (e != cudaSuccess) return bail(fail_cuda(e, "work in front of the load"));
        if ((e = c->packer->pack(*d, c->packed.as<char>(), st, &a.packed)) != cudaSuccess) return bail(fail_cuda(e, "packing the trace"));
    } else if (in == IN_PLACE) {
        a.prompt = (const int32_t*)in_place[0]; a.outlen = (const int32_t*)in_place[1]; a.ttft = (const float*)in_place[2];
        a.sp = (const uint8_t*)in_place[3]; a.dp = (const uint8_t*)in_place[4];
        a.st_ticks = c->st_ticks.as<uint32_t>(); a.st_ln = c->st_ln.as<uint32_t>(); a.st_g = c->st_g.as<uint8_t>();
    } else {
        a.prompt = d->prompt_len; a.outlen = d->output_len; a.ttft = d->server_ttft_s;
        a.sp = d->server_profile; a.dp = d->device_profile;
    }
    a.z = c->z; a.zero_bytes = c->zero_bytes; a.cnt = c->cnt; a.tick_cnt = c->tick_cnt;
    a.tick_start = c->tick_start.as<uint32_t>(); a.tick_at = a.tick_start + (size_t)c->G * kTickBins;
    a.binned = c->binned.as<uint32_t>();
    a.req = c->req.as<uint4>(); a.inv = c->inv.as<uint32_t>(); a.sorted = c->sorted.as<int32_t>();
    a.len_end = c->len_end.as<uint32_t>(); a.cum_mass = c->cum_mass.as<int64_t>(); a.grp_off = c->grp_off.as<uint32_t>();
    a.knots = c->knots.as<int32_t>(); a.fin_totals = c->fin_totals.as<uint64_t>();
    a.windows = c->windows;
    a.rounds = (n + 3000000u - 1) / 3000000u;                       // (3 million records and ticks take 60 MB)
    a.readback = c->rb;                                             // pinned host memory, written by the kernel
    // the profile table is read from pageable memory: this copy returns once it has been staged (a reload with the same
    // profiles skips it)
    const bool same_profiles = c->gc_dev_at == c->d_gc.p && c->gc_dev.size() == c->gc.size() &&
                               std::memcmp(c->gc_dev.data(), c->gc.data(), c->gc.size() * sizeof(GroupConst)) == 0;
    if (!same_profiles) {
        c->gc_dev_at = nullptr;
        if ((e = cudaMemcpyAsync(c->d_gc.p, c->gc.data(), c->gc.size() * sizeof(GroupConst), cudaMemcpyHostToDevice, st)) != cudaSuccess)
            return bail(fail_cuda(e, "profile copy"));
    }
    static const int32_t no_report[4] = {0, 0, 0, 2};               // what the host finds if the blocks lose each other
    std::memcpy(c->rb->err, no_report, sizeof no_report);
    const bool large = c->large_now;
    a.large = c->large;
    c->inv_there = !large;
    disco_ctx::Halves& hv = c->halves;
    const bool once = hv.at != nullptr;
    if (once) {
        a.once.windows = (unsigned long long*)c->windows;
        a.once.zeroed = hv.zero[hv.now];
        a.once.clear = (uint4*)((char*)c->zero.p + (hv.now ? -1 : 1) * (ptrdiff_t)((c->zero_bytes + 255) / 256 * 256));
        a.once.clear_vecs = (uint32_t)(c->zero_bytes / 16);
        hv.zero[0] = hv.zero[1] = false;                             // (until the load has succeeded)
    }
    if ((e = once ? run_load_once(a, c->sms, st) : large ? run_load_large(a, c->sms, st) : run_load(a, c->sms, st)) != cudaSuccess) return bail(fail_cuda(e, "trace ingestion kernels"));
    g_launches += large ? 6 : 1;
    // the few numbers the host needs (error word, group sizes, longest output, largest TTFT per group) are in rb
    HostReadback* rb = c->rb;
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return bail(fail_cuda(e, "trace ingestion"));
    if (int rc = debug_check()) return bail(rc);
    if (!same_profiles) { c->gc_dev = c->gc; c->gc_dev_at = c->d_gc.p; }      // the copy has landed
    if (rb->err[0]) {
        static const char* what[] = {"", "prompt length outside 1..4096", "output length outside 1..8192",
                                     "server TTFT not finite, not positive or above 2000 s", "profile id out of range"};
        return bail(fail(DISCO_EINVAL, std::string(what[rb->err[0]]) + " at request " + std::to_string(rb->err[1])));
    }
    if (rb->err[3] == 2) return bail(fail(DISCO_ECUDA, "internal error: the blocks of the ingestion kernel lost each other"));
    if (rb->err[3] == 1) {
        // a sample that the bin-wise sort gives up on: radix sort, then the knots of the sorted sample
        if (int rc = radix_sort(c, c->binned.as<int32_t>(), c->grp_off.as<uint32_t>(), n, c->sorted.as<int32_t>(), st)) return bail(rc);
        if ((e = launch_tables_imported(c->G, c->cnt, c->cum_mass.as<int64_t>(), c->sorted.as<int32_t>(), c->grp_off.as<uint32_t>(),
                                        c->knots.as<int32_t>(), st)) != cudaSuccess) return bail(fail_cuda(e, "group tables"));
        g_launches += 1;
        if (int rc = fetch_knots(c, st)) return bail(rc);
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return bail(fail_cuda(e, "trace ingestion"));
        if (int rc = debug_check()) return bail(rc);
        for (int g = 0; g < c->G; ++g) rb->knot_max[g] = host_knots(c, g)[kNKnots - 1];      // (the last knot is the largest tick)
    }
    c->F_sorted = c->sorted.as<int32_t>(); c->F_off = c->grp_off.as<uint32_t>();
    c->F_n.assign(rb->ng, rb->ng + c->G);
    if (once) hv.zero[hv.now ^ 1] = true;
    c->loaded = true;
    own.release();
    *pctx = c;
    return 0;
} DISCO_CATCH

int disco_eval_policies(disco_ctx_t* c, const disco_policy_t* pol, uint32_t P, uint64_t seed,
                        const disco_pair_out_t* out, void* stream) try {
    if (!c || !pol || P == 0) return fail(DISCO_EINVAL, "null context, null policies or P = 0");
    if (!c->loaded) return fail(DISCO_EINVAL, "no trace loaded");
    if (P > (1u << 19)) return fail(DISCO_EINVAL, "too many policies");
    cudaStream_t st = (cudaStream_t)stream;
    const int G = c->G;
    const uint32_t n = c->n;
    c->evaluated = c->reduced = false;

    // ---- policy constants and timeline classes
    std::vector<PolicyConst> pc(P);
    std::vector<ClassConst> classes;
    bool any_beta = false;                // some policy uses the Eq. 1-2 wait rule
    bool extras = false;                  // some policy routes at random or triggers on an expected length
    bool any_waits = false;               // Algorithm 2 decides for some policy in some group
    const bool any_constrained = std::any_of(c->gc.begin(), c->gc.end(), [](const GroupConst& g) { return g.auto_device_constrained != 0; });
    int64_t tau = 0, t_m = 0;
    for (uint32_t p = 0; p < P; ++p) {
        const disco_policy_t& q = pol[p];
        auto at = [p] { return " (policy " + std::to_string(p) + ")"; };
        if (!(q.budget >= 0.0f && q.budget <= 1.0f)) return fail(DISCO_EINVAL, "budget outside [0,1]" + at());
        if (!(q.alpha > 0.0f && q.alpha < 1.0f)) return fail(DISCO_EINVAL, "alpha outside (0,1)" + at());
        if (!(q.mig_threshold >= 0.0f)) return fail(DISCO_EINVAL, "migration threshold negative or NaN" + at());
        if (!(q.r_c > 0.0f) || !std::isfinite(q.r_c)) return fail(DISCO_EINVAL, "consumption rate must be positive" + at());
        if (!(q.t_m_s >= 0.0f) || !std::isfinite(q.t_m_s)) return fail(DISCO_EINVAL, "migration time must be >= 0" + at());
        const uint32_t mode = (q.flags >> 2) & 3u;
        if (mode == 3 || (q.flags >> 6)) return fail(DISCO_EINVAL, "unknown flags" + at());
        if (q.expected_len > (1u << 20)) return fail(DISCO_EINVAL, "expected length too large" + at());
        if (q.l_immediate > (uint32_t)kMaxPrompt) return fail(DISCO_EINVAL, "l_immediate above the longest prompt" + at());
        if (p == 0 || q.r_c != pol[p - 1].r_c || q.t_m_s != pol[p - 1].t_m_s) { tau = ticks_of_rate(q.r_c); t_m = ticks_of_seconds(q.t_m_s); }
        if (tau < 1 || tau >= (1 << 30)) return fail(DISCO_EINVAL, "consumption interval outside 1 .. 2^30 ticks" + at());
        const bool pacing = (q.flags & DISCO_FLAG_PACING) != 0, mig = (q.flags & DISCO_FLAG_MIGRATION) != 0;
        int64_t B = pacing ? (t_m + tau - 1) / tau : 0;               // Eq. 6, rounded up
        if (B > kMaxOutput) B = kMaxOutput;                            // a buffer no stream can fill
        PolicyConst& o = pc[p];
        o.budget = q.budget; o.alpha = q.alpha; o.theta = q.mig_threshold; o.flags = q.flags;
        o.tau = (int32_t)tau; o.B = (int32_t)B; o.mode = (int32_t)mode;
        o.expected_len = q.expected_len; o.l_immediate = q.l_immediate;
        if (q.flags & DISCO_FLAG_BETA_RULE) any_beta = true;
        any_waits = any_waits || mode == 1 || (mode == 0 && any_constrained);
        o.route_all = q.budget >= 1.0f ? 1 : 0;
        o.route_thr = o.route_all ? 0xFFFFFFFFu : (uint32_t)std::floor((double)q.budget * 4294967296.0);
        if ((q.flags & (DISCO_FLAG_STOCHASTIC | DISCO_FLAG_BETA_RULE)) || q.expected_len) extras = true;
        int cls = -1;
        for (size_t k = 0; k < classes.size(); ++k)
            if (classes[k].tau == o.tau && classes[k].B == o.B && classes[k].pacing == (int)pacing) { cls = (int)k; break; }
        if (cls < 0) {
            ClassConst cc;
            std::memset(&cc, 0, sizeof cc);
            cc.tau = o.tau; cc.tau_eff = pacing ? o.tau : 0; cc.B = o.B; cc.pacing = pacing;
            classes.push_back(cc);
            cls = (int)classes.size() - 1;
        }
        classes[cls].mig_any |= mig ? 1 : 0;
        o.cls = cls;
    }
    // ---- per class: 32-bit range proof, how each group's streams behave, histogram windows of the regular TBTs
    const HostReadback& rb = *c->rb;
    const int64_t n_max = rb.max_n;
    struct ClassPlan { uint32_t kinds = 0, batches[3] = {0, 0, 0}, search = 0; };
    std::vector<ClassPlan> plan(classes.size());
    size_t wmax[3] = {1, 1, 1};
    bool stored = false;                  // some class stores sums, maxima and windows
    for (size_t k = 0; k < classes.size(); ++k) {
        ClassConst& cc = classes[k];
        ClassPlan& pl = plan[k];
        int Wmax[3] = {1, 1, 1};
        for (int g = 0; g < G; ++g) {
            const GroupConst& gc = c->gc[g];
            const int64_t xs = gc.T_srv + (int64_t)gc.J_srv, xd = gc.T_dev + (int64_t)gc.J_dev;
            if (rb.ng[g]) {
                const int64_t step = std::max<int64_t>(cc.tau_eff, std::max(xs, xd));
                const int64_t Mmax = std::max<int64_t>(rb.knot_max[g], (int64_t)gc.kappa * (kMaxPrompt + n_max) + gc.c0);
                if ((n_max - 1) * step + Mmax >= (1LL << 31))
                    return fail(DISCO_EINVAL, "a decode stream could outlast 2^31 ticks (about 35 minutes)");
            }
            // which streams keep the pace at every token, and which wait for every token
            const int cand = cc.mig_any ? gc.candidate : 0;
            const bool even_s = cc.pacing && xs <= cc.tau, even_d = cc.pacing && xd <= cc.tau;
            const bool free_s = gc.T_srv - (int64_t)gc.J_srv >= cc.tau, free_d = gc.T_dev - (int64_t)gc.J_dev >= cc.tau;
            cc.even[g] = (uint8_t)((even_s ? 1 : 0) | (even_d ? 2 : 0));
            if (even_s && even_d) { cc.kind[g] = G_EXACT; cc.even[g] = 7; }
            else if (!cc.pacing) cc.kind[g] = G_FREE;
            else if ((even_s || free_s) && (even_d || free_d) &&
                     (cand == 0 || (cc.B > 0 && !(cand == 1 ? even_s : even_d)))) cc.kind[g] = G_FREE;   // (its buffer never fills)
            else cc.kind[g] = G_GENERAL;
            if (cc.kind[g] == G_EXACT) {
                const int64_t gain = cc.tau - (gc.candidate == 2 ? xd : xs), fill = (int64_t)std::max(cc.B - 1, 0) * cc.tau;
                int64_t need = gain > 0 ? fill / gain + 1 : (int64_t)kMaxOutput;
                if (cc.B == 0 || cand == 0) need = 1;                         // nothing to search for
                cc.search[g] = (uint32_t)std::min<int64_t>(need, kMaxOutput);
            }
            if (rb.ng[g]) {
                pl.kinds |= 1u << cc.kind[g];
                pl.batches[cc.kind[g]] += (rb.ng[g] + 31) / 32;
                if (cc.kind[g] == G_EXACT) pl.search = std::max(pl.search, cc.search[g]);
            }
            // shortest and longest regular interval of the streams: as generated where a stream waits for every token, else from
            // tau on
            const bool as_is[2] = {!cc.pacing || (cc.kind[g] == G_FREE && !even_s), !cc.pacing || (cc.kind[g] == G_FREE && !even_d)};
            int64_t lo_v[3], hi_v[3];
            lo_v[0] = as_is[0] ? gc.T_srv - (int64_t)gc.J_srv : cc.tau; hi_v[0] = as_is[0] ? xs : std::max<int64_t>(cc.tau, xs);
            lo_v[1] = as_is[1] ? gc.T_dev - (int64_t)gc.J_dev : cc.tau; hi_v[1] = as_is[1] ? xd : std::max<int64_t>(cc.tau, xd);
            lo_v[2] = std::min(lo_v[0], lo_v[1]); hi_v[2] = cc.kind[g] == G_GENERAL ? std::max(hi_v[0], hi_v[1]) : lo_v[2];
            for (int s = 0; s < 3; ++s) {
                const int lo = host_bin_of_ticks(lo_v[s]), hi = host_bin_of_ticks(hi_v[s]);
                cc.lo[g][s] = lo;
                cc.ktau[g][s] = cc.pacing && !(s < 2 && as_is[s]) ? host_bin_of_ticks(cc.tau) - lo : -1;
                Wmax[s] = std::max(Wmax[s], hi - lo + 1);
            }
        }
        for (int s = 0; s < 3; ++s) cc.W[s] = Wmax[s];
        if (!(pl.kinds & ~(1u << G_EXACT))) continue;                        // nothing but the hand-offs is stored
        stored = true;
        for (int s = 0; s < ((pl.kinds & (1u << G_GENERAL)) ? 3 : 2); ++s) wmax[s] = std::max<size_t>(wmax[s], Wmax[s]);   // (no other kind stores the third)
        if ((size_t)n * (Wmax[0] + Wmax[1] + Wmax[2]) * 2 > (48ull << 30))
            return fail(DISCO_ENOMEM, "per-request TBT windows would exceed 48 GB");
    }

    // ---- several classes are played out one after another and then reduced together (a wave of them), each into records of
    //      its own as long as those take no more than 512 MB
    const size_t N1 = n ? n : 1, n_classes = classes.size();
    Layout slot;
    const size_t o_ticket = slot.take(4), o_hand = slot.take(N1 * 8);
    size_t o_rec[6] = {}, o_win[3] = {};
    if (stored) {
        for (int k = 0; k < 6; ++k) o_rec[k] = slot.take(N1 * 4);
        for (int k = 0; k < 3; ++k) o_win[k] = slot.take(N1 * wmax[k] * 2);
    }
    const size_t rec_stride = (slot.bytes + 255) / 256 * 256;
    size_t wave = std::min(n_classes, std::max<size_t>(1, ((size_t)512 << 20) / rec_stride));
    cudaError_t e;
    while (wave > 1 && wave * rec_stride >= c->rec_too_much) wave = (wave + 1) / 2;
    while ((e = c->rec_mem.reserve(wave * rec_stride)) == cudaErrorMemoryAllocation && wave > 1) {      // (smaller waves, then)
        cudaGetLastError();
        c->rec_too_much = wave * rec_stride;
        wave = (wave + 1) / 2;
    }
    if (e != cudaSuccess) return fail_cuda(e, "device allocation for the evaluation");
    auto slot_of = [&](size_t k) { return k % wave; };
    // A class whose free streams are those of an earlier class of its wave -- as generated, next to streams that keep the pace --
    // has them played and stored by that class.
    std::vector<uint32_t> kinds_of(n_classes);
    std::vector<size_t> win_class(n_classes);
    std::vector<FreeMore> more(n_classes);
    for (size_t k = 0; k < n_classes; ++k) {
        kinds_of[k] = plan[k].kinds;
        win_class[k] = k;
        more[k].n = 0;
        const ClassConst& a = classes[k];
        if (!a.pacing || (plan[k].kinds & (1u << G_GENERAL)) || !(plan[k].kinds & (1u << G_FREE))) continue;
        for (size_t j = k - slot_of(k); j < k; ++j) {
            const ClassConst& b = classes[j];
            bool same = b.pacing && win_class[j] == j && more[j].n < kFreeMore && a.W[0] == b.W[0] && a.W[1] == b.W[1];
            for (int g = 0; g < G && same; ++g) {
                if (!rb.ng[g] || (a.kind[g] != G_FREE && b.kind[g] != G_FREE)) continue;
                same = a.kind[g] == b.kind[g] && a.even[g] == b.even[g];
                for (int s = 0; s < 2; ++s) same = same && (((a.even[g] >> s) & 1) || a.lo[g][s] == b.lo[g][s]);
            }
            if (!same) continue;
            win_class[k] = j;
            plan[k].kinds &= ~(1u << G_FREE);
            more[j].tau[more[j].n] = a.tau;
            more[j].off[more[j].n++] = (ptrdiff_t)((slot_of(k) - slot_of(j)) * rec_stride);
            break;
        }
    }
    // ---- the first class's play-out needs no more than this: it runs while the host lays out the policies
    {
        char* mem = (char*)c->rec_mem.p;
        c->play_ticket.p = mem + o_ticket; c->rec_hand.p = mem + o_hand;
        for (int k = 0; k < 6; ++k) c->rec_u32[k].p = mem + o_rec[k];
        for (int k = 0; k < 3; ++k) c->rec_win[k].p = mem + o_win[k];
    }
    TraceDev tr;
    tr.n = n; tr.n_groups = G; tr.req = c->req.as<uint4>(); tr.inv = c->inv.as<uint32_t>();
    tr.len_end = c->len_end.as<uint32_t>(); tr.grp_off = c->grp_off.as<uint32_t>();
    TimelineRec rec;
    rec.hand = c->rec_hand.as<uint2>();
    for (int k = 0; k < 3; ++k) {
        rec.sum[k] = c->rec_u32[2 * k].as<uint32_t>(); rec.max[k] = c->rec_u32[2 * k + 1].as<uint32_t>();
        rec.win[k] = c->rec_win[k].as<uint16_t>();
    }
    auto rec_of = [&](size_t k) {                  // a class's records
        TimelineRec r = rec;
        const size_t at = slot_of(k) * rec_stride, win_at = slot_of(win_class[k]) * rec_stride;
        r.hand = (uint2*)((char*)r.hand + at);
        for (int s = 0; s < 3; ++s) {
            r.sum[s] = (uint32_t*)((char*)r.sum[s] + at); r.max[s] = (uint32_t*)((char*)r.max[s] + at);
            r.win[s] = (uint16_t*)((char*)r.win[s] + win_at);
        }
        return r;
    };
    const GroupConst* gc = c->d_gc.as<GroupConst>();
    uint64_t out_tokens = 0;
    for (int g = 0; g < G; ++g) out_tokens += rb.grp_sum_n[g];
    const bool long_outputs = out_tokens >= 512ull * n;
    // the hash is keyed by the request's index in the whole trace: key = mix(k0 + (first_index + i) * C_REQ)
    const uint32_t k0 = seed_key(seed) + (uint32_t)c->first_index * kHashReq;
    c->timing_valid = false;
    const bool timed = c->timing && classes.size() == 1;
    auto play_out = [&](size_t k, bool beside) {
        g_launches += timeline_launches(plan[k].kinds);
        return launch_timeline(tr, gc, classes[k], c->knots.as<int32_t>(), k0, rec_of(k), c->err, c->play_ticket.as<uint32_t>(),
                               plan[k].kinds, plan[k].batches, plan[k].search, long_outputs, timed ? c->ev[1] : nullptr, more[k], &c->z->free_ticket, rb.ng, beside, k == 0 && !timed, c->sms, st);
    };
    if (n != 0 && !timed) CU(play_out(0, false));

    // ---- the policies of a class: plain ones form grids of budgets by overheads (grid.cu), at most kGridCols by kGridRows
    //      to a slab; random routing and the Eq. 1-2 rule go pair by pair
    std::vector<uint32_t> tab;                     // lists of policy indices, one after the other
    tab.reserve((size_t)4 * P + 64);
    std::vector<Slab> slabs;
    struct ClassLists { size_t all, n_all, ext, n_ext; };
    std::vector<ClassLists> lists(classes.size());
    bool any_mixed = false, any_pairs = false;
    constexpr uint32_t kNone = 0xFFFFFFFFu;
    auto theta_of = [&](uint32_t p) { return (pc[p].flags & DISCO_FLAG_MIGRATION) ? pc[p].theta : 0.0f; };   // (else it does not matter)
    // The place of x in an ascending list of distinct values, entered if it is new; `at`: where the last one was.  Grids are
    // given budget by budget or overhead by overhead: the next value mostly follows the last one.
    auto place_of = [](std::vector<float>& v, float x, size_t& at) {
        for (size_t k = at; k < v.size() && k < at + 2; ++k) if (v[k] == x) { at = k; return; }
        const auto it = std::lower_bound(v.begin(), v.end(), x);
        at = it - v.begin();
        if (it == v.end() || *it != x) v.insert(it, x);
    };
    struct Grid { uint32_t flags, expected_len; float alpha; std::vector<uint32_t> pols; std::vector<float> budgets, thetas; size_t b_at, t_at; };
    std::vector<Grid> grids;
    std::vector<uint32_t> cells, used, wide, cell_of;
    const size_t beta_at = tab.size();             // (group, policy) pairs whose slope of Eq. 1-2 is searched for
    for (int g = 0; any_beta && g < G; ++g)
        for (uint32_t p = 0; p < P; ++p)
            if ((pc[p].flags & DISCO_FLAG_BETA_RULE) && (pc[p].mode == 1 || (pc[p].mode == 0 && c->gc[g].auto_device_constrained)))
                tab.push_back((uint32_t)g * P + p);
    const uint32_t n_beta = (uint32_t)(tab.size() - beta_at);
    // (in a wave, the classes without windows first: their slabs go through the grid kernel together)
    auto wide_class = [&](size_t k) { return (kinds_of[k] & ~(1u << G_EXACT)) != 0; };
    std::vector<size_t> order(n_classes);
    std::iota(order.begin(), order.end(), (size_t)0);
    std::stable_sort(order.begin(), order.end(), [&](size_t x, size_t y) { return x / wave != y / wave ? x / wave < y / wave : wide_class(x) < wide_class(y); });
    for (size_t k : order) {
        ClassLists& L = lists[k];
        L.all = tab.size();
        if (classes.size() == 1) {
            tab.resize(L.all + P);
            std::iota(tab.begin() + L.all, tab.end(), 0u);
        } else {
            for (uint32_t p = 0; p < P; ++p) if (pc[p].cls == (int)k) tab.push_back(p);
        }
        L.n_all = tab.size() - L.all;
        L.ext = tab.size();
        grids.clear();
        Grid* last = nullptr;
        for (size_t i = L.all; i < L.all + L.n_all; ++i) {
            const uint32_t p = tab[i];
            const PolicyConst& q = pc[p];
            if (q.flags & (DISCO_FLAG_STOCHASTIC | DISCO_FLAG_BETA_RULE)) { tab.push_back(p); continue; }
            auto same = [&](const Grid& gr) { return gr.flags == q.flags && gr.expected_len == q.expected_len && gr.alpha == q.alpha; };
            Grid* at = last && same(*last) ? last : nullptr;           // (mostly the one of the policy before)
            for (size_t x = grids.size(); x-- > 0 && !at;) if (same(grids[x])) at = &grids[x];
            if (!at) {
                grids.push_back(Grid{q.flags, q.expected_len, q.alpha, {}, {}, {}, 0, 0});
                at = &grids.back();
                at->pols.reserve(L.n_all);
            }
            last = at;
            at->pols.push_back(p);
            place_of(at->budgets, q.budget, at->b_at);
            place_of(at->thetas, theta_of(p), at->t_at);
        }
        L.n_ext = tab.size() - L.ext;
        any_pairs = any_pairs || L.n_ext != 0;
        for (Grid& gr : grids) {
            const size_t n_b = gr.budgets.size(), n_t = gr.thetas.size(), n_p = gr.pols.size();
            auto open = [&](int T, bool mixed) {
                Slab sl;
                std::memset(&sl, 0, sizeof sl);
                sl.cls = (uint32_t)k; sl.slot = (uint32_t)slot_of(k); sl.win_slot = (uint32_t)slot_of(win_class[k]);
                sl.bin_tau = host_bin_of_ticks(classes[k].tau);
                sl.T = T; sl.expected_len = gr.expected_len; sl.mixed = mixed ? 1 : 0;
                sl.mig = (gr.flags & DISCO_FLAG_MIGRATION) ? 1 : 0;
                return sl;
            };
            // closes a slab of the columns [c0, c1) of `cells` (T policies each, kNone for none)
            auto close = [&](Slab sl, size_t c0, size_t c1) {
                const size_t T = (size_t)sl.T;
                sl.K = (int32_t)(c1 - c0);
                sl.cols = (uint32_t)tab.size();
                for (size_t x = c0; x < c1; ++x) {
                    size_t r = 0;
                    while (cells[x * T + r] == kNone) ++r;             // (a column has a policy)
                    tab.push_back(cells[x * T + r]);
                }
                sl.cells = (uint32_t)tab.size();
                tab.insert(tab.end(), cells.begin() + c0 * T, cells.begin() + c1 * T);
                sl.policies = (uint32_t)((c1 - c0) * T - std::count(cells.begin() + c0 * T, cells.begin() + c1 * T, kNone));
                slabs.push_back(sl);
            };
            if (n_t > 1 && 2 * n_p <= n_b * n_t) {
                // Most (budget, overhead) combinations are no policy: a column per policy instead, and what the overheads
                // of a slab's policies do not agree on goes pair by pair.
                cells = gr.pols;
                std::sort(cells.begin(), cells.end(), [&](uint32_t x, uint32_t y) { return pc[x].budget != pc[y].budget ? pc[x].budget < pc[y].budget : x < y; });
                for (size_t x0 = 0; x0 < n_p; x0 += kGridCols) {
                    const size_t x1 = std::min(n_p, x0 + (size_t)kGridCols);
                    Slab sl = open(1, true);
                    sl.theta[0] = sl.theta[1] = theta_of(cells[x0]);
                    for (size_t x = x0; x < x1; ++x) {
                        sl.theta[0] = std::min(sl.theta[0], theta_of(cells[x])); sl.theta[1] = std::max(sl.theta[1], theta_of(cells[x]));
                    }
                    close(sl, x0, x1);
                    any_mixed = any_pairs = true;
                }
                continue;
            }
            for (size_t r0 = 0; r0 < n_t; r0 += kGridRows) {
                const size_t r1 = std::min(n_t, r0 + (size_t)kGridRows), T = r1 - r0;
                Slab sl = open((int)T, false);
                for (size_t r = r0; r < r1; ++r) sl.theta[r - r0] = gr.thetas[r];
                // how many policies share a (budget, overhead): those after the first take further columns of their budget
                used.assign(n_b * kGridRows, 0);
                size_t b_at = 0, t_at = 0;
                wide.assign(n_b, 0);
                cell_of.resize(n_p);
                for (size_t x = 0; x < n_p; ++x) {
                    const uint32_t p = gr.pols[x];
                    place_of(gr.budgets, pc[p].budget, b_at); place_of(gr.thetas, theta_of(p), t_at);
                    cell_of[x] = kNone;
                    if (t_at < r0 || t_at >= r1) continue;
                    cell_of[x] = (uint32_t)(b_at * kGridRows + (t_at - r0));                 // (budget, overhead)
                    wide[b_at] = std::max(wide[b_at], ++used[cell_of[x]]);
                }
                size_t cols = 0;
                for (uint32_t& w : wide) { const uint32_t here = w; w = (uint32_t)cols; cols += here; }
                cells.assign(cols * T, kNone);
                used.assign(n_b * kGridRows, 0);
                for (size_t x = 0; x < n_p; ++x)
                    if (cell_of[x] != kNone) cells[(wide[cell_of[x] / kGridRows] + used[cell_of[x]]++) * T + cell_of[x] % kGridRows] = gr.pols[x];
                for (size_t c0 = 0; c0 < cols; c0 += kGridCols) close(sl, c0, std::min(cols, c0 + (size_t)kGridCols));
            }
        }
    }

    // ---- requests run by run or side by side: slab by slab, and within a wave's slabs with windows or without those of one way together
    int groups = 0;                                // that have requests
    for (int g = 0; g < G; ++g) groups += rb.ng[g] != 0;
    auto joins = [&](const Slab& sl) {
#ifdef DISCO_DEBUG
        if (std::getenv("DISCO_DEBUG_RUNS")) return false;
#endif
        bool inner = false;                                          // some budget parts the requests (0 and 1 do not)
        for (int x = 0; x < sl.K && !inner; ++x) { const float b = pc[tab[sl.cols + x]].budget; inner = b > 0.0f && b < 1.0f; }
        return !wide_class(sl.cls) && grid_joins(n, groups, sl.K, sl.T, inner);
    };
    for (size_t x = 0, end; x < slabs.size(); x = end) {
        auto like = [&](const Slab& sl) { return sl.cls / wave == slabs[x].cls / wave && wide_class(sl.cls) == wide_class(slabs[x].cls); };
        for (end = x + 1; end < slabs.size() && like(slabs[end]);) ++end;
        std::stable_partition(slabs.begin() + x, slabs.begin() + end, [&](const Slab& sl) { return !joins(sl); });
    }

    // ---- the difference tables of the slabs, laid out batch by batch: a batch's slabs have like numbers of rows, windows or
    //      none, and go one way.  Small ones lie side by side and are cleared by k_prep; beyond 64 MB a batch's tables are cleared, filled,
    //      added up and then belong to the next batch
    struct Batch { size_t first, count, wave; int T; bool wide, joined; uint64_t ttft, tbt, sums, at; };
    std::vector<Batch> batches;
    auto batch_bytes = [&](const Batch& b) { return (b.sums * 8 + b.tbt * (b.wide ? 8 : 4) + b.ttft * 4 + 15) / 16 * 16; };
    size_t most_slabs = 0;                         // of a batch that goes run by run
    int tallest = 1;
    for (size_t x = 0; x < slabs.size(); ++x) {
        Slab& sl = slabs[x];
        const bool wide_tables = wide_class(sl.cls), joined = joins(sl);
        if (batches.empty() || batch_bytes(batches.back()) > (256ull << 20) || grid_rows(batches.back().T) != grid_rows(sl.T) || sl.mixed ||
            slabs[x - 1].mixed || batches.back().wave != sl.cls / wave || batches.back().wide != wide_tables || batches.back().joined != joined)
            batches.push_back(Batch{x, 0, sl.cls / wave, 1, wide_tables, joined, 0, 0, 0, 0});
        Batch& b = batches.back();
        sl.ttft = b.ttft; sl.tbt = b.tbt; sl.sums = b.sums;
        b.ttft += grid_ttft_words(sl.K); b.tbt += grid_tbt_words(sl.K, sl.T); b.sums += grid_sum_words(sl.K, sl.T, G);
        ++b.count;
        b.T = std::max(b.T, sl.T);
        if (!joined) { most_slabs = std::max(most_slabs, b.count); tallest = std::max(tallest, sl.T); }
    }
    uint64_t grid_bytes = 0, all_bytes = 0;
    for (Batch& b : batches) { b.at = all_bytes; all_bytes += batch_bytes(b); grid_bytes = std::max(grid_bytes, batch_bytes(b)); }
    const bool side_by_side = all_bytes <= (64ull << 20);
    if (side_by_side) grid_bytes = all_bytes;
    else for (Batch& b : batches) b.at = 0;

    // ---- request chunks, of one group each: of the grid kernel, about two to each block that fits the GPU at once, 256
    //      requests (one a thread) or more (three to a block: k_grid and k_spread for 16 M requests in six groups under 128
    //      budgets by 8 overheads 369 us either way, under 16 by 2 218 instead of 205, in one group under 64 budgets 139
    //      instead of 133, a million 34 instead of 30)
    const uint32_t sms = (uint32_t)c->sms, kMaxChunk = 65280;
    auto chunk_size = [&](size_t want, uint32_t least) {
        const size_t ch = ((N1 + want - 1) / want + 255) / 256 * 256;
        return (uint32_t)std::min<size_t>(std::max<size_t>(ch, least), kMaxChunk);
    };
    // the chunks of the groups that Algorithm 1 finds device-constrained come first: Algorithm 2's wait map costs the
    // grid kernel more sweeps per chunk, and its blocks draw their work in list order, so the items drawn last (when
    // some blocks already idle) should be the cheap ones
    TablesIn tables;
    std::memset(&tables, 0, sizeof tables);
    auto plan_chunks = [&](int which, uint32_t CH) {
        uint32_t count = 0, &n_plan = tables.n_plan[which];
        for (int dear = 1; dear >= 0; --dear)
            for (int g = 0; g < G; ++g) {
                if ((c->gc[g].auto_device_constrained != 0) != (dear != 0) || rb.ng[g] == 0) continue;
                tables.plan[which][n_plan++] = ChunkPlan{count, rb.grp_off[g], rb.grp_off[g + 1], g};
                count += (rb.ng[g] - 1) / CH + 1;
            }
        tables.chunk_len[which] = CH; tables.n_chunks[which] = count;
    };
    const size_t at_once = (size_t)sms * grid_blocks_per_sm(tallest);
    if (most_slabs) plan_chunks(CHUNKS_RUNS, chunk_size(std::max<size_t>(2 * at_once / std::min<size_t>(most_slabs, 4), 1), 256));
    // (requests side by side: a chunk is a thread's request or a few)
    if (std::any_of(batches.begin(), batches.end(), [](const Batch& b) { return b.joined; })) plan_chunks(CHUNKS_JOINED, chunk_size((size_t)sms * 8, 256));
    if (any_pairs) {
        // of the pair kernel, whose blocks (a chunk and 32 policies each) take a multiprocessor's shared memory: the fewest whole rounds
        // of them, where a block costs as much as some 800 requests besides its own.  (300,000 requests in six groups under 32
        // policies, k_pairs_acc 56.7 us in chunks of 2,048 -- 150, two more than a round -- 50.7 in chunks of 1,024, 50.0 of 2,304.)
        size_t listed = 1;
        for (const ClassLists& L : lists) listed = std::max(listed, L.n_ext);
        for (const Slab& sl : slabs) if (sl.mixed) listed = std::max<size_t>(listed, sl.policies);
        const size_t tiles = (listed + 31) / 32;
        auto blocks = [&](size_t ch) { size_t k = 0; for (int g = 0; g < G; ++g) if (rb.ng[g]) k += (rb.ng[g] - 1) / ch + 1; return k * tiles; };
        uint32_t best = kMaxChunk;
        size_t least = ~(size_t)0;
        for (size_t rounds = 1; rounds <= 8; ++rounds) {
            const size_t at_most = rounds * sms;
            if ((size_t)groups * tiles > at_most) continue;
            size_t ch = chunk_size((at_most + tiles - 1) / tiles, 256);
            while (ch <= kMaxChunk && blocks(ch) > at_most) ch += 256;
            if (ch > kMaxChunk || rounds * (ch + 800) >= least) continue;
            best = (uint32_t)ch; least = rounds * (ch + 800);
        }
        plan_chunks(CHUNKS_PAIRS, best);
    }

    // ---- device memory: what must be clear comes first and together -- the work counters and tickets, the difference
    //      tables of the first batch, and the accumulators if some pairs are added to them one by one (k_spread writes those
    //      of all other policies)
    const size_t acc_bytes = (size_t)P * G * kNAcc * 8, hist_bytes = (size_t)P * kNBins * 8;
    const size_t first_bytes = side_by_side ? all_bytes : batches.empty() ? 0 : batch_bytes(batches[0]);
    const bool clear_accum = any_pairs || n == 0;
    Layout lay;
    const size_t o_work = lay.take(32 + batches.size() * 4), o_accum = clear_accum ? lay.take(acc_bytes + 2 * hist_bytes) : 0;
    const size_t o_grid = lay.bytes;
    lay.take(grid_bytes);
    const size_t clear_bytes = n == 0 ? o_grid : (o_grid + first_bytes + 15) / 16 * 16;      // (k_prep clears them)
    const bool clear_apart = clear_bytes > (64ull << 30);                                     // (beyond its 32-bit index)
    const size_t o_prep = lay.take((size_t)G * P * sizeof(Prep)), o_stats = lay.take(P * sizeof(disco_policy_stats_t) + 16);
    const size_t o_accum2 = clear_accum ? o_accum : lay.take(acc_bytes + 2 * hist_bytes);
    const size_t o_left = lay.take(any_mixed ? (N1 + kMaxGroups) * 4 : 0);
    std::vector<PolicyIn> policies_in(P);
    std::vector<PolicyKind> kinds;
    for (uint32_t p = 0, k = 0; p < P; ++p) {
        const PolicyConst& q = pc[p];
        auto like = [&](const PolicyKind& x) { return x.alpha == q.alpha && x.flags == q.flags && x.mode == q.mode && x.expected_len == q.expected_len && x.l_immediate == q.l_immediate; };
        if (k >= kinds.size() || !like(kinds[k])) {                  // (mostly that of the policy before; else one of the last few, or another)
            const size_t from = kinds.size() > 16 ? kinds.size() - 16 : 0;
            for (k = (uint32_t)from; k < kinds.size() && !like(kinds[k]);) ++k;
            if (k == kinds.size()) kinds.push_back(PolicyKind{q.alpha, q.flags, q.mode, q.expected_len, q.l_immediate, {0, 0, 0}});
        }
        policies_in[p] = PolicyIn{q.budget, q.theta, k, q.route_thr};
    }
    const size_t table_bytes = (size_t)P * sizeof(PolicyIn) + kinds.size() * sizeof(PolicyKind) + (classes.size() * sizeof(ClassConst) + 15) / 16 * 16 +
                               (tab.size() * 4 + 15) / 16 * 16 + (slabs.size() * sizeof(Slab) + 15) / 16 * 16;
    const size_t o_tables = lay.take(table_bytes);
    size_t o_chunks[kChunkTables];
    for (int k = 0; k < kChunkTables; ++k) o_chunks[k] = lay.take(tables.n_chunks[k] * sizeof(Chunk));
    if ((e = c->eval_mem.reserve(lay.bytes)) == cudaErrorMemoryAllocation && wave > 1) {
        cudaGetLastError();                                          // (again in smaller waves, which leave more room)
        c->rec_too_much = wave * rec_stride;
        c->rec_mem.release();
        return disco_eval_policies(c, pol, P, seed, out, stream);
    }
    if (e != cudaSuccess) return fail_cuda(e, "device allocation for the evaluation");
    char* mem = (char*)c->eval_mem.p;
    c->d_prep.p = mem + o_prep; c->d_accum.p = mem + o_accum2; c->d_stats.p = mem + o_stats; c->d_grid.p = mem + o_grid;
    c->d_left.p = mem + o_left; c->d_tables.p = mem + o_tables;
    c->d_acc.p = c->d_accum.p; c->d_hist_ttft.p = (char*)c->d_accum.p + acc_bytes;
    c->d_hist_tbt.p = (char*)c->d_accum.p + acc_bytes + hist_bytes;
    c->d_work.p = mem + o_work;
    uint32_t* tickets = (uint32_t*)((char*)c->d_work.p + 32);

    if (c->fin_imported) {            // an import replaced the totals the final reductions refer to: back to the trace's own
        c->fin_own.assign((size_t)2 * G, 0);
        for (int g = 0; g < G; ++g) { c->fin_own[g] = rb.grp_sum_n[g]; c->fin_own[G + g] = rb.ng[g]; }
        CU(cudaMemcpyAsync(c->fin_totals.p, c->fin_own.data(), c->fin_own.size() * 8, cudaMemcpyHostToDevice, st));
        c->fin_imported = false;
    }
    if (clear_apart) CU(cudaMemsetAsync(mem, 0, clear_bytes, st));

    // ---- small tables to the device with k_prep: one block, 16-byte aligned regions
    const bool in_launch = table_bytes <= kTablesInline;
    if (in_launch) c->tables_host.resize(kTablesInline / sizeof(uint4));
    else if (int rc = reserve_stage(c, table_bytes, st)) return rc;
    char *sp = in_launch ? (char*)c->tables_host.data() : (char*)c->stage, *dt = mem + o_tables;
    size_t off = 0;
    auto put = [&](const void* src, size_t bytes) {
        if (bytes) std::memcpy(sp + off, src, bytes);
        char* at = dt + off;
        off += (bytes + 15) / 16 * 16;
        return at;
    };
    const PolicyIn* d_pol = (const PolicyIn*)put(policies_in.data(), P * sizeof(PolicyIn));
    const PolicyKind* d_kinds = (const PolicyKind*)put(kinds.data(), kinds.size() * sizeof(PolicyKind));
    const uint32_t policy_vecs = (uint32_t)(off / 16);
    const ClassConst* d_classes = (const ClassConst*)put(classes.data(), classes.size() * sizeof(ClassConst));
    const uint32_t* d_tab = (const uint32_t*)put(tab.data(), tab.size() * 4);
    const Slab* d_slabs = (const Slab*)put(slabs.data(), slabs.size() * sizeof(Slab));
    const Chunk* d_pair_chunks = (const Chunk*)(mem + o_chunks[CHUNKS_PAIRS]);
    if (off / 16 > 0xFFFFFFFFull) return fail(DISCO_ENOMEM, "the tables of the policies are too large");

    // ---- Algorithms 1-3 for every (group, policy)
    tables.host = sp; tables.device = dt; tables.vecs = (uint32_t)(off / 16); tables.skip = n_beta ? 0u : policy_vecs;
    tables.kinds = (uint32_t)kinds.size();
    for (int k = 0; k < kChunkTables; ++k) tables.chunks[k] = (Chunk*)(mem + o_chunks[k]);
    tables.left = &c->z->tables_left; tables.read = c->stage_read; tables.turn = c->stage_turn + 1;
    CU(launch_prep(P, G, c->d_gc.as<GroupConst>(), c->cum_mass.as<int64_t>(),
                   c->cnt, c->F_sorted, c->F_off, c->d_prep.as<Prep>(), tables, mem, clear_apart ? 0 : clear_bytes, c->sms, st));
    if (!in_launch) ++c->stage_turn;
    g_launches += 1;
    // (one class, played out already, and a grid: the search's results are not needed before the pair kernel)
    const bool beside = n_beta && n_classes == 1 && n != 0 && !timed && !batches.empty() && !slabs[0].mixed;
    if (n_beta) {
        CU(launch_prep_beta(d_pol, d_kinds, P, c->cum_mass.as<int64_t>(), c->cnt, c->F_sorted,
                            c->F_off, c->tick_start.as<uint32_t>(), c->tick_cnt, d_tab + beta_at, n_beta,
                            *std::max_element(c->F_n.begin(), c->F_n.end()), c->d_prep.as<Prep>(), beside, st));
        g_launches += 1;
    }

    disco_pair_out_t po;
    std::memset(&po, 0, sizeof po);
    if (out) po = *out;
    const bool rows = po.ttft_s || po.tbt_mean_s || po.tbt_max_s || po.cost || po.tok_server || po.tok_device || po.mig_at ||
                      po.delayed || po.decision;

    uint32_t ticket = 0;
    const Prep* prep = c->d_prep.as<Prep>();
    uint64_t *acc = c->d_acc.as<uint64_t>(), *h_ttft = c->d_hist_ttft.as<uint64_t>(), *h_tbt = c->d_hist_tbt.as<uint64_t>(),
             *work = c->d_work.as<uint64_t>();
    size_t next = 0;                               // batch
    // ---- wave by wave: play every request out under the wave's classes, then evaluate their policies on the summaries
    for (size_t first = 0; first < n_classes && n != 0; first += wave) {
        const size_t last = std::min(n_classes, first + wave);
        if (timed) CU(cudaEventRecord(c->ev[0], st));
        ShortMany many;
        many.classes = d_classes; many.rec_stride = rec_stride; many.count = 0;
        for (size_t k = std::max<size_t>(first, 1); k < last && last - first > 1 && many.count < kShortMany; ++k) {
            if (!(plan[k].kinds & (1u << G_EXACT)) || !short_search(plan[k].search)) continue;
            plan[k].kinds &= ~(1u << G_EXACT);
            many.cls[many.count] = (uint32_t)k; many.slot[many.count++] = (uint32_t)slot_of(k);
        }
        // (free streams of other classes are played out beside these: nobody needs the others' results)
        size_t free_class = last;
        for (size_t k = std::max<size_t>(first, 1); k < last && many.count && !timed; ++k) {
            if (!plan[k].kinds) continue;
            if ((plan[k].kinds & (1u << G_FREE)) && !(plan[k].kinds & (1u << G_EXACT))) free_class = k;
            break;
        }
        if (many.count) {
            CU(launch_playout_many(tr, gc, c->knots.as<int32_t>(), k0, rec, many, free_class < last, c->sms, st));
            g_launches += 1;
        }
        for (size_t k = first; k < last; ++k)
            if ((k != 0 || timed) && plan[k].kinds) CU(play_out(k, k == free_class));
        if (timed) CU(cudaEventRecord(c->ev[2], st));
        while (next < batches.size() && batches[next].wave == first / wave) {
            // grids with tables of their own run beside each other (the one behind needs nothing of the one in front), then k_spread each
            size_t end = next + 1;
            const Slab& sl = slabs[batches[next].first];
            if (side_by_side && !sl.mixed)
                while (end < batches.size() && batches[end].wave == first / wave && !slabs[batches[end].first].mixed) ++end;
            auto tables_of = [&](const Batch& b) {
                char* base = (char*)c->d_grid.p + b.at;
                return GridTables{(uint32_t*)(base + b.sums * 8 + b.tbt * (b.wide ? 8 : 4)), base + b.sums * 8, (unsigned long long*)base};
            };
            LeftLists left = {nullptr, nullptr};
            if (sl.mixed) {
                left.list = c->d_left.as<uint32_t>(); left.count = left.list + N1;
                CU(cudaMemsetAsync(left.count, 0, (size_t)G * 4, st));
            }
            for (size_t k = next; k < end; ++k) {
                const Batch& b = batches[k];
                if (!side_by_side && k != 0) CU(cudaMemsetAsync((char*)c->d_grid.p + b.at, 0, batch_bytes(b), st));
                const int which = b.joined ? CHUNKS_JOINED : CHUNKS_RUNS;
                CU(launch_grid(tr, gc, d_classes, prep, P, d_slabs + b.first, (uint32_t)b.count, b.T, b.wide, d_tab, tables.chunks[which], tables.n_chunks[which], rec,
                               rec_stride, tables_of(b), left, k0, tickets + ticket, work, k > next || (beside && ticket == 0), k + 1 < end, any_waits,
                               b.joined, c->sms, st));
                ++ticket;
            }
            for (size_t k = next; k < end; ++k) {
                const Batch& b = batches[k];
                CU(launch_spread(tr, gc, d_slabs + b.first, (uint32_t)b.count, b.T, b.wide, d_tab, tables_of(b), acc, h_ttft, h_tbt, k > next, k + 1 < end, st));
                g_launches += 2;
            }
            if (sl.mixed) {
                const Batch& b = batches[next];
                CU(launch_pairs_acc(tr, gc, d_classes + sl.cls, prep, P, d_tab + sl.cells, sl.policies, d_pair_chunks,
                                    tables.n_chunks[CHUNKS_PAIRS], left.list, left.count, rec_of(sl.cls), acc, h_ttft, h_tbt, work, k0,
                                    sl.expected_len != 0, b.wide, st));
                g_launches += 1;
            }
            next = end;
        }
        for (size_t k = first; k < last; ++k) {
            if (!lists[k].n_ext) continue;
            CU(launch_pairs_acc(tr, gc, d_classes + k, prep, P, d_tab + lists[k].ext, (uint32_t)lists[k].n_ext,
                                d_pair_chunks, tables.n_chunks[CHUNKS_PAIRS], nullptr, nullptr, rec_of(k), acc, h_ttft, h_tbt,
                                work, k0, true, wide_class(k), st));
            g_launches += 1;
        }
        if (timed) CU(cudaEventRecord(c->ev[3], st));
        for (size_t k = first; k < last && rows; ++k) {
            if (!c->inv_there) {
                CU(launch_inverse(tr, c->inv.as<uint32_t>(), st));
                g_launches += 1;
                c->inv_there = true;
            }
            CU(launch_pairs_rows(tr, gc, d_classes + k, prep, P, d_tab + lists[k].all, (uint32_t)lists[k].n_all, rec_of(k), po, k0, extras, st));
            g_launches += 1;
        }
        if (timed) CU(cudaEventRecord(c->ev[4], st));
    }
    c->timing_valid = timed && n != 0;
    c->P = P; c->pol.swap(pc);
    c->evaluated = true;
    return 0;
} DISCO_CATCH

int disco_reduce_stats(disco_ctx_t* c, disco_policy_stats_t* stats, void* stream) try {
    if (!c || !stats) return fail(DISCO_EINVAL, "null argument");
    if (!c->evaluated) return fail(DISCO_EINVAL, "no evaluation to reduce");
    cudaStream_t st = (cudaStream_t)stream;
    // Statistics and the error word land in pinned host memory straight from the kernel: in the caller's array if it is
    // page-locked (from a few dozen records on, where the copy would count; the kernel writes words of eight bytes), else in
    // the context's.
    const size_t bytes = c->P * sizeof(disco_policy_stats_t);
    disco_policy_stats_t* to = nullptr;
    if (c->P >= 64 && (uintptr_t)stats % 8 == 0) {
        cudaPointerAttributes attr;
        if (cudaPointerGetAttributes(&attr, stats) != cudaSuccess) cudaGetLastError();
        else if (attr.type == cudaMemoryTypeHost && attr.devicePointer) to = (disco_policy_stats_t*)attr.devicePointer;
    }
    if (!to && bytes > c->stats_host_cap) {
        if (c->stats_host) cudaFreeHost(c->stats_host);
        c->stats_host = nullptr; c->stats_host_cap = 0;
        CU(cudaMallocHost(&c->stats_host, bytes));
        c->stats_host_cap = bytes;
    }
    CU(launch_finalize(c->P, c->G, c->d_gc.as<GroupConst>(), c->d_acc.as<uint64_t>(), c->d_hist_ttft.as<uint64_t>(),
                       c->d_hist_tbt.as<uint64_t>(), c->fin_totals.as<uint64_t>(),
                       c->d_stats.as<disco_policy_stats_t>(), to ? to : (disco_policy_stats_t*)c->stats_host, c->err, c->rb->err, st));
    CU(cudaStreamSynchronize(st));
    if (int rc = debug_check()) return rc;
    if (!to) std::memcpy(stats, c->stats_host, bytes);
    g_launches += 1;
    if (c->timing_valid) {
        for (int k = 0; k < 4; ++k) CU(cudaEventElapsedTime(&c->ms[k], c->ev[k], c->ev[k + 1]));
    }
    if (c->rb->err[2]) return fail(DISCO_ECUDA, "internal error: an inter-token interval fell outside its histogram window");
    c->reduced = true;
    return 0;
} DISCO_CATCH

int disco_select_policy(const disco_policy_stats_t* stats, uint32_t P, double cost_cap, float tbt_slo_s,
                        int32_t* best) try {
    if (!stats || !best || P == 0) return fail(DISCO_EINVAL, "null argument or P = 0");
    if (P > (1u << 19)) return fail(DISCO_EINVAL, "too many policies");
    // lexicographic objective: feasible first; then (P99 TTFT bin, mean TTFT, cost, index); none feasible: cheapest
    const double slo = (double)tbt_slo_s;
    int64_t pick = -1;
    bool pick_ok = false;
    for (uint32_t p = 0; p < P; ++p) {
        const disco_policy_stats_t& s = stats[p];
        if (s.bin_p99_tbt < 0 || s.bin_p99_tbt >= kNBins || s.bin_p99_ttft < 0 || s.bin_p99_ttft >= kNBins)
            return fail(DISCO_EINVAL, "histogram bin out of range (policy " + std::to_string(p) + ")");
        const bool ok = s.total_cost <= cost_cap && (double)host_bin_edge_ticks(s.bin_p99_tbt) * 1e-6 <= slo;
        bool take;
        if (pick < 0) take = true;
        else if (ok != pick_ok) take = ok;
        else {
            const disco_policy_stats_t& b = stats[pick];
            if (ok) {
                if (s.bin_p99_ttft != b.bin_p99_ttft) take = s.bin_p99_ttft < b.bin_p99_ttft;
                else if (s.mean_ttft_s != b.mean_ttft_s) take = s.mean_ttft_s < b.mean_ttft_s;
                else take = s.total_cost < b.total_cost;
            } else {
                take = s.total_cost < b.total_cost;
            }
        }
        if (take) { pick = p; pick_ok = ok; }
    }
    *best = (int32_t)pick;
    if (!pick_ok) return fail(DISCO_EINFEASIBLE, "no policy meets the cost cap and the TBT objective");
    return 0;
} DISCO_CATCH

int disco_select_policy_device(disco_ctx_t* c, double cost_cap, float tbt_slo_s, int32_t* best, void* stream) try {
    if (!c || !best) return fail(DISCO_EINVAL, "null argument");
    if (!c->reduced) return fail(DISCO_EINVAL, "reduce the statistics before selecting");
    cudaStream_t st = (cudaStream_t)stream;
    g_launches += 1;
    CU(launch_select(c->d_stats.as<disco_policy_stats_t>(), c->P, cost_cap, tbt_slo_s, c->sel_host, st));   // writes the pinned pair
    CU(cudaStreamSynchronize(st));
    if (int rc = debug_check()) return rc;
    *best = c->sel_host[1];
    if (c->sel_host[0] != 0) return fail(DISCO_EINFEASIBLE, "no policy meets the cost cap and the TBT objective");
    return 0;
} DISCO_CATCH

uint64_t disco_kernel_launch_count(void) { return g_launches.load(); }

int disco_set_timing(disco_ctx_t* c, int on) try {
    if (!c) return fail(DISCO_EINVAL, "null context");
    if (on) for (auto& e : c->ev) if (!e) CU(cudaEventCreate(&e));
    c->timing = on != 0;
    c->timing_valid = false;
    return 0;
} DISCO_CATCH

int disco_get_timing(disco_ctx_t* c, float* ms4) try {
    if (!c || !ms4) return fail(DISCO_EINVAL, "null argument");
    if (!c->timing_valid || !c->reduced) return fail(DISCO_EINVAL, "no timed evaluation has been reduced");
    for (int k = 0; k < 4; ++k) ms4[k] = c->ms[k];
    return 0;
} DISCO_CATCH

int disco_get_work_counts(disco_ctx_t* c, uint64_t* counts4, void* stream) try {
    if (!c || !counts4) return fail(DISCO_EINVAL, "null argument");
    if (!c->evaluated) return fail(DISCO_EINVAL, "no evaluation");
    cudaStream_t st = (cudaStream_t)stream;
    CU(cudaMemcpyAsync(counts4, c->d_work.p, 32, cudaMemcpyDeviceToHost, st));
    CU(cudaStreamSynchronize(st));
    return 0;
} DISCO_CATCH

int disco_get_histograms(disco_ctx_t* c, uint32_t p, uint64_t* ttft_hist, uint64_t* tbt_hist, void* stream) try {
    if (!c || !c->evaluated || p >= c->P) return fail(DISCO_EINVAL, "no evaluation or policy index out of range");
    cudaStream_t st = (cudaStream_t)stream;
    if (ttft_hist) CU(cudaMemcpyAsync(ttft_hist, c->d_hist_ttft.as<uint64_t>() + (size_t)p * kNBins, kNBins * 8, cudaMemcpyDeviceToHost, st));
    if (tbt_hist) CU(cudaMemcpyAsync(tbt_hist, c->d_hist_tbt.as<uint64_t>() + (size_t)p * kNBins, kNBins * 8, cudaMemcpyDeviceToHost, st));
    CU(cudaStreamSynchronize(st));
    return 0;
} DISCO_CATCH

int disco_get_prep(disco_ctx_t* c, uint32_t g, uint32_t p, disco_prep_t* out, void* stream) try {
    if (!c || !out || !c->evaluated || p >= c->P || g >= (uint32_t)c->G) return fail(DISCO_EINVAL, "bad argument");
    cudaStream_t st = (cudaStream_t)stream;
    Prep pr;
    CU(cudaMemcpyAsync(&pr, c->d_prep.as<Prep>() + (size_t)g * c->P + p, sizeof pr, cudaMemcpyDeviceToHost, st));
    CU(cudaStreamSynchronize(st));
    out->device_constrained = pr.device_constrained; out->l_th = pr.l_th; out->l_star = pr.l_star;
    out->B = c->pol[p].B; out->w_star = pr.w_star; out->w_tail = pr.w_tail; out->tau = c->pol[p].tau;
    out->beta_rule = pr.beta_rule; out->l_immediate = pr.beta_rule ? pr.l_star : 0; out->beta = pr.beta_rule ? pr.w_star : 0;
    if (pr.beta_rule) { out->l_star = 0; out->w_star = 0; }
    return 0;
} DISCO_CATCH

int64_t disco_get_group_tables(disco_ctx_t* c, uint32_t g, int64_t* cnt, int32_t* knots, int32_t* sorted_ticks,
                               uint64_t n_sorted, void* stream) try {
    if (!c || !c->loaded || g >= (uint32_t)c->G) return fail(DISCO_EINVAL, "bad argument");
    cudaStream_t st = (cudaStream_t)stream;
    // the tables Algorithms 1-3 read: the trace's own, or the whole trace's a caller has set
    const uint64_t ng = c->F_n[g];
    uint64_t off = c->rb->grp_off[g];
    if (c->tables_imported) { off = 0; for (uint32_t k = 0; k < g; ++k) off += c->F_n[k]; }
    // The length counts and knots of all groups come over together, with the first group's that is asked for after a load;
    // those of the others are then read from the copy.
    bool knots_on_host = true;
    if (knots) {
        cudaPointerAttributes attr;
        if (cudaPointerGetAttributes(&attr, knots) != cudaSuccess) cudaGetLastError();
        else knots_on_host = attr.type == cudaMemoryTypeHost || attr.type == cudaMemoryTypeUnregistered;
    }
    const bool fetch = (cnt || (knots && knots_on_host)) && !c->tab_host_now;
    if (fetch) {
        if (int rc = fetch_knots(c, st)) return rc;
        CU(cudaMemcpyAsync(c->tab_host, c->cnt, (size_t)c->G * kLengths * 4, cudaMemcpyDeviceToHost, st));
    }
    if (knots && !knots_on_host)
        CU(cudaMemcpyAsync(knots, c->knots.as<int32_t>() + (size_t)g * kNKnots, kNKnots * 4, cudaMemcpyDefault, st));
    const uint64_t k = std::min<uint64_t>(n_sorted, ng);
    if (sorted_ticks && k) CU(cudaMemcpyAsync(sorted_ticks, c->F_sorted + off, k * 4, cudaMemcpyDefault, st));
    // (what comes from the copy, or is known on the host, waits for nothing)
    if (fetch || (knots && !knots_on_host) || (sorted_ticks && k)) CU(cudaStreamSynchronize(st));
    if (fetch) c->tab_host_now = true;
    if (cnt) for (size_t i = 0; i < kLengths; ++i) cnt[i] = c->tab_host[g * kLengths + i];
    if (knots && knots_on_host) std::memcpy(knots, host_knots(c, (int)g), kNKnots * 4);
    return (int64_t)ng;
} DISCO_CATCH

int disco_set_group_tables(disco_ctx_t* c, const int64_t* cnt, const int32_t* ticks, const uint64_t* n_ticks,
                           void* stream) try {
    if (!c || !cnt || !n_ticks) return fail(DISCO_EINVAL, "null argument");
    if (!c->loaded) return fail(DISCO_EINVAL, "no trace loaded");
    cudaStream_t st = (cudaStream_t)stream;
    const int G = c->G;
    const size_t L = kLengths;
    uint64_t total = 0;
    if (int rc = reserve_stage(c, ((size_t)G * L + kMaxGroups + 1) * 4, st)) return rc;
    uint32_t *cnt32 = (uint32_t*)c->stage, *off = cnt32 + (size_t)G * L;      // counts of all groups, then the groups' offsets
    off[0] = 0;
    for (int g = 0; g < G; ++g) {
        const int64_t* from = cnt + (size_t)g * L;
        uint64_t by_length = 0, high = 0;
        for (size_t l = 0; l < L; ++l) {
            const uint64_t v = (uint64_t)from[l];
            high |= v >> 32; by_length += v;
            cnt32[(size_t)g * L + l] = (uint32_t)v;
        }
        if (high || from[0] != 0)
            return fail(DISCO_EINVAL, "length count negative, above 2^32 - 1 or at length 0 (group " + std::to_string(g) + ")");
        if (by_length != n_ticks[g])
            return fail(DISCO_EINVAL, "length counts do not add up to the number of TTFT ticks (group " + std::to_string(g) + ")");
        total += n_ticks[g];
        if (total > kMaxTicks) return fail(DISCO_EINVAL, "more than 2^32 - 2^20 requests behind the tables");
        off[g + 1] = (uint32_t)total;
    }
    if (total && !ticks) return fail(DISCO_EINVAL, "null argument");
    cudaError_t e;
    const size_t T1 = (size_t)std::max<uint64_t>(total, 1);
    const size_t tick_bytes = (size_t)G * kTickBins * 4;
    if ((e = c->F_sorted_imp.reserve(T1 * 4)) != cudaSuccess || (e = c->F_off_imp.reserve((size_t)(kMaxGroups + 1) * 4)) != cudaSuccess ||
        (e = c->sort_in.reserve(2 * ((T1 + 3) / 4 * 4) * 4 + std::max((size_t)sort_windows((uint32_t)total, G) * 8, (size_t)kOnceWindows * 16))) != cudaSuccess)
        return fail_cuda(e, "device allocation for the tables");
    // ticks in this device's memory are read where they are (another device's may not be mapped here, and a kernel cannot read
    // words across their alignment); sort_in: a copy of others, the same by bin, the windows
    bool on_device = false;
    if (total) {
        int dev = 0;
        CU(cudaGetDevice(&dev));
        cudaPointerAttributes attr;
        if (cudaPointerGetAttributes(&attr, ticks) != cudaSuccess) cudaGetLastError();
        else on_device = (attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged) && attr.device == dev && (uintptr_t)ticks % alignof(int32_t) == 0;
    }
    int32_t* copy = c->sort_in.as<int32_t>();
    const int32_t* in = on_device ? ticks : copy;
    const size_t T4 = (T1 + 3) / 4 * 4;
    if (total && !on_device) CU(cudaMemcpyAsync(copy, ticks, (size_t)total * 4, cudaMemcpyDefault, st));
    CU(cudaMemcpyAsync(c->F_off_imp.p, off, (size_t)(G + 1) * 4, cudaMemcpyHostToDevice, st));
    CU(cudaMemcpyAsync(c->cnt, cnt32, (size_t)G * L * 4, cudaMemcpyHostToDevice, st));
    CU(cudaEventRecord(c->stage_free, st));
    c->tab_host_now = false;
    LoadArgs a = {};
    a.n = (uint32_t)total; a.G = G; a.ticks = in; a.off = c->F_off_imp.as<uint32_t>();
    a.z = c->z; a.zero_bytes = sizeof(LoadZero) + tick_bytes; a.tick_cnt = c->tick_cnt; a.tick_start = c->tick_start.as<uint32_t>(); a.tick_at = a.tick_start + (size_t)G * kTickBins;
    a.binned = (uint32_t*)copy + T4; a.windows = (uint2*)(copy + 2 * T4); a.once.windows = (unsigned long long*)a.windows; a.rounds = 1; a.sorted = c->F_sorted_imp.as<int32_t>();
    if (!total) CU(cudaMemsetAsync(c->z, 0, sizeof(LoadZero), st));
    if (total) { CU(run_sort_ticks(a, c->sms, st)); g_launches += 1; }
    CU(launch_tables_imported(G, c->cnt, c->cum_mass.as<int64_t>(), c->F_sorted_imp.as<int32_t>(), c->F_off_imp.as<uint32_t>(),
                              c->knots.as<int32_t>(), st));
    g_launches += 1;
    // error word and each group's largest tick, the last of its knots (the largest hand-off latency a draw from F can give)
    if (int rc = fetch_knots(c, st)) return rc;
    int32_t* err_host = c->rb->err;
    CU(cudaMemcpyAsync(err_host, c->err, 16, cudaMemcpyDeviceToHost, st));
    CU(cudaStreamSynchronize(st));
    if (int rc = debug_check()) { c->loaded = false; return rc; }
    c->evaluated = c->reduced = false;
    if (err_host[3] == 2) { c->loaded = false; return fail(DISCO_ECUDA, "internal error: the blocks of the sort lost each other"); }
    if (!err_host[0] && err_host[3] == 1) {
        if (int rc = radix_sort(c, in, c->F_off_imp.as<uint32_t>(), (uint32_t)total, c->F_sorted_imp.as<int32_t>(), st)) { c->loaded = false; return rc; }
        CU(launch_tables_imported(G, c->cnt, c->cum_mass.as<int64_t>(), c->F_sorted_imp.as<int32_t>(), c->F_off_imp.as<uint32_t>(),
                                  c->knots.as<int32_t>(), st));
        g_launches += 1;
        if (int rc = fetch_knots(c, st)) return rc;
        CU(cudaStreamSynchronize(st));
        if (int rc = debug_check()) { c->loaded = false; return rc; }
    }
    if (err_host[0]) {
        c->loaded = false;                  // the length counts have been overwritten: the context must be reloaded
        return fail(DISCO_EINVAL, "negative TTFT tick at position " + std::to_string(err_host[1]) + "; reload the trace");
    }
    c->F_sorted = c->F_sorted_imp.as<int32_t>(); c->F_off = c->F_off_imp.as<uint32_t>();
    c->tables_imported = true;
    for (int g = 0; g < G; ++g) { c->F_n[g] = n_ticks[g]; c->rb->knot_max[g] = host_knots(c, g)[kNKnots - 1]; }
    return 0;
} DISCO_CATCH

uint64_t disco_accumulator_words(disco_ctx_t* c) {
    if (!c || !c->evaluated) return 0;
    return (uint64_t)c->P * c->G * kNAcc + 2ull * c->P * kNBins + 2ull * c->G;
}

int disco_export_accumulators(disco_ctx_t* c, uint64_t* words, void* stream) try {
    if (!c || !words) return fail(DISCO_EINVAL, "null argument");
    if (!c->evaluated) return fail(DISCO_EINVAL, "no evaluation to export");
    cudaStream_t st = (cudaStream_t)stream;
    const size_t head = (size_t)c->P * c->G * kNAcc + 2 * (size_t)c->P * kNBins;      // one block of d_accum
    CU(cudaMemcpyAsync(words, c->d_accum.p, head * 8, cudaMemcpyDefault, st));
    CU(cudaMemcpyAsync(words + head, c->fin_totals.p, (size_t)2 * c->G * 8, cudaMemcpyDefault, st));
    CU(cudaStreamSynchronize(st));
    return 0;
} DISCO_CATCH

int disco_import_accumulators(disco_ctx_t* c, const uint64_t* words, void* stream) try {
    if (!c || !words) return fail(DISCO_EINVAL, "null argument");
    if (!c->evaluated) return fail(DISCO_EINVAL, "evaluate the policies first: the accumulators take their shape from it");
    cudaStream_t st = (cudaStream_t)stream;
    const size_t head = (size_t)c->P * c->G * kNAcc + 2 * (size_t)c->P * kNBins;
    CU(cudaMemcpyAsync(c->d_accum.p, words, head * 8, cudaMemcpyDefault, st));
    CU(cudaMemcpyAsync(c->fin_totals.p, words + head, (size_t)2 * c->G * 8, cudaMemcpyDefault, st));
    CU(cudaStreamSynchronize(st));
    c->reduced = false;
    c->fin_imported = true;
    return 0;
} DISCO_CATCH

int disco_debug_selftest(void* stream) try {
#ifdef DISCO_DEBUG
    // a kernel offers an index beyond its bound to the check: the access is skipped, the record comes back as an error
    CU(run_debug_selftest((cudaStream_t)stream));
    CU(cudaStreamSynchronize((cudaStream_t)stream));
    g_launches += 1;
    return debug_check();
#else
    (void)stream;
    return fail(DISCO_EINVAL, "not a checked build (compile with -DDISCO_DEBUG)");
#endif
} DISCO_CATCH

int disco_measure_alu_peak(double* lane_instr_per_s, double* token_steps_per_s, void* stream) try {
    if (!lane_instr_per_s) return fail(DISCO_EINVAL, "null argument");
    int dev = 0, sms = 0;
    CU(cudaGetDevice(&dev));
    CU(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    double rate = 0.0;
    CU(run_alu_peak(sms, &rate, (cudaStream_t)stream));
    g_launches += 3;
    *lane_instr_per_s = rate * 13.0;
    if (token_steps_per_s) *token_steps_per_s = rate;
    return 0;
} DISCO_CATCH

}  // extern "C"
