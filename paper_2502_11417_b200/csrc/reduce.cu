// Final reductions per policy (Sec. 5.1 metrics: mean and tail TTFT, P99 TBT, cost) and policy selection.
#include "disco_internal.cuh"

namespace disco {

namespace {

__device__ __forceinline__ double bin_edge_seconds(int b) {
    long long edge = b < 32 ? b : ((long long)(32 + (b & 31)) << ((b >> 5) - 1));
    return __dmul_rn((double)edge, 1e-6);
}

// Nearest-rank quantiles of one 864-bin histogram by a warp: the bins are read side by side into shared memory, lane i
// then owns bins [27 i, 27 i + 27) (an odd stride: no bank conflicts beyond the two words of a count); the bin holding the
// ceil(q*M)-th smallest item is found from the lanes' prefix counts.  All lanes return the bins.
constexpr int kBinsPerLane = kNBins / 32;
static_assert(kBinsPerLane * 32 == kNBins, "864 bins split evenly over a warp");

template <int NQ>
__device__ __forceinline__ void warp_quantile_bins(const unsigned long long* __restrict__ hist, unsigned long long* s_hist,
                                                   unsigned long long M, const double (&qs)[NQ], int (&out)[NQ]) {
    const int lane = threadIdx.x & 31;
    unsigned long long v[kBinsPerLane];
#pragma unroll
    for (int i = 0; i < kBinsPerLane; ++i) v[i] = hist[i * 32 + lane];
#pragma unroll
    for (int i = 0; i < kBinsPerLane; ++i) s_hist[i * 32 + lane] = v[i];
    __syncwarp();
    const unsigned long long* mine = s_hist + lane * kBinsPerLane;
    unsigned long long sum = 0;
#pragma unroll
    for (int i = 0; i < kBinsPerLane; ++i) sum += mine[i];
    unsigned long long incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned long long up = __shfl_up_sync(0xFFFFFFFFu, incl, off);
        if (lane >= off) incl += up;
    }
    // every rank at once, on one walk over the lane's bins: the walks of the lanes that hold them took 0.7 us a rank one after
    // another
    const unsigned long long excl = incl - sum;
    unsigned long long rank[NQ];
    int found[NQ];
#pragma unroll
    for (int k = 0; k < NQ; ++k) {
        rank[k] = (unsigned long long)ceil(__dmul_rn(qs[k], (double)M));
        if (rank[k] < 1) rank[k] = 1;
        found[k] = 0;                                     // bins in front of the one that holds the rank
    }
    unsigned long long acc = excl;
#pragma unroll
    for (int i = 0; i < kBinsPerLane; ++i) {
        acc += mine[i];
#pragma unroll
        for (int k = 0; k < NQ; ++k) found[k] += acc < rank[k] ? 1 : 0;
    }
#pragma unroll
    for (int k = 0; k < NQ; ++k) {
        const unsigned owner = __ballot_sync(0xFFFFFFFFu, rank[k] > excl && rank[k] <= incl);
        int bin = __shfl_sync(0xFFFFFFFFu, lane * kBinsPerLane + found[k], owner ? __ffs(owner) - 1 : 0);
        if (!owner) bin = kNBins - 1;
        if (!DBG_OK(bin, kNBins, DBG_K_FINALIZE, DBG_BIN)) bin = kNBins - 1;
        out[k] = M ? bin : 0;
    }
}

// One block of three warps per policy: TTFT quantiles, TBT quantile, sums.  Bound: latency at few policies, the histograms
// (14 KB a policy) at many.
__global__ void __launch_bounds__(96)
k_finalize(uint32_t P, int G, const GroupConst* __restrict__ gc,
                           const unsigned long long* __restrict__ acc, const unsigned long long* __restrict__ hist_ttft,
                           const unsigned long long* __restrict__ hist_tbt,
                           const unsigned long long* __restrict__ fin_totals,
                           disco_policy_stats_t* __restrict__ stats, disco_policy_stats_t* __restrict__ stats_host,
                           const int32_t* __restrict__ err, int32_t* __restrict__ err_host) {
    // stats_host: pinned host memory, written straight from here (no copy operation behind the kernel)
    __shared__ unsigned long long s_hist[2][kNBins];
    __shared__ unsigned long long tot[kNAcc];
    __shared__ int qb[4];
    __shared__ disco_policy_stats_t s_out;
    const uint32_t p = blockIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    grid_dependency_wait();
    // fin_totals: output tokens and requests per group behind the accumulators (this trace's, or what a caller
    // merged from several shards)
    unsigned long long N = 0, sum_n = 0;
    for (int g = 0; g < G; ++g) { N += fin_totals[G + g]; sum_n += fin_totals[g]; }
    if (w == 0) {
        const double q[3] = {0.50, 0.95, 0.99};
        int b[3];
        warp_quantile_bins<3>(hist_ttft + (size_t)p * kNBins, s_hist[0], N, q, b);
        if (lane < 3) qb[lane] = lane == 0 ? b[0] : lane == 1 ? b[1] : b[2];
    } else if (w == 1) {
        const double q[1] = {0.99};
        int b[1];
        warp_quantile_bins<1>(hist_tbt + (size_t)p * kNBins, s_hist[1], sum_n - N, q, b);
        if (lane == 0) qb[3] = b[0];
    } else {
        if (p == 0 && lane < 4) err_host[lane] = err[lane];                                    // error word rides along
        if (lane < kNAcc) {
            unsigned long long s = 0;
            for (int g = 0; g < G; ++g) s += acc[((size_t)p * G + g) * kNAcc + lane];
            tot[lane] = s;
        }
        // Eq. 8 on the exact integer token totals of each group: a lane per group, added up in the groups' order
        double cost = 0.0;
        for (int g0 = 0; g0 < G; g0 += 32) {
            double x = 0.0;
            if (g0 + lane < G) {
                const int g = g0 + lane;
                const unsigned long long* a = acc + ((size_t)p * G + g) * kNAcc;
                const unsigned long long dev_tok = a[A_TOK_DEVICE];
                const double dts = (double)(fin_totals[g] - dev_tok), dtd = (double)dev_tok;
                const double pts = (double)a[A_PRE_SERVER], ptd = (double)a[A_PRE_DEVICE];
                const GroupConst& c = gc[g];
                const double srv = __dadd_rn(__dmul_rn(c.cps_d, pts), __dmul_rn(c.cds_d, dts));
                const double dev = __dadd_rn(__dmul_rn(c.cpd_d, ptd), __dmul_rn(c.cdd_d, dtd));
                x = __dadd_rn(srv, __dmul_rn(c.lambda_d, dev));
            }
            for (int k = 0; k < min(32, G - g0); ++k) cost = __dadd_rn(cost, __shfl_sync(0xFFFFFFFFu, x, k));
        }
        __syncwarp();
        if (lane == 0) {
            disco_policy_stats_t& s = s_out;
            s.mean_ttft_s = N ? __ddiv_rn(__dmul_rn((double)tot[A_TTFT_SUM], 1e-6), (double)N) : 0.0;
            s.total_cost = cost;
            s.n_requests = N; s.n_intervals = sum_n - N;
            s.n_device_only = tot[A_DEVICE_ONLY]; s.n_race = tot[A_RACE];
            s.n_server_only = N - s.n_device_only - s.n_race;          // every request takes exactly one decision
            s.n_device_started = s.n_device_only + s.n_race;           // the device ran in both of these
            s.n_device_won = tot[A_DEVICE_WON]; s.n_migrations = tot[A_MIGR];
            s.tok_device = tot[A_TOK_DEVICE]; s.tok_server = sum_n - tot[A_TOK_DEVICE];
            s.prefill_tok_server = tot[A_PRE_SERVER]; s.prefill_tok_device = tot[A_PRE_DEVICE];
            s.delayed_tokens = tot[A_DELAYED];
        }
    }
    __syncthreads();
    if (w != 0) return;
    if (lane == 0) {
        disco_policy_stats_t& s = s_out;
        s.bin_p50_ttft = qb[0]; s.bin_p95_ttft = qb[1]; s.bin_p99_ttft = qb[2]; s.bin_p99_tbt = qb[3];
    }
    if (lane < 4) (&s_out.p50_ttft_s)[lane] = (float)bin_edge_seconds(qb[lane]);
    __syncwarp();
    // (a record leaves in words side by side: single fields would cross the link one by one)
    constexpr int kWords = (int)(sizeof(disco_policy_stats_t) / 8);
    static_assert(sizeof(disco_policy_stats_t) % 8 == 0 && kWords <= 32, "a lane per word");
    if (lane < kWords) {
        const unsigned long long v = ((const unsigned long long*)&s_out)[lane];
        ((unsigned long long*)(stats + p))[lane] = v;
        ((unsigned long long*)(stats_host + p))[lane] = v;
    }
}

// Lexicographic objective of the selection: (tail TTFT bin, mean TTFT, cost, index), feasible policies only.
struct Pick { int feasible; int bin; double mean, cost; int idx; };

__device__ __forceinline__ bool better(const Pick& a, const Pick& b) {
    if (b.idx < 0) return a.idx >= 0;
    if (a.idx < 0) return false;
    if (a.feasible != b.feasible) return a.feasible > b.feasible;
    if (a.feasible) {
        if (a.bin != b.bin) return a.bin < b.bin;
        if (a.mean != b.mean) return a.mean < b.mean;
        if (a.cost != b.cost) return a.cost < b.cost;
    } else {
        if (a.cost != b.cost) return a.cost < b.cost;        // none feasible: cheapest
    }
    return a.idx < b.idx;
}

__global__ void k_select(const disco_policy_stats_t* __restrict__ stats, uint32_t P, double cost_cap, double tbt_slo,
                         int32_t* __restrict__ result) {
    __shared__ Pick best[256];
    Pick mine = {0, 0, 0.0, 0.0, -1};
    for (uint32_t p = threadIdx.x; p < P; p += blockDim.x) {
        const disco_policy_stats_t& s = stats[p];
        Pick c;
        c.feasible = (s.total_cost <= cost_cap) && (bin_edge_seconds(s.bin_p99_tbt) <= tbt_slo);
        c.bin = s.bin_p99_ttft; c.mean = s.mean_ttft_s; c.cost = s.total_cost; c.idx = (int)p;
        if (better(c, mine)) mine = c;
    }
    best[threadIdx.x] = mine;
    __syncthreads();
    for (int off = 128; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off && better(best[threadIdx.x + off], best[threadIdx.x]))
            best[threadIdx.x] = best[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        result[0] = best[0].feasible ? 0 : DISCO_EINFEASIBLE;
        result[1] = best[0].idx;
    }
}

}  // namespace

DBG_TRANSLATION_UNIT()

cudaError_t launch_finalize(uint32_t P, int G, const GroupConst* gc, const uint64_t* acc, const uint64_t* hist_ttft,
                            const uint64_t* hist_tbt, const uint64_t* fin_totals,
                            disco_policy_stats_t* stats, disco_policy_stats_t* stats_host, const int32_t* err, int32_t* err_host,
                            cudaStream_t st) {
    return launch_after(k_finalize, P, 96, 0, st, P, G, gc, (const unsigned long long*)acc,
                        (const unsigned long long*)hist_ttft, (const unsigned long long*)hist_tbt,
                        (const unsigned long long*)fin_totals, stats, stats_host, err, err_host);
}

cudaError_t launch_select(const disco_policy_stats_t* stats, uint32_t P, double cost_cap, float tbt_slo_s,
                          int32_t* result, cudaStream_t st) {
    k_select<<<1, 256, 0, st>>>(stats, P, cost_cap, (double)tbt_slo_s, result);
    return cudaGetLastError();
}

}  // namespace disco
