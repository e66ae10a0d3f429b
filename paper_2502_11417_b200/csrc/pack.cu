// Traces in pageable host memory: packed to nine bytes a request in page-locked slots by several threads, and copied to the
// device chunk by chunk while the next ones are packed.  Bound: reading the caller's columns (14 bytes a request, which
// one thread does at some 12 GB/s: 2.4 ms for 2 million requests through the driver's own staging) and the link (9 bytes a
// request).
#include "pack.cuh"

#include <algorithm>

namespace disco {

namespace {

void pack_range(const disco_trace_desc_t& d, uint32_t lo, uint32_t n, char* out) {
    uint32_t* ln = (uint32_t*)out;
    float* t = (float*)(out + (size_t)kPackChunk * 4);
    uint8_t* g = (uint8_t*)(out + (size_t)kPackChunk * 8);
    const int32_t *prompt = d.prompt_len + lo, *outlen = d.output_len + lo;
    for (uint32_t i = 0; i < n; ++i) {
        const uint32_t l = (uint32_t)prompt[i], o = (uint32_t)outlen[i];
        ln[i] = (l - 1u < (uint32_t)kMaxPrompt ? l : 0u) | (o - 1u < (uint32_t)kMaxOutput ? o : 0u) << 16;
    }
    std::copy(d.server_ttft_s + lo, d.server_ttft_s + lo + n, t);
    const uint32_t ns = d.n_servers, nd = d.n_devices;
    if (d.server_profile && d.device_profile) {
        const uint8_t *sp = d.server_profile + lo, *dp = d.device_profile + lo;
        for (uint32_t i = 0; i < n; ++i) { const uint32_t s = sp[i], v = dp[i]; g[i] = (uint8_t)(s < ns && v < nd ? s * nd + v : 255u); }
    } else if (d.server_profile) {
        const uint8_t* sp = d.server_profile + lo;
        for (uint32_t i = 0; i < n; ++i) g[i] = (uint8_t)(sp[i] < ns ? sp[i] * nd : 255u);
    } else if (d.device_profile) {
        const uint8_t* dp = d.device_profile + lo;
        for (uint32_t i = 0; i < n; ++i) g[i] = (uint8_t)(dp[i] < nd ? dp[i] : 255u);
    } else {
        std::fill(g, g + n, (uint8_t)0);
    }
}

}  // namespace

Packer::~Packer() {
    {
        std::lock_guard<std::mutex> lock(m_);
        stop_ = true;
    }
    wake_.notify_all();
    for (auto& t : threads_) t.join();
    for (Lane& l : lanes_)
        for (int k = 0; k < 2; ++k) {
            if (l.free[k]) cudaEventDestroy(l.free[k]);
            if (l.slot[k]) cudaFreeHost(l.slot[k]);
        }
}

cudaError_t Packer::open_lane(Lane& l, bool both) {
    for (int k = 0; k < (both ? 2 : 1); ++k) {
        cudaError_t e;
        if (!l.slot[k] && (e = cudaMallocHost((void**)&l.slot[k], kPackBytes))) { l.slot[k] = nullptr; return e; }
        if (!l.free[k] && (e = cudaEventCreateWithFlags(&l.free[k], cudaEventDisableTiming))) { l.free[k] = nullptr; return e; }
    }
    return cudaSuccess;
}

// Takes chunks until there are none left.
cudaError_t Packer::work(Lane& l) {
    const uint32_t n = (uint32_t)d_->n, chunks = (n + kPackChunk - 1) / kPackChunk;
    cudaError_t e;
    if ((e = open_lane(l, true))) return e;
    for (uint32_t c; (c = chunk_.fetch_add(1)) < chunks;) {
        const int k = l.next;
        l.next ^= 1;
        if ((e = cudaEventSynchronize(l.free[k]))) return e;           // the slot's last copy (none: returns at once)
        const uint32_t lo = c * kPackChunk;
        pack_range(*d_, lo, std::min(kPackChunk, n - lo), l.slot[k]);
        if ((e = cudaMemcpyAsync(dev_ + (size_t)c * kPackBytes, l.slot[k], kPackBytes, cudaMemcpyHostToDevice, st_))) return e;
        if ((e = cudaEventRecord(l.free[k], st_))) return e;
    }
    return cudaSuccess;
}

void Packer::run(size_t lane) {
    uint64_t seen = 0;
    cudaSetDevice(device_);
    for (;;) {
        {
            std::unique_lock<std::mutex> lock(m_);
            wake_.wait(lock, [&] { return stop_ || job_ != seen; });
            if (stop_) return;
            seen = job_;
        }
        const cudaError_t e = work(lanes_[lane]);
        if (e) error_.store((int)e);
        {
            std::lock_guard<std::mutex> lock(m_);
            --running_;
        }
        done_.notify_one();
    }
}

cudaError_t Packer::pack(const disco_trace_desc_t& d, char* dev, cudaStream_t st, const char** at) {
    const uint32_t n = (uint32_t)d.n, chunks = (n + kPackChunk - 1) / kPackChunk;
    cudaError_t e;
    if (lanes_.empty()) {
        if ((e = cudaGetDevice(&device_))) return e;
        lanes_.resize(8);
    }
    if (n <= kPackInPlace) {
        if ((e = open_lane(lanes_[0], false)) || (e = cudaEventSynchronize(lanes_[0].free[0]))) return e;
        pack_range(d, 0, n, lanes_[0].slot[0]);
        *at = lanes_[0].slot[0];
        return cudaSuccess;
    }
    // four chunks or more to each thread that is started; at most seven beside the caller, and half the host's cores
    const size_t want = std::min<size_t>({chunks / 4, (size_t)std::thread::hardware_concurrency() / 2, lanes_.size() - 1});
    d_ = &d; dev_ = dev; st_ = st;
    chunk_.store(0);
    error_.store(0);
    if (want) {
        std::lock_guard<std::mutex> lock(m_);
        try {
            while (threads_.size() < want) threads_.emplace_back(&Packer::run, this, threads_.size() + 1);
        } catch (...) {}                                               // fewer threads, then
        running_ = threads_.size();
        ++job_;
    }
    if (want) wake_.notify_all();
    e = work(lanes_[0]);
    if (want) {
        std::unique_lock<std::mutex> lock(m_);
        done_.wait(lock, [&] { return running_ == 0; });
    }
    if (!e) e = (cudaError_t)error_.load();
    *at = dev;
    return e;
}

}  // namespace disco
