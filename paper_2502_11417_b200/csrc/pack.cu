// Traces in pageable host memory: packed to nine bytes a request in page-locked slots by several threads, while the calling
// thread copies to the device what is packed, several neighbouring chunks at a time (a copy costs some 5 us besides its
// bytes, and copies issued by several threads wait for one another).  Bound: reading the caller's columns (14 bytes a
// request, 10 GB/s a thread, 54 GB/s eight) and the link (9 bytes a request).
#include "pack.cuh"

#include <algorithm>
#if defined(__SSE2__)
#include <emmintrin.h>
#endif

namespace disco {

namespace {

// Requests [lo, lo + n) of the trace, packed.
void pack_range(const disco_trace_desc_t& d, uint32_t lo, uint32_t n, char* out) {
    uint32_t* ln = (uint32_t*)out;
    float* t = (float*)(out + (size_t)kPackChunk * 4);
    uint8_t* g = (uint8_t*)(out + (size_t)kPackChunk * 8);
    const int32_t *prompt = d.prompt_len + lo, *outlen = d.output_len + lo;
    const float* ttft = d.server_ttft_s + lo;
    static const uint8_t none[kPackChunk] = {};
    const uint8_t *sp = d.server_profile ? d.server_profile + lo : none, *dp = d.device_profile ? d.device_profile + lo : none;
    const uint32_t ns = d.n_servers, nd = d.n_devices;                    // (at most 64 each)
    uint32_t i = 0;
#if defined(__SSE2__)
    // Stored past the caches: the copy engine reads lines that other cores hold at 12 GB/s instead of 54 (18 MB packed by
    // eight threads: 0.4 + 1.5 ms, past the caches 0.25 + 0.35).
    const __m128i zero = _mm_setzero_si128(), all = _mm_set1_epi32(-1);
    const __m128i l_end = _mm_set1_epi32(kMaxPrompt + 1), o_end = _mm_set1_epi32(kMaxOutput + 1);
    const __m128i s_max = _mm_set1_epi8((char)(ns - 1u)), d_max = _mm_set1_epi8((char)(nd - 1u)), nd16 = _mm_set1_epi16((short)nd);
    auto get = [](const void* p) { return _mm_loadu_si128((const __m128i*)p); };
    for (; i + 16 <= n; i += 16) {
        for (uint32_t k = i; k < i + 16; k += 4) {
            const __m128i l = get(prompt + k), o = get(outlen + k);
            const __m128i l_ok = _mm_and_si128(_mm_cmplt_epi32(l, l_end), _mm_cmpgt_epi32(l, zero));
            const __m128i o_ok = _mm_and_si128(_mm_cmplt_epi32(o, o_end), _mm_cmpgt_epi32(o, zero));
            _mm_stream_si128((__m128i*)(ln + k), _mm_or_si128(_mm_and_si128(l, l_ok), _mm_slli_epi32(_mm_and_si128(o, o_ok), 16)));
            _mm_stream_si128((__m128i*)(t + k), get(ttft + k));
        }
        const __m128i s = get(sp + i), v = get(dp + i);
        const __m128i ok = _mm_and_si128(_mm_cmpeq_epi8(_mm_min_epu8(s, s_max), s), _mm_cmpeq_epi8(_mm_min_epu8(v, d_max), v));
        const __m128i a = _mm_add_epi16(_mm_mullo_epi16(_mm_unpacklo_epi8(s, zero), nd16), _mm_unpacklo_epi8(v, zero));
        const __m128i b = _mm_add_epi16(_mm_mullo_epi16(_mm_unpackhi_epi8(s, zero), nd16), _mm_unpackhi_epi8(v, zero));
        _mm_stream_si128((__m128i*)(g + i), _mm_or_si128(_mm_and_si128(_mm_packus_epi16(a, b), ok), _mm_andnot_si128(ok, all)));
    }
#endif
    for (; i < n; ++i) {
        const uint32_t l = (uint32_t)prompt[i], o = (uint32_t)outlen[i], s = sp[i], v = dp[i];
        ln[i] = (l - 1u < (uint32_t)kMaxPrompt ? l : 0u) | (o - 1u < (uint32_t)kMaxOutput ? o : 0u) << 16;
        t[i] = ttft[i];
        g[i] = (uint8_t)(s < ns && v < nd ? s * nd + v : 255u);
    }
#if defined(__SSE2__)
    _mm_sfence();
#endif
}

}  // namespace

Packer::~Packer() {
    {
        std::lock_guard<std::mutex> lock(m_);
        stop_ = true;
    }
    wake_.notify_all();
    for (auto& t : threads_) t.join();
    for (cudaEvent_t e : copied_) if (e) cudaEventDestroy(e);
    if (slots_) cudaFreeHost(slots_);
}

cudaError_t Packer::reserve_slots(uint32_t slots) {
    cudaError_t e;
    if (slots > have_) {
        if (slots_) cudaFreeHost(slots_);
        slots_ = nullptr; have_ = 0;
        if ((e = cudaMallocHost((void**)&slots_, slots * kPackBytes))) { slots_ = nullptr; return e; }
        have_ = slots;
    }
    for (uint32_t k = 0; k < slots; ++k)
        if (!copied_[k] && (e = cudaEventCreateWithFlags(&copied_[k], cudaEventDisableTiming))) { copied_[k] = nullptr; return e; }
    return cudaSuccess;
}

// A packing thread: takes chunks until there are none left.
void Packer::run() {
    uint64_t seen = 0;
    for (;;) {
        {
            std::unique_lock<std::mutex> lock(m_);
            wake_.wait(lock, [&] { return stop_ || job_ != seen; });
            if (stop_) return;
            seen = job_;
        }
        const uint32_t n = (uint32_t)d_->n, chunks = (n + kPackChunk - 1) / kPackChunk;
        for (uint32_t c; (c = chunk_.fetch_add(1)) < chunks;) {
            while (c >= freed_.load(std::memory_order_acquire) + have_) std::this_thread::yield();   // (ends: the caller counts a failed copy as done)
            const uint32_t lo = c * kPackChunk;
            pack_range(*d_, lo, std::min(kPackChunk, n - lo), slots_ + (c % have_) * kPackBytes);
            packed_[c % have_].store(c + 1, std::memory_order_release);
        }
        {
            std::lock_guard<std::mutex> lock(m_);
            --running_;
        }
        done_.notify_one();
    }
}

// The calling thread: copies what the others have packed, in order.
cudaError_t Packer::copy_runs(uint32_t chunks, char* dev, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    uint32_t issued = 0, freed = 0, ends[kSlots];                     // of the copies under way, where they end
    uint32_t first = 0, last = 0;
    while (issued < chunks) {
        uint32_t k = issued;
        while (k < chunks && k - issued < kRun && k % have_ >= issued % have_ && packed_[k % have_].load(std::memory_order_acquire) == k + 1) ++k;
        if (k > issued) {
            if (!e) {
                const uint32_t s = issued % have_;
                e = cudaMemcpyAsync(dev + (size_t)issued * kPackBytes, slots_ + s * kPackBytes, (k - issued) * kPackBytes, cudaMemcpyHostToDevice, st);
                if (!e) e = cudaEventRecord(copied_[(k - 1) % have_], st);
            }
            ends[last++ % kSlots] = k;
            issued = k;
        } else if (first != last && issued - freed > have_ / 2) {
            // the packers may soon want the slots
            const uint32_t end = ends[first % kSlots];
            const cudaError_t q = e ? cudaSuccess : cudaEventQuery(copied_[(end - 1) % have_]);
            if (q != cudaErrorNotReady) {
                if (q) e = q;
                ++first;
                freed_.store(freed = end, std::memory_order_release);
            }
        } else {
            std::this_thread::yield();
        }
    }
    return e;
}

cudaError_t Packer::pack(const disco_trace_desc_t& d, char* dev, cudaStream_t st, const char** at) {
    const uint32_t n = (uint32_t)d.n, chunks = (n + kPackChunk - 1) / kPackChunk;
    cudaError_t e;
    if ((e = reserve_slots(std::min(chunks, kSlots)))) return e;
    // (copies of an earlier call are done: the ingestion kernel behind them has run)
    if (n <= kPackInPlace) {
        pack_range(d, 0, n, slots_);
        *at = slots_;
        return cudaSuccess;
    }
    *at = dev;
    // two chunks or more to each thread that is started; at most eight, and half the host's cores
    const size_t want = std::min<size_t>({chunks / 2, (size_t)std::thread::hardware_concurrency() / 2, 8});
    d_ = &d;
    chunk_.store(0);
    freed_.store(0);
    for (auto& p : packed_) p.store(0);
    if (want > 1) {
        std::lock_guard<std::mutex> lock(m_);
        try {
            while (threads_.size() < want) threads_.emplace_back(&Packer::run, this);
        } catch (...) {}                                               // fewer threads, then
        running_ = threads_.size();
        if (running_) ++job_;
    }
    if (want <= 1 || threads_.empty()) {
        for (uint32_t c = 0; c < chunks; ++c) {
            const uint32_t s = c % have_, lo = c * kPackChunk;
            if (c >= have_ && (e = cudaEventSynchronize(copied_[s]))) return e;
            pack_range(d, lo, std::min(kPackChunk, n - lo), slots_ + s * kPackBytes);
            if ((e = cudaMemcpyAsync(dev + (size_t)c * kPackBytes, slots_ + s * kPackBytes, kPackBytes, cudaMemcpyHostToDevice, st)) ||
                (e = cudaEventRecord(copied_[s], st))) return e;
        }
        return cudaSuccess;
    }
    wake_.notify_all();
    e = copy_runs(chunks, dev, st);
    std::unique_lock<std::mutex> lock(m_);
    done_.wait(lock, [&] { return running_ == 0; });
    return e;
}

}  // namespace disco
