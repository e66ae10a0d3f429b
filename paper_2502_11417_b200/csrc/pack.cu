// Traces in pageable host memory: packed to nine bytes a request in page-locked slots by several threads, while the calling
// thread copies to the device what is packed, several neighbouring chunks at a time (a copy costs some 5 us besides its
// bytes, 2 of them behind the one in front, and copies issued by several threads wait for one another), and packs itself while there
// is nothing to copy.  Bound: reading the caller's columns (14 bytes a request, 11 GB/s a thread, 55 GB/s eight, 74 twelve, 77 sixteen of
// 16 cores; with prefetches half of that) and the link (9 bytes a request).
// (Loads from pageable arrays, us, with chunks of 32,768 requests, eight threads and a calling thread that only copies, and now: 50,000
// requests 119 and 90, 100,000 131 and 101, 200,000 151 and 126, 2 million 652 and 597, 16 million 5,030 and 4,170.)
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
    for (uint32_t k = 0; k < std::min(slots, kCopies); ++k)
        if (!copied_[k] && (e = cudaEventCreateWithFlags(&copied_[k], cudaEventDisableTiming))) { copied_[k] = nullptr; return e; }
    return cudaSuccess;
}

void Packer::pack_chunk(uint32_t c) {
    const uint32_t lo = c * kPackChunk;
    pack_range(*d_, lo, std::min(kPackChunk, (uint32_t)d_->n - lo), slots_ + (c % have_) * kPackBytes);
    packed_[c % have_].store(c + 1, std::memory_order_release);
}

// A packing thread: takes chunks until there are none left.
void Packer::run() {
    for (;;) {
        {
            std::unique_lock<std::mutex> lock(m_);
            wake_.wait(lock, [&] { return stop_ || calls_ != 0; });
            if (stop_) return;
            --calls_;
        }
        const uint32_t chunks = ((uint32_t)d_->n + kPackChunk - 1) / kPackChunk;
        for (uint32_t c; (c = chunk_.fetch_add(1)) < chunks;) {
            while (c >= freed_.load(std::memory_order_acquire) + have_) std::this_thread::yield();   // (ends: the caller counts a failed copy as done)
            pack_chunk(c);
        }
        {
            std::lock_guard<std::mutex> lock(m_);
            --running_;
        }
        done_.notify_one();
    }
}

// The calling thread: copies what has been packed, in order, and packs while there is nothing to copy.
cudaError_t Packer::copy_runs(uint32_t chunks, char* dev, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    uint32_t issued = 0, freed = 0, ends[kCopies];                    // of the copies under way, where they end
    uint32_t first = 0, last = 0, mine = chunks;                      // mine: a chunk taken whose slot is not free yet
    auto ready = [&](uint32_t c) { return packed_[c % have_].load(std::memory_order_acquire) == c + 1; };
    while (issued < chunks) {
        uint32_t k = issued;
        while (k < chunks && k - issued < kRun && k % have_ >= issued % have_ && ready(k)) ++k;
        // (a few chunks at a time, but for the last ones and those in front of the ring's end)
        if (last - first < kCopies && (k - issued >= kRunMin || (k > issued && (k == chunks || k % have_ == 0)))) {
            if (!e) {
                const uint32_t s = issued % have_;
                e = cudaMemcpyAsync(dev + (size_t)issued * kPackBytes, slots_ + s * kPackBytes, (k - issued) * kPackBytes, cudaMemcpyHostToDevice, st);
                if (!e) e = cudaEventRecord(copied_[last % kCopies], st);
            }
            ends[last++ % kCopies] = k;
            issued = k;
        } else if (first != last && (issued - freed > have_ / 2 || last - first == kCopies)) {
            // the packers may soon want the slots
            const cudaError_t q = e ? cudaSuccess : cudaEventQuery(copied_[first % kCopies]);
            if (q != cudaErrorNotReady) {
                if (q) e = q;
                freed_.store(freed = ends[first++ % kCopies], std::memory_order_release);
                continue;
            }
        }
        if (mine == chunks && chunk_.load(std::memory_order_relaxed) < chunks) mine = std::min(chunks, chunk_.fetch_add(1));
        if (mine < chunks && mine < freed + have_) { pack_chunk(mine); mine = chunks; }
        else std::this_thread::yield();
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
    // two chunks or more to each thread that is started; at most twelve, and three quarters of the host's cores
    const size_t want = std::min<size_t>({chunks / 2, (size_t)std::thread::hardware_concurrency() * 3 / 4, kThreadsMost});
    d_ = &d;
    chunk_.store(0);
    freed_.store(0);
    for (auto& p : packed_) p.store(0);
    size_t called = 0;
    if (want > 1) {
        std::lock_guard<std::mutex> lock(m_);
        try {
            while (threads_.size() < want) threads_.emplace_back(&Packer::run, this);
        } catch (...) {}                                               // fewer threads, then
        called = calls_ = running_ = std::min(want, threads_.size());
    }
    for (size_t k = 0; k < called; ++k) wake_.notify_one();
    e = copy_runs(chunks, dev, st);
    std::unique_lock<std::mutex> lock(m_);
    running_ -= calls_;                                                // (who has not come by now is not needed)
    calls_ = 0;
    done_.wait(lock, [&] { return running_ == 0; });
    return e;
}

}  // namespace disco
