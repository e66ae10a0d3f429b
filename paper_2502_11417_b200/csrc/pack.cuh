// Traces in pageable host memory on their way to the device (pack.cu).
#pragma once

#include <atomic>
#include <condition_variable>
#include <mutex>
#include <thread>
#include <vector>

#include "disco_internal.cuh"

namespace disco {

// Packed requests, a chunk of 8,192 after another: lengths (prompt | output << 16), TTFTs, groups (a byte each).  A length
// or profile out of range is packed as 0 or 255, which the ingestion kernel refuses with the same error.
constexpr uint32_t kPackChunk = 8192;
constexpr size_t kPackBytes = (size_t)kPackChunk * 9;
constexpr uint32_t kPackInPlace = 8192;       // traces up to this size are read from the pinned slots, without a copy
inline size_t packed_bytes(uint32_t n) { return ((size_t)n + kPackChunk - 1) / kPackChunk * kPackBytes; }

// Packs with a few threads of its own.  One per context: its threads and its page-locked slots live as long.
class Packer {
public:
    Packer() = default;
    ~Packer();
    Packer(const Packer&) = delete;
    Packer& operator=(const Packer&) = delete;
    // Packs the trace into `dev` (packed_bytes(n) of it) by copies on the stream, or, up to kPackInPlace requests, into
    // page-locked memory of its own; *at receives where.  Must not be called again before the kernel that reads the result
    // has run.
    cudaError_t pack(const disco_trace_desc_t& d, char* dev, cudaStream_t st, const char** at);

private:
    static constexpr uint32_t kSlots = 128;   // chunks in page-locked memory at a time (9 MB)
    static constexpr uint32_t kCopies = 32;   // copies under way, at most
    static constexpr uint32_t kRunMin = 8, kRun = 32;   // chunks that go with one copy
    static constexpr size_t kThreadsMost = 12;
    cudaError_t reserve_slots(uint32_t slots);
    cudaError_t copy_runs(uint32_t chunks, char* dev, cudaStream_t st);
    void pack_chunk(uint32_t c);
    void run();

    char* slots_ = nullptr;
    uint32_t have_ = 0;
    cudaEvent_t copied_[kCopies] = {};        // after each copy, by turns
    std::vector<std::thread> threads_;
    std::mutex m_;
    std::condition_variable wake_, done_;
    size_t calls_ = 0;                        // threads the job in work still asks for
    size_t running_ = 0;                      // ... and those that have not ended their part
    bool stop_ = false;
    const disco_trace_desc_t* d_ = nullptr;   // the job in work
    std::atomic<uint32_t> chunk_{0};          // next chunk to pack
    std::atomic<uint32_t> freed_{0};          // chunks whose copies are done: their slots are free
    std::atomic<uint32_t> packed_[kSlots] = {};   // 1 + the chunk that a slot holds
};

}  // namespace disco
