// A CUDA runtime that runs nothing, for tests of the library's host side on a machine without a GPU (preloaded in front of
// the real one).  Device and page-locked memory is ordinary memory, kernels are not run; the ingestion kernel's launch
// leaves a report of an accepted trace and is remembered.  A test says what memory a range of addresses is to be taken for.
#include <cuda_runtime_api.h>
#include <sys/mman.h>

#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "load.cuh"

namespace {
struct Range { const char* at; size_t bytes; cudaMemoryType type; int device; };
std::vector<Range> ranges;
std::map<const void*, std::string> kernels;
uint64_t copied = 0, loads = 0;                 // bytes copied out of the ranges; ingestion kernels launched
const void* last_ticks = nullptr;               // what the last of them was given
const void* last_stats = nullptr;               // where the statistics' kernel was to write on the host
uint32_t first_packed = 0;                      // ... and the lengths of the first request, if it was given a packed trace
unsigned last_blocks = 0;                       // ... its grid, and whether its words were said to be zero
bool last_zeroed = false;
int multiprocessors = 148;
size_t device_left = ~(size_t)0;                // bytes that cudaMalloc gives out
std::map<void*, size_t> device;                 // what it has given out
std::vector<std::pair<void*, size_t>> given_back;
cudaError_t last_error = cudaSuccess;
void* symbol = nullptr;                         // where the library's device array lies
std::map<const char*, size_t> locked;           // host memory that the library has page-locked
const void *last_words = nullptr, *last_report = nullptr;
struct Write { void* to; const void* from; size_t bytes; };
std::vector<Write> pending;                     // work that a stream still holds
struct Word { volatile uint32_t* to; uint32_t value; };
std::vector<Word> reports;                      // words that kernels under way will write
uint64_t device_waits = 0;
std::map<std::string, uint64_t> launched;       // by (mangled) name
void finish() {
    for (const Write& w : pending) std::memcpy(w.to, w.from, w.bytes);
    for (const Word& w : reports) *w.to = w.value;
    pending.clear();
    reports.clear();
}

const Range* range_of(const void* p) {
    for (const Range& r : ranges) if ((const char*)p >= r.at && (const char*)p < r.at + r.bytes) return &r;
    return nullptr;
}
cudaError_t launch(const void* f, dim3 grid, void** args) {
    ++launched[kernels[f]];
    if (kernels[f].find("k_finalize") != std::string::npos) last_stats = *(const void**)args[8];
    if (kernels[f].find("k_prep") != std::string::npos && kernels[f].find("k_prep_beta") == std::string::npos) {
        const disco::TablesIn& in = *(const disco::TablesIn*)args[8];
        if ((size_t)in.vecs * 16 > disco::kTablesInline) reports.push_back({in.read, in.turn});
    }
    if (kernels[f].find("k_load") == std::string::npos) return cudaSuccess;
    const disco::LoadArgs& a = *(const disco::LoadArgs*)args[0];
    ++loads;
    last_ticks = a.ticks;
    last_blocks = grid.x;
    last_zeroed = a.once.zeroed;
    last_words = a.z;
    last_report = a.readback;
    if (a.packed) first_packed = *(const uint32_t*)a.packed;
    if (a.readback) {
        std::memset(a.readback, 0, sizeof *a.readback);
        a.readback->ng[0] = a.readback->grp_off[1] = a.n;
        a.readback->max_n = 1;
    }
    return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- the test's side
void fake_memory(const void* at, size_t bytes, int type, int device) { ranges.push_back({(const char*)at, bytes, (cudaMemoryType)type, device}); }
uint64_t fake_copied(void) { return copied; }
uint64_t fake_loads(void) { return loads; }
const void* fake_last_ticks(void) { return last_ticks; }
const void* fake_last_stats(void) { return last_stats; }
uint32_t fake_first_packed(void) { return first_packed; }
unsigned fake_last_blocks(void) { return last_blocks; }
int fake_last_zeroed(void) { return last_zeroed; }
void fake_multiprocessors(int n) { multiprocessors = n; }
void fake_device_left(uint64_t bytes) { device_left = bytes; }
void fake_reset_device(void) { symbol = nullptr; locked.clear(); }
int fake_last_words_in_place(void) { return last_words >= symbol && (const char*)last_words < (const char*)symbol + (16 << 20); }
int fake_last_report_locked(void) { void* p; return cudaHostGetDevicePointer(&p, (void*)last_report, 0) == cudaSuccess; }
uint64_t fake_device_waits(void) { return device_waits; }
uint64_t fake_launched(const char* part) {      // kernels launched whose names hold `part`
    uint64_t n = 0;
    for (const auto& k : launched) if (k.first.find(part) != std::string::npos) n += k.second;
    return n;
}
void fake_pending(void* to, const void* from, size_t bytes) { pending.push_back({to, from, bytes}); }

// ---- what the library calls
void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { kernels[f] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t* smem, void* stream) { *smem = 0; *(void**)stream = nullptr; return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void* f, dim3 grid, dim3, void** args, size_t, cudaStream_t) { return launch(f, grid, args); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) { return launch(f, c->gridDim, args); }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = multiprocessors; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 1; return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) {
    // (a mapping: large sizes cost nothing until they are touched; not given back, a case is a short process)
    *p = mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    return *p != MAP_FAILED ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaMalloc(void** p, size_t n) {
    if (n > device_left) { last_error = cudaErrorMemoryAllocation; return last_error; }
    // what was given back is given out again, with what has been written there
    for (auto f = given_back.begin(); f != given_back.end(); ++f)
        if (f->second == n) { *p = f->first; given_back.erase(f); device[*p] = n; device_left -= n; return cudaSuccess; }
    const cudaError_t e = cudaMallocHost(p, n);
    if (e == cudaSuccess) { device[*p] = n; device_left -= n; }
    return e;
}
cudaError_t cudaFree(void* p) {
    const auto f = device.find(p);
    if (f == device.end()) return cudaSuccess;
    device_left += f->second;
    given_back.push_back(*f);
    device.erase(f);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void*) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* to, const void* from, size_t n, cudaMemcpyKind, cudaStream_t) {
    finish();                                     // (in stream order)
    if (range_of(from)) copied += n;              // (may not be readable here)
    else std::memcpy(to, from, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    std::memset(a, 0, sizeof *a);
    const Range* r = range_of(p);
    a->type = r ? r->type : cudaMemoryTypeUnregistered;
    a->device = r ? r->device : -2;
    a->devicePointer = r ? (void*)p : nullptr;
    a->hostPointer = r && r->type != cudaMemoryTypeDevice ? (void*)p : nullptr;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    if (!symbol) cudaMallocHost(&symbol, 16 << 20);
    *p = symbol;
    return cudaSuccess;
}
cudaError_t cudaHostRegister(void* p, size_t n, unsigned) { locked[(const char*)p] = n; return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void** p, void* host, unsigned) {
    for (const auto& r : locked) if ((const char*)host >= r.first && (const char*)host < r.first + r.second) { *p = host; return cudaSuccess; }
    return last_error = cudaErrorInvalidValue;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { finish(); return cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t) {
    if (pending.empty() && reports.empty()) return cudaSuccess;
    if (pending.empty()) finish();                // (kernels get on meanwhile)
    return cudaErrorNotReady;
}
cudaError_t cudaDeviceSynchronize(void) { ++device_waits; finish(); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)&ranges; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.0f; return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { const cudaError_t e = last_error; last_error = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return "an error of the fake runtime"; }
}
