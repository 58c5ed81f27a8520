// A stand-in for the CUDA runtime that runs no kernel: the library's host code, linked against it, runs on a machine
// without a GPU, and a test can make any call fail.  Device memory is host memory; copies and memsets of up to 4096 bytes
// are made, larger ones are not (a large copy to the host is filled with one byte value).  Work that is queued on a stream
// stays pending until something waits for the stream, directly or through an event; a large block that is given back
// while any work is pending is counted (the real cudaFree would wait, the library's pool of idle blocks does not).
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

constexpr size_t kSmall = 4096, kPooled = 64ull << 20;      // blocks above kPooled never enter the library's pool

struct Op {
    long prev, dep;
    bool done;
};
std::vector<Op> ops;
long pending = 0;
struct Stream {
    long tail = -1;
    bool capturing = false;
};
struct Event {
    long op = -1;
    bool capturing = false;
};
std::map<cudaStream_t, Stream> streams;
std::map<cudaEvent_t, Event> events;
std::map<void*, size_t> blocks;
std::map<const void*, std::string> names;
std::vector<std::string> launched;
long calls = 0, fail_at = -1, violations = 0;
std::uint64_t free_bytes = 1ull << 38;
cudaError_t last = cudaSuccess;
bool scalar_on = false;
long no_memory = 0, fail_n = 1l << 60;                       // allocations still to fail, those that fail together
double scalar = 0.0;
int fill = 0;
struct Config {
    dim3 g, b;
    size_t smem;
    cudaStream_t st;
} config;

// Counts a call that may fail; the armed one does.
bool fails(cudaError_t e) {
    if (calls++ != fail_at) return false;
    last = e;
    return true;
}
void queue(cudaStream_t st, long dep = -1) {
    Stream& s = streams[st];
    if (s.capturing) return;
    ops.push_back({s.tail, dep, false});
    s.tail = (long)ops.size() - 1;
    pending++;
}
void finish(long op) {
    std::vector<long> todo{op};
    while (!todo.empty()) {
        const long i = todo.back();
        todo.pop_back();
        if (i < 0 || ops[i].done) continue;
        ops[i].done = true;
        pending--;
        todo.push_back(ops[i].prev);
        todo.push_back(ops[i].dep);
    }
}
void finish_all() {
    for (Op& o : ops) o.done = true;
    pending = 0;
}
bool on_device(const void* p) {
    auto it = blocks.upper_bound(const_cast<void*>(p));
    if (it == blocks.begin()) return false;
    --it;
    return static_cast<const char*>(p) < static_cast<char*>(it->first) + it->second;
}
void copy(void* dst, const void* src, size_t n) {
    if (n == 8 && scalar_on && !on_device(dst)) std::memcpy(dst, &scalar, 8);
    else if (n <= kSmall) std::memcpy(dst, src, n);
    else if (!on_device(dst)) std::memset(dst, fill, n);
}

}  // namespace

extern "C" {

// ---- what a test sets and reads
void fake_reset() {
    finish_all();
    ops.clear();
    for (auto& s : streams) s.second = Stream();
    for (auto& e : events) e.second = Event();
    launched.clear();
    calls = violations = 0;
    fail_at = -1;
    last = cudaSuccess;
    scalar_on = false;
    no_memory = 0;
    fill = 0;
}
// The k-th call from now fails; an allocation with the next n - 1 ones, or with all after it (n = 0).
void fake_fail_at(long k, long n) { calls = 0; fail_at = k; no_memory = 0; fail_n = n ? n : 1l << 60; }
long fake_calls() { return calls; }
long fake_violations() { return violations; }
void fake_scalar(double v) { scalar_on = true; scalar = v; }      // the value of every 8-byte copy to the host
void fake_fill(int byte) { fill = byte; }
void fake_free_bytes(uint64_t n) { free_bytes = n; }
uint64_t fake_held() {
    uint64_t n = 0;
    for (auto& b : blocks) n += b.second;
    return n;
}
long fake_blocks() { return (long)blocks.size(); }
long fake_launched(const char* part) {
    long n = 0;
    for (auto& s : launched) n += s.find(part) != std::string::npos;
    return n;
}

// ---- memory
cudaError_t cudaMalloc(void** p, size_t n) {
    if (fails(cudaErrorMemoryAllocation)) no_memory = fail_n;
    if (no_memory > 0) {
        no_memory--;
        return last = cudaErrorMemoryAllocation;
    }
    *p = std::malloc(n);
    if (n <= kSmall) std::memset(*p, 0xa5, n);
    blocks[*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    if (!p) return cudaSuccess;
    auto it = blocks.find(p);
    if (it == blocks.end()) std::abort();                        // freed twice
    if (it->second > kPooled && pending > 0) violations++;
    finish_all();
    blocks.erase(it);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = free_bytes; *t = 1ull << 38; return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind, cudaStream_t st) {
    if (fails(cudaErrorUnknown)) return cudaErrorUnknown;
    copy(dst, src, n);
    queue(st);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* dst, const void* src, size_t n, cudaMemcpyKind) {
    if (fails(cudaErrorUnknown)) return cudaErrorUnknown;
    copy(dst, src, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t st) {
    if (fails(cudaErrorUnknown)) return cudaErrorUnknown;
    if (n <= kSmall) std::memset(p, v, n);
    queue(st);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { return cudaMemsetAsync(p, v, n, nullptr); }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    std::memset(a, 0, sizeof *a);
    a->type = on_device(p) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = const_cast<void*>(s); return cudaSuccess; }

// ---- devices and errors
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { finish_all(); return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return "made to fail"; }
const char* cudaGetErrorName(cudaError_t) { return "made to fail"; }

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    if (fails(cudaErrorUnknown)) return cudaErrorUnknown;
    static uintptr_t next = 0x1000;
    *s = reinterpret_cast<cudaStream_t>(next += 16);
    streams[*s] = Stream();
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { streams.erase(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { finish(streams[s].tail); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    if (fails(cudaErrorUnknown)) return cudaErrorUnknown;
    static uintptr_t next = 0x100000;
    *e = reinterpret_cast<cudaEvent_t>(next += 16);
    events[*e] = Event();
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { events.erase(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    if (fails(cudaErrorUnknown)) return cudaErrorUnknown;
    events[e] = Event{streams[s].tail, streams[s].capturing};
    return cudaSuccess;
}
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned) { return cudaEventRecord(e, s); }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    if (fails(cudaErrorUnknown)) return cudaErrorUnknown;
    if (events[e].capturing) streams[s].capturing = true;
    else queue(s, events[e].op);
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { finish(events[e].op); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    if (fails(cudaErrorUnknown)) return cudaErrorUnknown;
    streams[s].capturing = true;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    for (auto& s : streams) s.second.capturing = false;
    for (auto& e : events) e.second.capturing = false;
    if (fails(cudaErrorUnknown)) return cudaErrorUnknown;
    *g = reinterpret_cast<cudaGraph_t>(1);
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
    if (fails(cudaErrorUnknown)) return cudaErrorUnknown;
    *x = reinterpret_cast<cudaGraphExec_t>(1);
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) {
    if (fails(cudaErrorUnknown)) return cudaErrorUnknown;
    queue(s);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

// ---- kernels
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) {
    return fails(cudaErrorUnknown) ? cudaErrorUnknown : cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 1;
    return fails(cudaErrorUnknown) ? cudaErrorUnknown : cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult*) {
    *p = nullptr;
    return cudaErrorUnknown;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* st) {
    config = Config{g, b, smem, st};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
    *g = config.g;
    *b = config.b;
    *smem = config.smem;
    *static_cast<cudaStream_t*>(st) = config.st;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t st) {
    if (fails(cudaErrorUnknown)) return cudaErrorUnknown;
    launched.push_back(names[reinterpret_cast<const void*>(k)]);
    queue(st);
    return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}

}  // extern "C"
