// A CUDA runtime without a GPU, for tests of the library's host side: the library's own objects are linked against this
// file instead of the CUDA runtime.  Device memory is host memory that remembers its device, copies happen at once, a
// launch runs nothing except for the few kernels whose sizes the host reads back, which report what the test asked for.
// Calls that a real runtime would refuse (a block freed twice, a launch with a stream of another device) are counted.
#include <cuda_runtime_api.h>
#include <stdint.h>
#include <string.h>

#include <cstdlib>
#include <map>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "grf_internal.cuh"

namespace {

constexpr int DEVICES = 2;

struct Block { size_t bytes; int device; };

std::recursive_mutex lock;
std::map<char*, Block> blocks;                       // device memory by address
std::map<const void*, std::string>& kernels()        // host stub -> kernel name (filled before this file's own statics exist)
{
    static auto* m = new std::map<const void*, std::string>;
    return *m;
}
std::vector<std::string> log_;                       // launches and waits, in order
size_t live[DEVICES], limit[DEVICES];
long mallocs, frees, refused, errors;
thread_local int current = 0;
thread_local cudaError_t last = cudaSuccess;
// what the kernels report: non-zeros of Phi and Psi, deposits of both, edges, node-list entries, key entries, positions,
// longest list
int64_t report[9];

void* captured = nullptr;                            // the stream that is captured
cudaStreamCaptureMode capture_mode = cudaStreamCaptureModeGlobal;
void* denominators = nullptr;                        // where the last launch of the plain gather's kernel writes them

bool no_heap = false;                                // the library's operator new throws
struct Own {                                         // ... while this file's own calls do not
    bool was = no_heap;
    Own() { no_heap = false; }
    ~Own() { no_heap = was; }
};

struct Stream { int device; };
struct Event { int device; };

cudaError_t fail(cudaError_t e) { last = e; return e; }
cudaError_t bad() { ++errors; return fail(cudaErrorInvalidValue); }
// calls that a thread may not make while a stream is captured, unless it says that it knows what it does
bool unsafe() { return captured && capture_mode != cudaStreamCaptureModeRelaxed; }
cudaError_t invalidates() { ++errors; return fail(cudaErrorStreamCaptureUnsupported); }

int device_of(const void* p)
{
    auto it = blocks.upper_bound((char*)p);
    if (it == blocks.begin()) return -1;
    --it;
    return (char*)p < it->first + it->second.bytes ? it->second.device : -1;
}

}  // namespace

void* operator new(size_t n)
{
    void* p = no_heap ? nullptr : malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void* operator new(size_t n, const std::nothrow_t&) noexcept { return no_heap ? nullptr : malloc(n ? n : 1); }
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }

extern "C" {

// ---- what a test sets and reads
void fake_reset()
{
    std::lock_guard<std::recursive_mutex> g(lock);
    const Own own;
    for (int d = 0; d < DEVICES; ++d) limit[d] = ~(size_t)0;
    mallocs = frees = refused = errors = 0;
    no_heap = false;
    memset(report, 0, sizeof(report));
    log_.clear();
    current = 0;
    captured = denominators = nullptr;
    capture_mode = cudaStreamCaptureModeGlobal;
}
void fake_capture(void* stream) { captured = stream; }
void* fake_denominators() { return denominators; }
void fake_report(int which, int64_t value) { report[which] = value; }
void fake_no_heap(int on) { no_heap = on != 0; }
void fake_limit(int device, size_t bytes) { limit[device] = bytes; }      // an allocation beyond it fails
size_t fake_live(int device) { return live[device]; }
long fake_mallocs() { return mallocs; }
long fake_frees() { return frees; }
long fake_refused() { return refused; }
long fake_errors() { return errors; }
int fake_device_of(const void* p) { std::lock_guard<std::recursive_mutex> g(lock); return device_of(p); }
int fake_current() { return current; }
void fake_set_current(int d) { current = d; }
void* fake_stream(int device) { return new Stream{device}; }
int fake_log_size() { return (int)log_.size(); }
const char* fake_log(int i) { return log_[i].c_str(); }
void fake_log_clear() { log_.clear(); }

// ---- devices
cudaError_t cudaGetDeviceCount(int* n) { *n = DEVICES; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = current; return cudaSuccess; }
cudaError_t cudaSetDevice(int d)
{
    if (d < 0 || d >= DEVICES) return bad();
    current = d;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize()
{
    if (captured) return invalidates();
    const Own own;
    log_.push_back("sync device " + std::to_string(current));
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode* m) { std::swap(*m, capture_mode); return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }

// ---- memory
cudaError_t cudaMalloc(void** p, size_t bytes)
{
    std::lock_guard<std::recursive_mutex> g(lock);
    const Own own;
    if (unsafe()) return invalidates();
    if (bytes > limit[current] || live[current] + bytes > limit[current]) { ++refused; return fail(cudaErrorMemoryAllocation); }
    char* q = (char*)calloc(bytes ? bytes : 1, 1);
    if (!q) return fail(cudaErrorMemoryAllocation);
    blocks[q] = {bytes, current};
    live[current] += bytes;
    ++mallocs;
    *p = q;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p)
{
    std::lock_guard<std::recursive_mutex> g(lock);
    const Own own;
    if (!p) return cudaSuccess;
    if (unsafe()) return invalidates();
    auto it = blocks.find((char*)p);
    if (it == blocks.end()) return bad();
    live[it->second.device] -= it->second.bytes;
    ++frees;
    free(p);
    blocks.erase(it);
    return cudaSuccess;
}
// (not zeroed, like the real one)
cudaError_t cudaMallocHost(void** p, size_t bytes)
{
    *p = malloc(bytes);
    memset(*p, 0x7f, bytes);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t bytes, cudaMemcpyKind, cudaStream_t s)
{
    if (s && ((Stream*)s)->device != current) return bad();
    memcpy(dst, src, bytes);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t bytes) { memset(p, v, bytes); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t bytes, cudaStream_t) { memset(p, v, bytes); return cudaSuccess; }

// ---- streams and events
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { const Own own; *s = (cudaStream_t) new Stream{current}; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { delete (Stream*)s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s)
{
    if (captured && (s == captured || unsafe())) return invalidates();
    const Own own;
    char t[64];
    snprintf(t, sizeof t, "sync stream %p", (void*)s);
    log_.push_back(t);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned)
{
    const Own own;
    char t[64];
    snprintf(t, sizeof t, "wait stream %p", (void*)s);
    log_.push_back(t);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { const Own own; *e = (cudaEvent_t) new Event{current}; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete (Event*)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    // an event can be recorded only in a stream of its device (the default stream is the current device's)
    if (((Event*)e)->device != (s ? ((Stream*)s)->device : current)) return bad();
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { const Own own; log_.push_back("sync event"); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st)
{
    *st = captured && s == captured ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.0f; return cudaSuccess; }

// ---- kernels
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return fail(cudaErrorInvalidSymbol); }
cudaError_t cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* r)
{
    *fn = nullptr;
    if (r) *r = cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void** args, size_t, cudaStream_t s)
{
    std::lock_guard<std::recursive_mutex> g(lock);
    const Own own;
    if (s && ((Stream*)s)->device != current) return bad();
    const std::string& name = kernels()[f];
    auto is = [&](const char* what) { return name.find(what) != std::string::npos; };
    log_.push_back("launch " + name + (captured && s != captured ? " beside" : ""));
    if (is("edge_records_kernel")) {
        if (*(int64_t*)args[1] > 0 && device_of(*(void**)args[6]) != current) ++errors;     // the room for the records
        if (report[4] > *(int64_t*)args[1]) **(int32_t**)args[9] = (int32_t)report[4];
    } else if (is("scan_direct_kernel")) {
        const grf_scan_jobs& j = *(const grf_scan_jobs*)args[0];
        for (int x = 0; x < 3; ++x) {
            const int32_t n = *(int32_t*)args[1];
            if (j.job[x].out) j.job[x].out[n] = (int32_t)report[x > 1 ? 1 : x];
            if (j.job[x].host_total) *j.job[x].host_total = (int32_t)report[x];
        }
    } else if (is("gather_denominators_kernel")) {
        denominators = *(void**)args[7];
    } else if (is("block_plan_kernel")) {
        **(int32_t**)args[7] = (int32_t)report[5];
    } else if (is("mask_structure_kernel")) {
        int32_t* host = *(int32_t**)args[20];
        host[0] = (int32_t)report[6]; host[1] = (int32_t)report[7]; host[2] = (int32_t)report[8];
    }
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args)
{
    return cudaLaunchKernel(f, c->gridDim, c->blockDim, args, c->dynamicSmemBytes, c->stream);
}
static thread_local struct { dim3 g, b; size_t smem; void* s; } config;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void* s) { config = {g, b, smem, s}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s)
{
    *g = config.g; *b = config.b; *smem = config.smem; *(void**)s = config.s;
    return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* stub, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*)
{
    kernels()[stub] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}

}  // extern "C"
