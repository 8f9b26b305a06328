// fake_cudart.cpp -- the CUDA runtime calls libsfft makes, on the host alone: device memory is reserved
// address space, copies and clears act at once, launches run nothing.  Every call that orders work is
// written to a log ("launch <kernel> <stream>", "record <event> <stream>", "wait <stream> <event>"), a chosen
// launch can be made to fail, and a callback can stand in for what a kernel writes.  The library's own
// objects are linked against it, so the host code under test is the one that ships.
#include <cuda_runtime.h>
#include <sys/mman.h>

#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {
std::string g_log;
std::map<const void*, size_t> g_allocs;
size_t g_bytes = 0, g_memory = size_t(1) << 38;
int g_fail_launch = -1;
std::map<const void*, std::string>& names() {  // filled while the library's own objects are initialised
    static std::map<const void*, std::string> m;
    return m;
}
uintptr_t g_handles = 0;
cudaError_t g_last = cudaSuccess;
using LaunchFn = void (*)(const char* kernel, void** args);
LaunchFn g_on_launch = nullptr;
struct Config {
    dim3 grid, block;
    size_t smem = 0;
    void* stream = nullptr;
} g_config;

void note(const char* fmt, const void* a, const void* b) {
    char line[64];
    std::snprintf(line, sizeof line, fmt, a, b);
    g_log += line;
}
cudaError_t launch(const void* kernel, void** args, void* stream) {
    const std::string& name = names()[kernel];
    if (g_fail_launch == 0) {
        g_fail_launch = -1;
        return g_last = cudaErrorLaunchOutOfResources;
    }
    if (g_fail_launch > 0) --g_fail_launch;
    g_log += "launch " + name;
    note(" %p%s\n", stream, "");
    if (g_on_launch) g_on_launch(name.c_str(), args);
    return cudaSuccess;
}
}  // namespace

extern "C" {
// the test's side
void fake_reset() {
    g_log.clear();
    g_fail_launch = -1;
    g_on_launch = nullptr;
    g_last = cudaSuccess;
    g_memory = size_t(1) << 38;
}
const char* fake_log() { return g_log.c_str(); }
void fake_fail_launch(int after) { g_fail_launch = after; }  // the launch after that many successful ones
void fake_on_launch(LaunchFn f) { g_on_launch = f; }
size_t fake_bytes() { return g_bytes; }
void fake_memory(size_t bytes) { g_memory = bytes; }  // what the other users of the device leave of 2^38

// kernels
void** __cudaRegisterFatBinary(void*) {
    static void* handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    names()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t st) {
    g_config.grid = grid;
    g_config.block = block;
    g_config.smem = smem;
    g_config.stream = st;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* st) {
    *grid = g_config.grid;
    *block = g_config.block;
    *smem = g_config.smem;
    *static_cast<void**>(st) = g_config.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) {
    *k = (cudaKernel_t)host;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t st) {
    return launch((const void*)k, args, st);
}
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void** args, size_t, cudaStream_t st) { return launch(f, args, st); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) { return launch(f, args, c->stream); }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaLaunchHostFunc(cudaStream_t, cudaHostFn_t, void*) { return cudaSuccess; }

// memory
cudaError_t cudaMalloc(void** p, size_t bytes) {
    if (g_bytes + bytes > g_memory) return g_last = cudaErrorMemoryAllocation;
    *p = mmap(nullptr, bytes ? bytes : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (*p == MAP_FAILED) return g_last = cudaErrorMemoryAllocation;
    g_allocs[*p] = bytes ? bytes : 1;
    g_bytes += bytes;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    auto it = g_allocs.find(p);
    if (it == g_allocs.end()) return cudaSuccess;
    munmap(p, it->second);
    g_bytes -= it->second;
    g_allocs.erase(it);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t bytes) {
    *p = std::calloc(1, bytes ? bytes : 1);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) {
    *f = g_memory - g_bytes;
    *t = size_t(1) << 38;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
    std::memset(a, 0, sizeof *a);
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    *p = nullptr;
    return cudaSuccess;
}

// streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = (cudaStream_t)(++g_handles << 12);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    note("wait %p %p\n", s, e);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    *e = (cudaEvent_t)(++g_handles << 12);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    note("record %p %p\n", e, s);
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 0;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

// device and errors
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceSetLimit(cudaLimit, size_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "a call made to fail"; }
}
