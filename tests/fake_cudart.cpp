// fake_cudart.cpp -- a CUDA runtime for tests of the library's host code without a GPU: memory is the
// host's, copies happen at once, kernels do not run.  Every call that orders or changes work is written
// to a log ("<call> <stream> ..."), and the n-th call of a name can be made to fail.
#include <cuda_runtime_api.h>
#include <sys/mman.h>

#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {

std::string g_log;
std::map<const void*, std::string> g_names;  // host stub -> kernel
std::map<void*, size_t> g_sizes;              // allocations
std::string g_fail_call;
int g_fail_nth = 0;
cudaError_t g_fail_code = cudaSuccess, g_last = cudaSuccess;
size_t g_next = 1, g_limit = 0;  // handles; largest allocation allowed (0: any)

void say(const char* fmt, ...)
{
    char line[512];
    va_list a;
    va_start(a, fmt);
    vsnprintf(line, sizeof line, fmt, a);
    va_end(a);
    g_log += line;
    g_log += '\n';
}

// The status of a call: success, or the failure asked for.
cudaError_t done(const char* call)
{
    if (g_fail_nth > 0 && g_fail_call == call && --g_fail_nth == 0) {
        say("FAIL %s", call);
        return g_last = g_fail_code;
    }
    return cudaSuccess;
}

size_t id(const void* p) { return (size_t)p; }

cudaError_t launch(const void* func, dim3 grid, cudaStream_t st)
{
    const cudaError_t e = done("launch");
    const char* name = g_names.count(func) ? g_names[func].c_str() : "?";
    if (e == cudaSuccess) say("launch %zu %s %zu", id(st), name, (size_t)grid.x * grid.y * grid.z);
    return e;
}

}  // namespace

extern "C" {

const char* fake_log() { return g_log.c_str(); }
void fake_reset() { g_log.clear(), g_fail_nth = 0, g_last = cudaSuccess, g_limit = 0; }
void fake_fail(const char* call, int nth, int code)
{
    g_fail_call = call, g_fail_nth = nth, g_fail_code = (cudaError_t)code;
}
void fake_limit(size_t bytes) { g_limit = bytes; }
static int g_device = 0;
void fake_device(int device) { g_device = device; }

// ------------------------------------------------------------ kernels
void** __cudaRegisterFatBinary(void*)
{
    static void* h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* stub, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*)
{
    g_names[stub] = name;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* stub) { return *k = (cudaKernel_t)stub, cudaSuccess; }
static thread_local struct {
    dim3 grid, block;
    size_t smem;
    cudaStream_t st;
} t_config;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t st)
{
    t_config = {grid, block, smem, st};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* st)
{
    *grid = t_config.grid, *block = t_config.block, *smem = t_config.smem, *(cudaStream_t*)st = t_config.st;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void**, size_t, cudaStream_t st)
{
    return launch((const void*)k, grid, st);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**)
{
    return launch(f, c->gridDim, c->stream);
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t)
{
    return *n = 2, cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned)
{
    return *n = 2, cudaSuccess;
}

// ------------------------------------------------------------- memory
static cudaError_t get(const char* call, void** p, size_t n)
{
    const cudaError_t e = done(call);
    if (e != cudaSuccess) return e;
    if (g_limit && n > g_limit) return g_last = cudaErrorMemoryAllocation;
    // zeros, and no memory for what nothing touches (fields of production size)
    *p = mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (*p == MAP_FAILED) return g_last = cudaErrorMemoryAllocation;
    g_sizes[*p] = n;
    say("%s %zu %zu", call, n, id(*p));
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { return get("malloc", p, n); }
cudaError_t cudaMallocHost(void** p, size_t n) { return get("mallochost", p, n); }
cudaError_t cudaFree(void* p)
{
    if (p) say("free");
    return cudaFreeHost(p);
}
cudaError_t cudaFreeHost(void* p)
{
    if (p) munmap(p, g_sizes[p]), g_sizes.erase(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st)
{
    const cudaError_t e = done("copy");
    if (e != cudaSuccess) return e;
    memmove(d, s, n);
    say("copy %zu %zu", id(st), n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return memmove(d, s, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st)
{
    const cudaError_t e = done("memset");
    if (e != cudaSuccess) return e;
    memset(d, v, n);
    say("memset %zu %zu", id(st), n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { return memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { return *f = *t = (size_t)1 << 38, cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*)
{
    static char array[4 << 20];
    return *p = array, cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes*, const void*) { return g_last = cudaErrorInvalidValue; }

// -------------------------------------------------- streams and events
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned)
{
    const cudaError_t e = done("stream");
    if (e == cudaSuccess) *s = (cudaStream_t)(0x1000 + g_next++);
    return e;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s)
{
    return *s = cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t st)
{
    const cudaError_t e = done("sync");
    if (e == cudaSuccess) say("sync %zu", id(st));
    return e;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* v, unsigned)
{
    const cudaError_t e = done("event");
    if (e == cudaSuccess) *v = (cudaEvent_t)(0x100000 + g_next++);
    return e;
}
cudaError_t cudaEventCreate(cudaEvent_t* v) { return cudaEventCreateWithFlags(v, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t v, cudaStream_t st)
{
    const cudaError_t e = done("record");
    if (e == cudaSuccess) say("record %zu %zu", id(st), id(v));
    return e;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t v, unsigned)
{
    const cudaError_t e = done("wait");
    if (e == cudaSuccess) say("wait %zu %zu", id(st), id(v));
    return e;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }

// -------------------------------------------------------------- others
cudaError_t cudaGetDevice(int* d) { return *d = g_device, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
static int encode_nothing() { return 0; }  // the tensor-map encoder
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q)
{
    const bool have = !strcmp(name, "cuTensorMapEncodeTiled");
    *f = have ? (void*)encode_nothing : nullptr;
    *q = have ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaGetLastError()
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t) { return "fake"; }

}  // extern "C"
