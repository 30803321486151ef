// A stand-in for the CUDA runtime that records calls instead of using a GPU.  Linked with the library's own objects
// in place of the runtime, it lets a test without a GPU run the host code of an entry point and check what it issued:
// the order of the launches and copies on the streams, and the device memory it asked for.  "Device" memory is host
// memory (zeroed); kernels do nothing.
#include <cuda_runtime_api.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>

namespace {
std::map<const void*, std::string> g_kernels;
std::map<void*, size_t> g_live;
size_t g_live_bytes = 0, g_peak_bytes = 0, g_limit = 0;
std::string g_log;
bool g_fill = false;
uint64_t g_word = 0;
uintptr_t g_handle = 0x1000;
struct Call { dim3 grid, block; size_t smem; void* stream; } g_call;

void* handle() { return (void*)(g_handle += 16); }
void log(const char* op, const void* stream, const std::string& what = "-")
{
    g_log += std::string(op) + " " + std::to_string((uintptr_t)stream) + " " + what + "\n";
}
std::string id(const void* p) { return std::to_string((uintptr_t)p); }
cudaError_t launch(const void* fn, const void* stream)
{
    auto it = g_kernels.find(fn);
    log("launch", stream, it == g_kernels.end() ? "unknown" : it->second);
    return it == g_kernels.end() ? cudaErrorInvalidDeviceFunction : cudaSuccess;
}
void copy(void* dst, const void* src, size_t n, cudaMemcpyKind kind)
{
    if (kind == cudaMemcpyDeviceToHost && g_fill)
        for (size_t i = 0; i < n; i++) ((char*)dst)[i] = ((const char*)&g_word)[i % 8];
    else
        memmove(dst, src, n);
}
}  // namespace

extern "C" {
// ------------------------------------------------------------ for the test --
const char* rec_log() { return g_log.c_str(); }
void rec_clear() { g_log.clear(); g_peak_bytes = g_live_bytes; }
unsigned long long rec_live_bytes() { return g_live_bytes; }
unsigned long long rec_peak_bytes() { return g_peak_bytes; }
void rec_set_limit(unsigned long long bytes) { g_limit = bytes; }  // 0: none
void rec_read_words(int on, unsigned long long word)               // copies to the host deliver this 64-bit word
{
    g_fill = on != 0;
    g_word = word;
}

void rec_launch(unsigned long long stream, const char* name) { log("launch", (void*)stream, name); }  // the caller's own

// -------------------------------------------------------------- the runtime --
void** __cudaRegisterFatBinary(void*) { return (void**)handle(); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* fn, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*)
{
    g_kernels[fn] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* stream)
{
    g_call = {grid, block, smem, stream};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream)
{
    *grid = g_call.grid;
    *block = g_call.block;
    *smem = g_call.smem;
    *(void**)stream = g_call.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn)
{
    *k = (cudaKernel_t)fn;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t s) { return launch((const void*)k, s); }
cudaError_t cudaLaunchKernel(const void* fn, dim3, dim3, void**, size_t, cudaStream_t s) { return launch(fn, s); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void**) { return launch(fn, c->stream); }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "recorded"; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*)
{
    memset(a, 0, sizeof(*a));
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol)
{
    *p = (void*)symbol;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceCount(int* n)
{
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d)
{
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int)
{
    memset(p, 0, sizeof(*p));
    strcpy(p->name, "recorded sm_103");
    p->major = 10;
    p->minor = 3;
    p->multiProcessorCount = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int)
{
    *v = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetLimit(size_t* v, cudaLimit)
{
    *v = 1024;
    return cudaSuccess;
}
cudaError_t cudaDeviceSetLimit(cudaLimit, size_t) { return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int* least, int* greatest)
{
    *least = 0;
    *greatest = -5;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n)
{
    if (g_limit && g_live_bytes + n > g_limit) return cudaErrorMemoryAllocation;
    *p = calloc(n, 1);
    if (!*p) return cudaErrorMemoryAllocation;
    g_live[*p] = n;
    g_live_bytes += n;
    if (g_live_bytes > g_peak_bytes) g_peak_bytes = g_live_bytes;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p)
{
    auto it = g_live.find(p);
    if (it == g_live.end()) return cudaErrorInvalidValue;
    g_live_bytes -= it->second;
    g_live.erase(it);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* dst, const void* src, size_t n, cudaMemcpyKind kind)
{
    copy(dst, src, n, kind);
    log("copy", nullptr);
    log("sync", nullptr);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind kind, cudaStream_t s)
{
    copy(dst, src, n, kind);
    log("copy", s);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s)
{
    memset(p, v, n);
    log("set", s);
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned)
{
    *s = (cudaStream_t)handle();
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) { return cudaStreamCreateWithFlags(s, 0); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s)
{
    log("sync", s);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned)
{
    log("wait", s, id(e));
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned)
{
    *e = (cudaEvent_t)handle();
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    log("record", s, id(e));
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e)
{
    log("eventsync", nullptr, id(e));
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t)
{
    *ms = 1.0f;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode)
{
    log("capture", s);
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g)
{
    log("captured", s);
    *g = (cudaGraph_t)handle();
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long)
{
    *x = (cudaGraphExec_t)handle();
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s)
{
    log("graph", s);
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
}
