// A CUDA runtime without a GPU, for tests of the library's host code: the
// functions its translation units call, over host memory.  Allocations are
// zeroed host memory, copies and memsets are done at once, and a kernel launch
// does nothing; every call that orders work, launches, allocates or frees is
// written to a log that the test reads.  Devices, failures and page-locked
// ranges are whatever the test sets.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#undef cudaGetDriverEntryPointByVersion

namespace {

struct Range {
    size_t bytes;
};
struct Fault {
    int after, code;  // the call after `after` more returns code; every call when after < 0
};
std::recursive_mutex mu;
std::string lines;
std::map<std::string, Fault> faults;
std::map<const void*, std::string> kernels;
std::map<char*, Range> locked;               // page-locked host ranges
std::map<void*, std::pair<size_t, int>> live;  // device allocations: bytes, 1 when from a pool
std::map<std::string, int> peers;            // "a b": a can reach b
int n_devices = 1;
thread_local int device = 0;
thread_local cudaError_t last = cudaSuccess;
size_t used = 0, reserved = 0, threshold = 0;
bool later = false;                          // frees on a stream take effect when something waits
std::vector<void*> freed;
int streams = 0;

void log(const char* fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    std::lock_guard<std::recursive_mutex> lk(mu);
    lines += buf;
    lines += '\n';
}

cudaError_t result(const char* fn)
{
    std::lock_guard<std::recursive_mutex> lk(mu);
    auto f = faults.find(fn);
    if (f == faults.end()) return cudaSuccess;
    const int code = f->second.code;
    if (f->second.after >= 0) {
        if (f->second.after-- > 0) return cudaSuccess;
        faults.erase(f);
    }
    log("%s fails", fn);
    return last = (cudaError_t)code;
}

cudaError_t take(void** p, size_t bytes, int pool)
{
    *p = calloc(bytes ? bytes : 1, 1);
    std::lock_guard<std::recursive_mutex> lk(mu);
    live[*p] = {bytes, pool};
    if (pool) {
        used += bytes;
        if (reserved < used) reserved = used;
    }
    return cudaSuccess;
}

void give(void* p)
{
    std::lock_guard<std::recursive_mutex> lk(mu);
    auto it = live.find(p);
    if (it == live.end()) { log("free of what is not allocated"); return; }
    if (it->second.second) used -= it->second.first;
    live.erase(it);
    free(p);
}

// a wait: what was freed on a stream is free, and the pool keeps its threshold
void waited()
{
    std::lock_guard<std::recursive_mutex> lk(mu);
    for (void* p : freed) give(p);
    freed.clear();
    const size_t keep = threshold > used ? threshold : used;
    if (reserved > keep) reserved = keep;
}

std::map<char*, Range>::iterator range_of(const void* p)
{
    auto it = locked.upper_bound((char*)p);
    if (it == locked.begin()) return locked.end();
    --it;
    return (char*)p < it->first + it->second.bytes ? it : locked.end();
}

CUresult pointer_attribute(void* data, CUpointer_attribute what, CUdeviceptr p)
{
    std::lock_guard<std::recursive_mutex> lk(mu);
    auto it = range_of((const void*)p);
    if (it == locked.end()) return CUDA_ERROR_INVALID_VALUE;
    if (what == CU_POINTER_ATTRIBUTE_RANGE_START_ADDR) *(CUdeviceptr*)data = (CUdeviceptr)it->first;
    else if (what == CU_POINTER_ATTRIBUTE_RANGE_SIZE) *(size_t*)data = it->second.bytes;
    else return CUDA_ERROR_NOT_SUPPORTED;
    return CUDA_SUCCESS;
}

const char* name_of(const void* f)
{
    auto it = kernels.find(f);
    return it == kernels.end() ? "?" : it->second.c_str();
}

}  // namespace

// ---- what a test sets and reads --------------------------------------------
extern "C" {
void fake_reset(int devices)
{
    std::lock_guard<std::recursive_mutex> lk(mu);
    lines.clear();
    faults.clear();
    locked.clear();
    peers.clear();
    n_devices = devices;
    device = 0;
    last = cudaSuccess;
}
const char* fake_log() { return lines.c_str(); }
void fake_clear() { lines.clear(); }
void fake_fail(const char* fn, int after, int code) { faults[fn] = {after, code}; }
void fake_lock(void* p, size_t bytes) { locked[(char*)p] = {bytes}; }
void fake_peer(int a, int b) { peers[std::to_string(a) + " " + std::to_string(b)] = 1; }
void fake_free_later(int on) { later = on; }
long long fake_live() { return (long long)live.size(); }
long long fake_reserved() { return (long long)reserved; }

// ---- devices, errors ---------------------------------------------------------
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d)
{
    if (d < 0 || d >= n_devices) return last = cudaErrorInvalidDevice;
    device = d;
    return result("cudaSetDevice");
}
cudaError_t cudaGetDeviceCount(int* n) { *n = n_devices; return cudaSuccess; }
cudaError_t cudaDeviceCanAccessPeer(int* can, int a, int b)
{
    *can = peers.count(std::to_string(a) + " " + std::to_string(b)) ? 1 : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrL2CacheSize ? 129 << 20 : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetLimit(size_t* v, cudaLimit) { *v = 0; return cudaSuccess; }
cudaError_t cudaDeviceSetLimit(cudaLimit, size_t) { return cudaSuccess; }
cudaError_t cudaCtxResetPersistingL2Cache() { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize()
{
    log("device %d synchronize", device);
    waited();
    return result("cudaDeviceSynchronize");
}
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorName(cudaError_t) { return "error"; }
const char* cudaGetErrorString(cudaError_t) { return "an error of the fake runtime"; }

// ---- memory --------------------------------------------------------------------
cudaError_t cudaMalloc(void** p, size_t bytes)
{
    const cudaError_t e = result("cudaMalloc");
    return e == cudaSuccess ? take(p, bytes, 0) : e;
}
cudaError_t cudaFree(void* p) { log("device %d cudaFree", device); give(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t bytes)
{
    const cudaError_t e = result("cudaMallocHost");
    if (e == cudaSuccess) *p = calloc(bytes, 1);
    return e;
}
cudaError_t cudaMallocAsync(void** p, size_t bytes, cudaStream_t)
{
    const cudaError_t e = result("cudaMallocAsync");
    return e == cudaSuccess ? take(p, bytes, 0) : e;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t bytes, cudaMemPool_t, cudaStream_t)
{
    const cudaError_t e = result("cudaMallocFromPoolAsync");
    return e == cudaSuccess ? take(p, bytes, 1) : e;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t s) 
{
    log("free %p on stream %zx", p, (size_t)s);
    if (later) freed.push_back(p);
    else give(p);
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps* props)
{
    *p = (cudaMemPool_t)(size_t)(0x100 + props->location.id);
    log("pool of device %d", props->location.id);
    return result("cudaMemPoolCreate");
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAccess(cudaMemPool_t p, const cudaMemAccessDesc* d, size_t n)
{
    for (size_t i = 0; i < n; ++i)
        log("pool of device %d open to device %d", (int)(size_t)p - 0x100, d[i].flags == cudaMemAccessFlagsProtReadWrite ? d[i].location.id : -1);
    return result("cudaMemPoolSetAccess");
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr a, void* v)
{
    if (a == cudaMemPoolAttrReleaseThreshold) threshold = *(uint64_t*)v;
    return cudaSuccess;
}
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr a, void* v)
{
    *(uint64_t*)v = a == cudaMemPoolAttrUsedMemCurrent ? used : reserved;
    return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t keep)
{
    log("trim to %zu", keep);
    if (reserved > keep) reserved = keep > used ? keep : used;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t)
{
    log("copy %s %zu", k == cudaMemcpyHostToDevice ? "up" : k == cudaMemcpyDeviceToHost ? "down" : "across", n);
    memcpy(d, s, n);
    return result("cudaMemcpyAsync");
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t)
{
    memset(d, v, n);
    return result("cudaMemsetAsync");
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p)
{
    *a = cudaPointerAttributes{};
    a->type = range_of(p) == locked.end() ? cudaMemoryTypeUnregistered : cudaMemoryTypeHost;
    if (a->type == cudaMemoryTypeHost) a->devicePointer = a->hostPointer = (void*)p;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* found)
{
    const bool known = strcmp(name, "cuPointerGetAttribute") == 0;
    *f = known ? (void*)pointer_attribute : nullptr;
    if (found) *found = known ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}

// ---- streams, events, graphs ------------------------------------------------------
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned)
{
    *s = (cudaStream_t)(size_t)(0x1000 + ++streams);
    log("stream %zx on device %d", (size_t)*s, device);
    return result("cudaStreamCreateWithFlags");
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s)
{
    log("stream %zx synchronize", (size_t)s);
    waited();
    return result("cudaStreamSynchronize");
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { log("begin capture"); return result("cudaStreamBeginCapture"); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = (cudaGraph_t)1; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) { *x = (cudaGraphExec_t)1; return result("cudaGraphInstantiate"); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { log("graph launch"); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }

// ---- kernels ------------------------------------------------------------------------
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*)
{
    // the identifier inside the mangled name
    const char* k = strstr(name, "k_");
    kernels[host] = k ? std::string(k, strspn(k, "abcdefghijklmnopqrstuvwxyz0123456789_")) : name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) { *k = (cudaKernel_t)host; return cudaSuccess; }
thread_local dim3 cfg_grid, cfg_block;
thread_local size_t cfg_smem;
thread_local void* cfg_stream;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, void* s) { cfg_grid = g; cfg_block = b; cfg_smem = m; cfg_stream = s; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s)
{
    *g = cfg_grid; *b = cfg_block; *m = cfg_smem; *(void**)s = cfg_stream;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t s)
{
    log("kernel %s on stream %zx", name_of(k), (size_t)s);
    return result("launch");
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**)
{
    log("kernel %s on stream %zx", name_of(f), (size_t)c->stream);
    return result("launch");
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t s)
{
    const cudaError_t e = result("cudaLaunchCooperativeKernel");
    if (e == cudaSuccess) log("kernel %s on stream %zx", name_of(f), (size_t)s);
    return e;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { static char mem[256]; *p = mem; return cudaSuccess; }
}
