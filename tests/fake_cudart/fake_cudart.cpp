// fake_cudart.cpp -- a CUDA runtime without a GPU, for tests of the library's host code: device memory is
// host memory, launches run nothing and are recorded, and what a launch needs (a kernel's shared
// memory limit and cluster permission, per device) is enforced as the runtime does.  Loaded with
// global visibility before the library.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <utility>

namespace {
std::recursive_mutex mu;   // recursive: a launch looks attributes up under it
std::map<const void*, std::string> names;
std::map<std::pair<int, const void*>, std::map<int, int>> attrs;   // (device, kernel) -> attribute -> value
std::string launches;
thread_local int device = 0;
thread_local cudaError_t last = cudaSuccess;
thread_local dim3 cfg_grid, cfg_block;
thread_local size_t cfg_smem;
thread_local void* cfg_stream;
int ctas_per_sm = 7, clusters = 1, capturing = 0, fail_next = 0, sms = 152, l2_kb = 129 << 10;
float event_ms = 1.0f;

cudaError_t fail(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}

cudaError_t launch(const void* func, dim3 g, dim3 b, size_t smem, bool chained, unsigned cluster) {
    std::lock_guard<std::recursive_mutex> l(mu);
    if (fail_next != 0) {
        const cudaError_t e = (cudaError_t)fail_next;
        fail_next = 0;
        return fail(e);
    }
    auto& a = attrs[{device, func}];
    if (g.x == 0 || g.y == 0 || g.z == 0) return fail(cudaErrorInvalidConfiguration);
    if (smem > 48 * 1024 && a[cudaFuncAttributeMaxDynamicSharedMemorySize] < (int)smem) return fail(cudaErrorInvalidValue);
    if (cluster > 8 && !a[cudaFuncAttributeNonPortableClusterSizeAllowed]) return fail(cudaErrorInvalidClusterSize);
    char line[1024];
    std::snprintf(line, sizeof(line), "%d %s %u %u %u %u %zu %d %u\n", device, names[func].c_str(), g.x, g.y, g.z, b.x, smem,
                  chained ? 1 : 0, cluster);
    launches += line;
    return cudaSuccess;
}
int encode_tiled(...) { return 0; }
}  // namespace

extern "C" {
// ---- what the tests set and read
void fake_device(int d) { device = d; }
void fake_set(const char* what, int v) {
    if (!std::strcmp(what, "ctas_per_sm")) ctas_per_sm = v;
    else if (!std::strcmp(what, "clusters")) clusters = v;
    else if (!std::strcmp(what, "capturing")) capturing = v;
    else if (!std::strcmp(what, "fail_next")) fail_next = v;
    else if (!std::strcmp(what, "sms")) sms = v;
    else if (!std::strcmp(what, "l2_kb")) l2_kb = v;
}
void fake_clear() { launches.clear(); }
const char* fake_launches() { return launches.c_str(); }

// ---- registration and launches
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
    names[host] = name;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void* st) {
    cfg_grid = g; cfg_block = b; cfg_smem = s; cfg_stream = st;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
    *g = cfg_grid; *b = cfg_block; *s = cfg_smem; *(void**)st = cfg_stream;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t smem, cudaStream_t) {
    return launch((const void*)k, g, b, smem, false, 1);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* func, void**) {
    bool chained = false;
    unsigned cluster = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i) {
        if (c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization)
            chained = c->attrs[i].val.programmaticStreamSerializationAllowed != 0;
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[i].val.clusterDim.x;
    }
    return launch(func, c->gridDim, c->blockDim, c->dynamicSmemBytes, chained, cluster);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute at, int v) {
    std::lock_guard<std::recursive_mutex> l(mu);
    attrs[{device, f}][at] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = ctas_per_sm;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { *n = clusters; return cudaSuccess; }

// ---- device
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? sms : a == cudaDevAttrL2CacheSize ? l2_kb << 10 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) { std::memset(p, 0, sizeof(*p)); std::strcpy(p->name, "fake"); return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t e) { static thread_local char s[32]; std::snprintf(s, sizeof(s), "error %d", (int)e); return s; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q) {
    *f = (void*)&encode_tiled;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) { static char mem[1 << 20]; *p = mem; return cudaSuccess; }

// ---- memory
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::calloc(n ? n : 1, 1); return *p ? cudaSuccess : fail(cudaErrorMemoryAllocation); }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { *p = (cudaMemPool_t)1; return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
    std::memset(a, 0, sizeof(*a));
    a->type = cudaMemoryTypeUnregistered;
    return cudaSuccess;
}

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)1; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = (cudaGraph_t)1; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = event_ms; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) { *x = (cudaGraphExec_t)1; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
}
