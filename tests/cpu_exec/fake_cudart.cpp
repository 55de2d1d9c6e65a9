// fake_cudart.cpp -- TEST-ONLY stand-in for the CUDA runtime, so that the host
// side of the library (what it copies when, what it allocates and gives back,
// what it does with errors) runs on a machine without a GPU.  Linked with the
// library's own objects in place of libcudart, never part of libsp.so.
//
// Device memory is host memory with a capacity; kernels do nothing; an
// asynchronous copy or fill is carried out when its stream is waited for (or a
// blocking call is made) and not before, which is the latest that CUDA allows.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <vector>

namespace {

struct Op {
    char *dst;
    const char *src;  // null: fill
    int value;
    size_t bytes;
};

size_t g_capacity, g_used, g_peak;
bool g_deferred;
unsigned g_refused_cluster;  // occupancy queries of clusters this large fail (0: none)
cudaError_t g_last;
std::map<void *, size_t> g_mem;
std::vector<Op> g_ops, g_done;

cudaError_t result(cudaError_t e)
{
    if (e != cudaSuccess) g_last = e;
    return e;
}

void run(const Op &o)
{
    if (o.src)
        std::memcpy(o.dst, o.src, o.bytes);
    else
        std::memset(o.dst, o.value, o.bytes);
    g_done.push_back(o);
}

void drain()
{
    for (const Op &o : g_ops) run(o);
    g_ops.clear();
}

void enqueue(const Op &o)
{
    if (g_deferred)
        g_ops.push_back(o);
    else
        run(o);
}

}  // namespace

extern "C" {

// ---- control ----
void fake_reset(size_t capacity, int deferred, unsigned refused_cluster)
{
    g_capacity = capacity, g_deferred = deferred != 0, g_refused_cluster = refused_cluster, g_last = cudaSuccess;
    g_peak = g_used;
    g_done.clear();
}
size_t fake_used() { return g_used; }
size_t fake_peak() { return g_peak; }
void fake_set_capacity(size_t capacity) { g_capacity = capacity; }
// Destinations of the copies and fills of exactly `bytes` bytes so far, in order.
int fake_copies(size_t bytes, void **dst, int max)
{
    int n = 0;
    for (const Op &o : g_done)
        if (o.src && o.bytes == bytes && n < max) dst[n++] = o.dst;
    return n;
}

// ---- memory ----
cudaError_t cudaMalloc(void **p, size_t bytes)
{
    if (g_used + bytes > g_capacity) return result(cudaErrorMemoryAllocation);
    *p = std::aligned_alloc(256, (bytes + 255) & ~(size_t)255);
    if (!*p) return result(cudaErrorMemoryAllocation);
    g_mem[*p] = bytes;
    g_used += bytes;
    g_peak = g_used > g_peak ? g_used : g_peak;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    if (!p) return cudaSuccess;
    const auto it = g_mem.find(p);
    if (it == g_mem.end()) return result(cudaErrorInvalidValue);
    drain();
    g_used -= it->second;
    g_mem.erase(it);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t *free_b, size_t *total_b)
{
    *free_b = g_capacity > g_used ? g_capacity - g_used : 0, *total_b = g_capacity;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t bytes, enum cudaMemcpyKind, cudaStream_t)
{
    enqueue({(char *)dst, (const char *)src, 0, bytes});
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *dst, const void *src, size_t bytes, enum cudaMemcpyKind)
{
    drain();
    run({(char *)dst, (const char *)src, 0, bytes});
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *dst, int value, size_t bytes, cudaStream_t)
{
    enqueue({(char *)dst, nullptr, value, bytes});
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *)
{
    static char scratch[1 << 24];
    *p = scratch;
    return cudaSuccess;
}

// ---- streams, events, graphs ----
cudaError_t cudaStreamSynchronize(cudaStream_t) { return drain(), cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, enum cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { return *g = nullptr, cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long)
{
    return *e = (cudaGraphExec_t)(uintptr_t)16, cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return *e = (cudaEvent_t)(uintptr_t)16, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return drain(), cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }

// ---- device, functions, errors ----
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes *a, const void *)
{
    std::memset(a, 0, sizeof *a);
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, enum cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) { return *n = 1, cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned)
{
    return *n = 1, cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *c)
{
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension && g_refused_cluster &&
            c->attrs[i].val.clusterDim.x >= g_refused_cluster)
            return *n = 0, result(cudaErrorInvalidValue);
    return *n = 4, cudaSuccess;
}
cudaError_t cudaGetLastError(void)
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}

// ---- launches (arguments ignored) ----
cudaError_t cudaLaunchKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) { return cudaSuccess; }
int __cudaGetKernel() { return 0; }
int __cudaLaunchKernel() { return 0; }
unsigned __cudaPushCallConfiguration() { return 0; }
int __cudaPopCallConfiguration() { return 0; }
void **__cudaRegisterFatBinary(void *)
{
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd() {}
void __cudaRegisterFunction() {}
void __cudaRegisterVar() {}
void __cudaUnregisterFatBinary() {}

}  // extern "C"
