// A stand-in for the CUDA runtime, linked with the library's own objects: "device"
// memory is host memory and no kernel runs, so the host side (tables, copies, launch
// choices, errors) can be followed without a GPU.  A copy from host memory is due at
// the next wait, and until then its source has to keep its contents.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace {

struct Copy {
    const void* src;
    void* dst;
    std::string data;
};
std::vector<Copy> pending;
std::mutex mu;  // of `pending`
std::map<std::string, long long> vals = {{"cluster_max", 16}, {"cluster_error", 0}};
int device_tag, stream_tag;
cudaError_t last = cudaSuccess;

cudaError_t fail(cudaError_t e)
{
    last = e;
    return e;
}

cudaError_t wait_all()
{
    std::lock_guard<std::mutex> lk(mu);
    for (const Copy& c : pending) {
        if (memcmp(c.src, c.data.data(), c.data.size())) vals["stale_copies"]++;
        memcpy(c.dst, c.data.data(), c.data.size());
    }
    pending.clear();
    return cudaSuccess;
}

int cluster_of(const cudaLaunchConfig_t* c)
{
    for (unsigned i = 0; i < c->numAttrs; i++)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return (int)c->attrs[i].val.clusterDim.x;
    return 1;
}

cudaError_t alloc(void** p, size_t n)
{
    *p = calloc(1, n ? n : 1);
    return *p ? cudaSuccess : fail(cudaErrorMemoryAllocation);
}

}  // namespace

extern "C" {

void fake_set(const char* k, long long v) { vals[k] = v; }
long long fake_get(const char* k) { return vals[k]; }

// compiler glue: a launch configuration that is refused skips its kernel
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t)
{
    vals["launches"]++;
    return 1;
}
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaErrorInvalidConfiguration; }
cudaError_t __cudaGetKernel(cudaKernel_t*, const void*) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**)
{
    const int t = cluster_of(c);
    if (t > vals["cluster_max"]) return fail(cudaErrorInvalidClusterSize);
    if (vals["cluster_error"]) return fail((cudaError_t)vals["cluster_error"]);
    vals["cluster_launches"]++;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c)
{
    *n = cluster_of(c) <= vals["cluster_max"] ? 1 : 0;
    return cudaSuccess;
}
cudaError_t cudaLaunchCooperativeKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t)
{
    vals["grid_launches"]++;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t)
{
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned)
{
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*)
{
    memset(a, 0, sizeof(*a));
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }

cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount ? 152
         : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448
         : a == cudaDevAttrClockRate ? 2000000 : 1;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError()
{
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char* cudaGetErrorName(cudaError_t) { return "fake"; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }

cudaError_t cudaMalloc(void** p, size_t n) { return alloc(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return alloc(p, n); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return alloc(p, n); }
// (kept: a copy may still be due to a freed block, whose stream orders the two)
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaFreeAsync(void*, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { return *f = *t = (size_t)1 << 33, cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { return *p = (cudaMemPool_t)&device_tag, cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return alloc(p, (size_t)1 << 30); }

cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind kind, cudaStream_t)
{
    std::lock_guard<std::mutex> lk(mu);
    if (kind == cudaMemcpyHostToDevice) pending.push_back(Copy{src, dst, std::string((const char*)src, n)});
    else memcpy(dst, src, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* dst, const void* src, size_t n, cudaMemcpyKind)
{
    wait_all();
    memcpy(dst, src, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { return memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { return memset(p, v, n), cudaSuccess; }

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = (cudaStream_t)&stream_tag, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return wait_all(); }
cudaError_t cudaDeviceSynchronize() { return wait_all(); }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)&stream_tag, cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = (cudaEvent_t)&stream_tag, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return wait_all(); }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 0.f, cudaSuccess; }

}  // extern "C"
