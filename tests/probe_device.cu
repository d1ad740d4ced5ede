// Kernels that call the library's device functions by themselves
// (test_gpu_device_parts.py compiles and loads this file).  Every entry returns the
// launch's error; pointers are device pointers.
#include "ir_kernel.cuh"

using namespace spai;

namespace {

cudaError_t finish() { return cudaGetLastError() != cudaSuccess ? cudaErrorLaunchFailure : cudaDeviceSynchronize(); }

// out = M x of one block's rows; `most` entries before the 64-bit loop takes over
template <class T, int64_t MOST>
__global__ void k_sell(int rows, const int64_t* soff, const int32_t* col, const T* val, const T* x, T* out)
{
    sell_mul_direct<false, MOST>(rows, soff, col, val, XIn<T, T, LD_PLAIN>{x, T(0), T(0), 0}, out);
}

template <class T>
int sell(int rows, bool wide, const int64_t* soff, const int32_t* col, const void* val, const void* x, void* out)
{
    if (wide) k_sell<T, 0><<<1, 256>>>(rows, soff, col, (const T*)val, (const T*)x, (T*)out);
    else k_sell<T, SELL_INT><<<1, 256>>>(rows, soff, col, (const T*)val, (const T*)x, (T*)out);
    return finish();
}

}  // namespace

extern "C" int probe_sell(int dbl, int rows, int wide, const int64_t* soff, const int32_t* col, const void* val,
                          const void* x, void* out)
{
    return dbl ? sell<double>(rows, wide, soff, col, val, x, out) : sell<float>(rows, wide, soff, col, val, x, out);
}

extern "C" int64_t probe_sell_int() { return SELL_INT; }
