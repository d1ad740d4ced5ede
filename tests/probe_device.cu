// Kernels that call the library's device functions by themselves
// (test_gpu_device_parts.py compiles and loads this file).  Every entry returns the
// launch's error; pointers are device pointers.
#include "ir_kernel.cuh"

using namespace spai;

namespace {

cudaError_t finish() { return cudaGetLastError() != cudaSuccess ? cudaErrorLaunchFailure : cudaDeviceSynchronize(); }

// out = M x of one block's rows
template <class T, bool WIDE>
__global__ void k_sell(int rows, const int64_t* soff, const int32_t* col, const T* val, const T* x, T* out, bool scat)
{
    sell_mul_direct<WIDE>(rows, soff, col, val, XIn<T, T, LD_PLAIN>{x, T(0), T(0), 0}, out, scat);
}

// the sum of 32 N values by one warp, as each lane has it
template <int N> __global__ void k_wsum(const double* x, double* out)
{
    double v[N];
    for (int k = 0; k < N; k++) v[k] = x[32 * k + threadIdx.x];
    out[threadIdx.x] = warp_sum_fx_n<N>(v);
}
__global__ void k_wsum1(const double* x, double* out) { out[threadIdx.x] = warp_sum_fx(x[threadIdx.x]); }

}  // namespace

extern "C" int probe_wsum(int n, const double* x, double* out)
{
    if (n == 1) k_wsum1<<<1, 32>>>(x, out);
    else if (n == 2) k_wsum<2><<<1, 32>>>(x, out);
    else if (n == 3) k_wsum<3><<<1, 32>>>(x, out);
    else if (n == 5) k_wsum<5><<<1, 32>>>(x, out);
    else k_wsum<8><<<1, 32>>>(x, out);
    return finish();
}

extern "C" int probe_sell(int dbl, int rows, const int64_t* soff, const int32_t* col, const void* val, const void* x,
                          void* out, int scat, int wide)
{
    if (dbl && wide) k_sell<double, true><<<1, 256>>>(rows, soff, col, (const double*)val, (const double*)x, (double*)out, scat);
    else if (dbl) k_sell<double, false><<<1, 256>>>(rows, soff, col, (const double*)val, (const double*)x, (double*)out, scat);
    else if (wide) k_sell<float, true><<<1, 256>>>(rows, soff, col, (const float*)val, (const float*)x, (float*)out, scat);
    else k_sell<float, false><<<1, 256>>>(rows, soff, col, (const float*)val, (const float*)x, (float*)out, scat);
    return finish();
}

// one lane's sum of cnt values and the tree of 16, as the sums over blocks use them
static __global__ void k_lane_sum(int cnt, const float* x, float* out)
{
    float t[16];
    for (int w = 0; w < 16; w++) t[w] = strided_sum<12, float>(cnt, [&](int k) { return x[w * cnt + k]; });
    *out = tree_sum(t);
}
extern "C" int probe_lane_sum(int cnt, const float* x, float* out)
{
    k_lane_sum<<<1, 1>>>(cnt, x, out);
    return finish();
}

// one thread's sum of squares in turn
static __global__ void k_turns(int cnt, const float* x, float* out)
{
    float a = 0.f, b = 0.f;
    for (int i = 0; i < cnt; i++) {
        a = fmaf(x[i], x[i], a);
        in_turn(a, b);
    }
    *out = both(a, b);
}
extern "C" int probe_turns(int cnt, const float* x, float* out)
{
    k_turns<<<1, 1>>>(cnt, x, out);
    return finish();
}

// x / d as the owner of a vector forms it (own) and as a product's input (read)
template <class T> static __global__ void k_quot(int n, const T* x, T d, T* own, T* read, int* fast)
{
    const Quot<T> qd(d);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        own[i] = qd(x[i]);
        read[i] = qd.fast ? XIn<T, T, LD_QUOT>{x, d, qd.y, 0}.of(x[i]) : XIn<T, T, LD_DIV>{x, d, qd.y, 0}.of(x[i]);
    }
    *fast = qd.fast;
}
extern "C" int probe_quot(int dbl, int n, const void* x, double d, void* own, void* read, int* fast)
{
    if (dbl) k_quot<double><<<1, 256>>>(n, (const double*)x, d, (double*)own, (double*)read, fast);
    else k_quot<float><<<1, 256>>>(n, (const float*)x, (float)d, (float*)own, (float*)read, fast);
    return finish();
}
