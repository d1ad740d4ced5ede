// Device-side building blocks shared by the SPAI and GMRES-IR kernels:
// precision storage types, warp/block reductions, double-double arithmetic
// and a bounded grid-wide barrier for co-resident (cooperative) launches.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/spai_ir.h"

namespace spai {

// ---------------------------------------------------------------- precision

template <class S> struct Compute { typedef float T; };       // half, float -> float
template <> struct Compute<double> { typedef double T; };     // double -> double

__device__ __forceinline__ float to_c(__half v) { return __half2float(v); }
__device__ __forceinline__ float to_c(float v) { return v; }
__device__ __forceinline__ double to_c(double v) { return v; }

template <class S> __device__ __forceinline__ S from_f(float v);
template <> __device__ __forceinline__ __half from_f<__half>(float v) { return __float2half_rn(v); }
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <class S> __device__ __forceinline__ S from_d(double v);
template <> __device__ __forceinline__ __half from_d<__half>(double v) { return __double2half(v); }
template <> __device__ __forceinline__ float from_d<float>(double v) { return __double2float_rn(v); }
template <> __device__ __forceinline__ double from_d<double>(double v) { return v; }

// round a compute-type value to the storage precision S, returned in the
// compute type (the "store in u_f" step of the FP16-storage model)
template <class S> __device__ __forceinline__ typename Compute<S>::T rnd(typename Compute<S>::T v);
template <> __device__ __forceinline__ float rnd<__half>(float v) { return __half2float(__float2half_rn(v)); }
template <> __device__ __forceinline__ float rnd<float>(float v) { return v; }
template <> __device__ __forceinline__ double rnd<double>(double v) { return v; }

template <class T> __device__ __forceinline__ T ldcg(const T* p) { return __ldcg(p); }
template <> __device__ __forceinline__ __half ldcg<__half>(const __half* p)
{
    unsigned short r;
    asm volatile("ld.global.cg.u16 %0, [%1];" : "=h"(r) : "l"(p));
    return __ushort_as_half(r);
}

// ---------------------------------------------------------------- reductions

template <class T> __device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// Sum of a double over a warp, off the FP64 pipe: the values are aligned to
// the largest exponent as 58-bit integers (rounded to 2^-58 of that power of
// two), the integers summed exactly by three integer warp reductions of 26, 26
// and 12 bits, and the sum rounded once to double.  (One shared exponent and
// integer sums: the pre-rounded summation of Demmel and Nguyen, "Fast
// reproducible floating-point summation", ARITH 2013, with one bin.)  Its
// error is at most 32 x 2^-58 of the largest value plus one rounding, below
// the bound of the shuffle tree's five roundings, and it does not depend on
// the order.  An FP64 instruction of a warp holds its sub-partition's pipe for
// 64 cycles here: the tree took 545 cycles for one warp and 1550 for each of 16,
// this about 150.  Infinities, NaNs and values near the ends of the exponent
// range go through the tree.
__device__ __forceinline__ double warp_sum_fx(double v)
{
    const unsigned FULL = 0xffffffffu;
    const long long b = __double_as_longlong(v);
    const unsigned e = (unsigned)(b >> 52) & 0x7ffu;
    const unsigned em = __reduce_max_sync(FULL, e);
    if (em - 100u > 1900u) return warp_sum(v);  // (the same in every lane)
    const unsigned sh = em - e;
    const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull;
    // (a zero or subnormal has e = 0 and is shifted out)
    unsigned long long x = 0;
    if (sh < 59u) x = ((m << 5) + ((1ull << sh) >> 1)) >> sh;
    const long long sx = b < 0 ? -(long long)x : (long long)x;
    const unsigned l0 = (unsigned)sx & 0x3ffffffu, l1 = (unsigned)(sx >> 26) & 0x3ffffffu;
    const int l2 = (int)(sx >> 52);
    const unsigned s0 = __reduce_add_sync(FULL, l0), s1 = __reduce_add_sync(FULL, l1);
    const int s2 = __reduce_add_sync(FULL, l2);
    const long long S = (long long)s0 + ((long long)s1 << 26) + ((long long)s2 << 52);
    if (S == 0) return 0.0;
    // S counts units of 2^(em - 1023 - 57); the exponent field stays inside its range (em in 100..2000)
    return __longlong_as_double(__double_as_longlong(__ll2double_rn(S)) + ((long long)((int)em - 1080) << 52));
}
// The same for N <= 8 values a lane: one exponent, the lane's integers added first.
// With N = 5 (160 blocks) its error is at most 160 x 2^-58 of the largest value's power
// of two plus one rounding, where a lane's chain and the tree made up to ten roundings of
// 2^-53.  The sum may take 66 bits; past 62 its last four are folded into one sticky
// bit, which leaves its rounding to double the same.
template <int N> __device__ __forceinline__ double warp_sum_fx_n(const double (&v)[N])
{
    static_assert(N <= 8, "66 bits");
    const unsigned FULL = 0xffffffffu;
    unsigned e = 0;
#pragma unroll
    for (int k = 0; k < N; k++) e = max(e, (unsigned)(__double_as_longlong(v[k]) >> 52) & 0x7ffu);
    const unsigned em = __reduce_max_sync(FULL, e);
    if (em - 100u > 1900u) {
        double t = 0.0;
#pragma unroll
        for (int k = 0; k < N; k++) t += v[k];
        return warp_sum(t);
    }
    long long sx = 0;
#pragma unroll
    for (int k = 0; k < N; k++) {
        const long long b = __double_as_longlong(v[k]);
        const unsigned sh = em - ((unsigned)(b >> 52) & 0x7ffu);
        const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull;
        unsigned long long x = 0;
        if (sh < 59u) x = ((m << 5) + ((1ull << sh) >> 1)) >> sh;
        sx += b < 0 ? -(long long)x : (long long)x;
    }
    const unsigned l0 = (unsigned)sx & 0x3ffffffu, l1 = (unsigned)(sx >> 26) & 0x3ffffffu;
    const int l2 = (int)(sx >> 52);
    const unsigned s0 = __reduce_add_sync(FULL, l0), s1 = __reduce_add_sync(FULL, l1);
    const int s2 = __reduce_add_sync(FULL, l2);
    // the sum is H 2^26 + L
    const long long H = (long long)s1 + (s0 >> 26) + ((long long)s2 << 26);
    const unsigned L = s0 & 0x3ffffffu;
    const bool wide = H >= (1ll << 36) || H < -(1ll << 36);
    const long long S = wide ? (H << 22) + (long long)((L >> 4) | ((L & 15u) ? 1u : 0u)) : (H << 26) + (long long)L;
    if (S == 0) return 0.0;
    return __longlong_as_double(__double_as_longlong(__ll2double_rn(S)) + ((long long)((int)em - (wide ? 1076 : 1080)) << 52));
}
// Sum of N values by a tree: ceil(log2 N) roundings on the way of any of them.
template <int N, class T> __device__ __forceinline__ T tree_sum(T (&x)[N])
{
#pragma unroll
    for (int s = 1; s < N; s <<= 1)
#pragma unroll
        for (int i = 0; i + s < N; i += 2 * s) x[i] += x[i + s];
    return x[0];
}
// Sum of load(0) .. load(cnt - 1), N at a time in flight: each N by a tree, the trees'
// sums by two chains in turn (one of 50 values, N = 12: seven roundings).
template <int N, class T, class Load> __device__ __forceinline__ T strided_sum(int cnt, const Load& load)
{
    T a0 = T(0), a1 = T(0);
#pragma unroll 1
    for (int k0 = 0; k0 < cnt; k0 += N) {
        T x[N];
#pragma unroll
        for (int e = 0; e < N; e++) x[e] = k0 + e < cnt ? load(k0 + e) : T(0);
        const T t = a0 + tree_sum(x);
        a0 = a1;
        a1 = t;
    }
    return a0 + a1;
}
// Two float sums of a warp in one butterfly: lanes 0..15 get the sum of a,
// lanes 16..31 that of b (five shuffles, as for one).
__device__ __forceinline__ float warp_sum2(float a, float b)
{
    const bool up = threadIdx.x & 16;
    float v = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// the warp sum of the refinement kernels: shuffles for float, warp_sum_fx for double
__device__ __forceinline__ float wsum(float v) { return warp_sum(v); }
__device__ __forceinline__ double wsum(double v) { return warp_sum_fx(v); }

// x / d by y = 1 / d and one residual step (Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", 1990): q = x y, q + (x - q d) y, the
// correctly rounded quotient as long as x - q d is exact: |x| of at least 2^-100 in
// single or 2^-960 in double and a quotient in the normal range.  Below, within two units in the last
// place.  An infinite x (or x y) gives NaN, where a division gives an infinity: the
// callers' x are bounded by a norm that d or an earlier test has found finite.
template <class T> __device__ __forceinline__ T quot_by(T x, T d, T y)
{
    const T q = x * y;
    return fma(fma(-q, d, x), y, q);
}

// x / d for many x and one d by quot_by, whose three fused operations replace about
// nine FP64 instructions of a division in double (560 cycles of a sub-partition's pipe for a
// warp).  Divisors whose reciprocal could leave the exponent range keep the division.
// (Single too: the products' readers form v = w / h by quot_by, and the owner of v stores
// the same bits.)
template <class T> struct Quot {
    T d, y;
    bool fast;
    __device__ __forceinline__ explicit Quot(T d_) : d(d_), y(T(1) / d_)
    {
        const T big = sizeof(T) == 8 ? (T)1.0e250 : (T)1.0e30;
        fast = fabs(d_) < big && fabs(y) < big;
    }
    __device__ __forceinline__ T operator()(T x) const { return fast ? quot_by(x, d, y) : x / d; }
};

// Largest |v| over values and lanes as its bit pattern (non-negative numbers
// order like their bits), off the FP64 pipe; a NaN counts as infinite.
__device__ __forceinline__ unsigned long long abs_key(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    return b > 0x7ff0000000000000ull ? 0x7ff0000000000000ull : b;
}
__device__ __forceinline__ unsigned abs_key(float v)
{
    const unsigned b = __float_as_uint(v) & 0x7fffffffu;
    return b > 0x7f800000u ? 0x7f800000u : b;
}
__device__ __forceinline__ double key_value(unsigned long long k) { return __longlong_as_double((long long)k); }
__device__ __forceinline__ double key_value(unsigned k) { return (double)__uint_as_float(k); }
// the largest key of a warp, in every lane
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long k)
{
    const unsigned hi = (unsigned)(k >> 32);
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)k : 0u);
    return ((unsigned long long)mh << 32) | ml;
}

template <class T> __device__ __forceinline__ T warp_max(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
// sum within aligned groups of L lanes (L a power of two <= 32)
template <int L, class T> __device__ __forceinline__ T group_sum(T v)
{
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Deterministic block-wide sum; every thread gets the result.  red must
// hold 33 elements of T in shared memory.
template <class T> __device__ T block_sum(T v, T* red)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    v = warp_sum(v);
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        T t = lane < nw ? red[lane] : T(0);
        t = warp_sum(t);
        if (lane == 0) red[32] = t;
    }
    __syncthreads();
    T r = red[32];
    __syncthreads();
    return r;
}

// ---------------------------------------------------------------- double-double
// Error-free transformations (Knuth TwoSum, FMA-based TwoProd; Dekker 1971,
// Ogita-Rump-Oishi 2005) used for the quad-precision residual.

__device__ __forceinline__ void two_sum(double a, double b, double& s, double& e)
{
    s = a + b;
    double bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ void two_prod(double a, double b, double& p, double& e)
{
    p = a * b;
    e = fma(a, b, -p);
}
// (hi, lo) += a (double)
__device__ __forceinline__ void dd_add(double& hi, double& lo, double a)
{
    double s, e;
    two_sum(hi, a, s, e);
    e += lo;
    hi = s + e;
    lo = e - (hi - s);
}
// (hi, lo) -= a * b exactly-rounded product accumulation
__device__ __forceinline__ void dd_sub_prod(double& hi, double& lo, double a, double b)
{
    double p, pe;
    two_prod(a, b, p, pe);
    double s, e;
    two_sum(hi, -p, s, e);
    e += lo - pe;
    hi = s + e;
    lo = e - (hi - s);
}

// ---------------------------------------------------------------- grid barrier
// A barrier over all blocks of a co-resident (cooperative) launch.  The
// counter is monotonic: barrier number e completes when it reaches
// e * gridDim.x.  Every wait is bounded by a clock budget; on expiry the
// block records SPAI_ERR_TIMEOUT in *err and the barrier returns false, and
// any block that sees a non-zero *err also returns false, so all blocks
// leave the kernel.

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_relaxed_i32(const int* p)
{
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_add_u32(unsigned* p, unsigned v)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

struct GridBarrier {
    unsigned* count;   // zeroed before the launch
    int* err;          // zeroed before the launch
    long long limit;   // clock64 cycles before a wait gives up
    unsigned nblocks;  // blocks taking part (the grid, or one system's blocks of a batch)
};

struct NoBarrierWork {
    __device__ void operator()() const {}
};

// `epoch` is a per-block counter kept in shared memory by the caller and
// advanced identically by every block.  `work` runs on thread 0 after the
// block has arrived and before it starts waiting for the others (short
// serial work hides in the wait); the wait's clock budget starts after it.
template <class Work = NoBarrierWork>
__device__ __forceinline__ bool grid_sync(const GridBarrier& gb, unsigned* epoch, int* s_flag,
                                          const Work& work = Work())
{
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned e = *epoch + 1u;
        *epoch = e;
        const unsigned target = e * gb.nblocks;
        // release: the bar.sync above orders the block's writes before it
        red_release_add_u32(gb.count, 1u);
        work();
        int ok = 1;
        const long long t0 = clock64();
        unsigned spins = 0;
        while (ld_acquire_u32(gb.count) < target) {
            if (((++spins) & 63u) == 0u) {
                if (ld_relaxed_i32(gb.err) != 0) { ok = 0; break; }
                if (clock64() - t0 > gb.limit) {
                    atomicCAS(gb.err, 0, SPAI_ERR_TIMEOUT);
                    ok = 0;
                    break;
                }
            }
        }
        *s_flag = ok;
    }
    __syncthreads();
    return *s_flag != 0;
}

}  // namespace spai

// The structural check of a CSR on the device, one thread per row: rowptr[0]
// = 0, rowptr[n] = nnz, rows in order and inside [0, nnz], columns inside
// [0, n) and strictly ascending (flag 1); empty rows (flag 2) unless
// allow_empty.  Internal linkage: each translation unit that launches it
// has its own copy.
static __device__ __forceinline__ void csr_check_rows(int64_t n, int64_t nnz, const int64_t* __restrict__ rp,
                                                      const int32_t* __restrict__ col, int* __restrict__ flags,
                                                      int allow_empty)
{
    int f = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = rp[i], e = rp[i + 1];
        if ((i == 0 && b != 0) || (i == n - 1 && e != nnz)) f |= 1;
        if (b < 0 || e < b || e > nnz) { f |= 1; continue; }
        if (e == b) {
            if (!allow_empty) f |= 2;
            continue;
        }
        int prev = -1;
        for (int64_t q = b; q < e; q++) {
            const int c = col[q];
            if (c < 0 || c >= n || c <= prev) { f |= 1; break; }
            prev = c;
        }
    }
    if (f) atomicOr(flags, f);
}
static __global__ void k_csr_check(int64_t n, int64_t nnz, const int64_t* __restrict__ rp,
                                   const int32_t* __restrict__ col, int* __restrict__ flags, int allow_empty)
{
    csr_check_rows(n, nnz, rp, col, flags, allow_empty);
}

#define SPAI_CUDA_TRY(expr)                                   \
    do {                                                      \
        cudaError_t _e = (expr);                              \
        if (_e != cudaSuccess) {                              \
            spai_set_last_cuda_error(_e);                     \
            return _e == cudaErrorMemoryAllocation ? SPAI_ERR_NO_MEMORY : SPAI_ERR_CUDA; \
        }                                                     \
    } while (0)

void spai_set_last_cuda_error(cudaError_t e);
