// SPAI-GMRES-IR on the GPU: Algorithm 3 of the paper.
//
//   x0 = P b in u_f, stored in u                     (k_x0)
//   for i = 0 .. i_max-1:
//       r_i = b - A x_i in u_r, stored in u          (residual phase)
//       solve P A d_i = P r_i by left-preconditioned
//       MGS-GMRES in u_g, products with A, P in u_p  (Arnoldi phases)
//       x_{i+1} = x_i + d_i in u                      (update phase)
//
// The whole refinement loop is ONE persistent kernel (k_ir on a co-resident
// grid; k_ir_local on one thread-block cluster for small systems and batches):
// each block owns a contiguous slice of rows, keeps its slice of the
// Arnoldi vector w in shared memory, and meets the other blocks only at
// bounded grid barriers or cluster barriers.  For every grid-wide dot product the
// blocks write partials, and after the barrier every block adds them the same
// way (single in one order, double as integers), so all blocks hold
// bit-identical scalars and take identical control-flow decisions (GMRES
// convergence, refinement stop) without another barrier.  The Givens
// rotations, H, g and y are double precision in every block.
//
// Per Arnoldi iteration j: barrier after t = A v_j, one for the MGS dots of
// every two (double) or four (single) basis vectors, one for ||w||.  v_{j+1} = w / h_{j+1,j} is never re-published:
// readers form w_c / h from the published w themselves, the quotient the
// owner stores into V.
#include <algorithm>
#include <climits>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <map>
#include <set>
#include <vector>

#include "common.cuh"
#include "internal.h"
#include "ir_kernel.cuh"

using namespace spai;

namespace {

// ---------------------------------------------------------------- SELL-32 conversion

// the longest row of slice s (a warp), in lane 0
__device__ __forceinline__ int slice_width(int64_t n, const int64_t* __restrict__ rp, int64_t s)
{
    const int64_t row = s * 32 + (threadIdx.x & 31);
    int len = row < n ? (int)(rp[row + 1] - rp[row]) : 0;
    return (int)__reduce_max_sync(0xffffffffu, (unsigned)len);
}

// width of each 32-row slice (longest row), times 32
__global__ void k_sell_width(int64_t n, const int64_t* __restrict__ rp, int32_t* __restrict__ w32)
{
    const int lane = threadIdx.x & 31;
    const int64_t nsl = (n + 31) >> 5;
    for (int64_t s = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; s < nsl;
         s += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int len = slice_width(n, rp, s);
        if (lane == 0) w32[s] = len * 32;
    }
}

template <class TP>
__device__ __forceinline__ void sell_fill(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                          const double* __restrict__ val, const int64_t* __restrict__ off,
                                          int32_t* __restrict__ scol, TP* __restrict__ sval)
{
    const int lane = threadIdx.x & 31;
    const int64_t nsl = (n + 31) >> 5;
    for (int64_t s = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; s < nsl;
         s += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int64_t row = s * 32 + lane;
        const int w = (int)((off[s + 1] - off[s]) >> 5);
        const int64_t b = row < n ? rp[row] : 0;
        const int len = row < n ? (int)(rp[row + 1] - b) : 0;
        for (int c = 0; c < w; c++) {
            int64_t o = off[s] + 32 * c + lane;
            if (c < len) { scol[o] = ci[b + c]; sval[o] = from_d<TP>(val[b + c]); }
            else { scol[o] = row < n ? (int32_t)row : 0; sval[o] = from_d<TP>(0.0); }
        }
    }
}

template <class TP>
__global__ void k_sell_fill(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                            const double* __restrict__ val, const int64_t* __restrict__ off, int32_t* __restrict__ scol,
                            TP* __restrict__ sval)
{
    sell_fill<TP>(n, rp, ci, val, off, scol, sval);
}

// x0 = P_f b in u_f (FP16 storage / FP32 accumulation at half), stored in u
template <class S, class TU>
__device__ __forceinline__ void x0_rows(int64_t n, const int64_t* __restrict__ prp, const int32_t* __restrict__ pci,
                                        const S* __restrict__ pv, const double* __restrict__ b, TU* __restrict__ x)
{
    typedef typename Compute<S>::T C;
    for (int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; row < n; row += (int64_t)gridDim.x * blockDim.x) {
        C acc = C(0);
        if (prp) {
            for (int64_t q = prp[row]; q < prp[row + 1]; q++)
                acc = fma(to_c(pv[q]), to_c(from_d<S>(b[pci[q]])), acc);
        } else {
            acc = to_c(from_d<S>(b[row]));
        }
        x[row] = (TU)to_c(from_d<S>((double)acc));
    }
}

template <class S, class TU>
__global__ void k_x0(int64_t n, const int64_t* __restrict__ prp, const int32_t* __restrict__ pci,
                     const S* __restrict__ pv, const double* __restrict__ b, TU* __restrict__ x)
{
    x0_rows<S, TU>(n, prp, pci, pv, b, x);
}

template <class TU>
__global__ void k_to_double(int64_t n, const TU* __restrict__ x, double* __restrict__ out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (double)x[i];
}


// ||A||_inf, ||b||_inf, the largest row count q (per-block maxima, then one
// atomic per block and value) and the sum of the entries' distances |i - j|
// from the diagonal (out[5])
__device__ __forceinline__ void norms_rows(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                           const double* __restrict__ val, const double* __restrict__ b,
                                           unsigned long long* __restrict__ out)
{
    __shared__ double sa[32], sb[32];
    __shared__ int sq[32];
    __shared__ unsigned long long sd[32];
    double an = 0.0, bn = 0.0;
    int q = 0;
    unsigned long long dist = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int64_t p = rp[i]; p < rp[i + 1]; p++) {
            s += fabs(val[p]);
            const int64_t t = i - col[p];
            dist += (unsigned long long)(t < 0 ? -t : t);
        }
        an = fmax(an, s);
        bn = fmax(bn, fabs(b[i]));
        q = max(q, (int)(rp[i + 1] - rp[i]));
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    an = warp_max(an);
    bn = warp_max(bn);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q = max(q, __shfl_xor_sync(0xffffffffu, q, o));
    dist = warp_sum(dist);
    if (lane == 0) { sa[wid] = an; sb[wid] = bn; sq[wid] = q; sd[wid] = dist; }
    __syncthreads();
    if (wid == 0) {
        an = lane < nw ? sa[lane] : 0.0;
        bn = lane < nw ? sb[lane] : 0.0;
        q = lane < nw ? sq[lane] : 0;
        dist = warp_sum(lane < nw ? sd[lane] : 0ull);
        an = warp_max(an);
        bn = warp_max(bn);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) q = max(q, __shfl_xor_sync(0xffffffffu, q, o));
        if (lane == 0) {
            // non-negative doubles order like their bit patterns
            atomicMax(&out[0], (unsigned long long)__double_as_longlong(an));
            atomicMax(&out[1], (unsigned long long)__double_as_longlong(bn));
            atomicMax(&out[2], (unsigned long long)q);
            atomicAdd(&out[5], dist);
        }
    }
}

__global__ void k_norms(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                        const double* __restrict__ val, const double* __restrict__ b,
                        unsigned long long* __restrict__ out)
{
    norms_rows(n, rp, col, val, b, out);
}

// the kernels of the run-time precision tuple (u, u_g, u_p), u_r and orth
int ir_kernels(int u, int ug, int up, int ur, int orth, IrKernels* k)
{
    const int rm = ur == SPAI_QUAD ? 2 : 1;
    const bool ls = orth == 2;
    const bool ud = u == SPAI_DOUBLE;
    if (ug == SPAI_HALF || up == SPAI_HALF) {
        k->one = nullptr;
        if (ug == SPAI_HALF && up == SPAI_HALF) (ud ? ir_kernels_dhh : ir_kernels_fhh)(rm, ls, k);
        else if (ug == SPAI_HALF && up == SPAI_SINGLE) (ud ? ir_kernels_dhf : ir_kernels_fhf)(rm, ls, k);
        else if (ug == SPAI_SINGLE && up == SPAI_HALF) (ud ? ir_kernels_dfh : ir_kernels_ffh)(rm, ls, k);
        return k->one ? 0 : SPAI_ERR_UNSUPPORTED;
    }
    const int key = (u == SPAI_DOUBLE) * 4 + (ug == SPAI_DOUBLE) * 2 + (up == SPAI_DOUBLE);
    switch (key) {
    case 0: ir_kernels_fff(rm, ls, k); break;
    case 1: ir_kernels_ffd(rm, ls, k); break;
    case 2: ir_kernels_fdf(rm, ls, k); break;
    case 3: ir_kernels_fdd(rm, ls, k); break;
    case 4: ir_kernels_dff(rm, ls, k); break;
    case 5: ir_kernels_dfd(rm, ls, k); break;
    case 6: ir_kernels_ddf(rm, ls, k); break;
    default: ir_kernels_ddd(rm, ls, k); break;
    }
    return k->one ? 0 : SPAI_ERR_UNSUPPORTED;
}

// The order up to which a single system runs as one thread-block cluster
// instead of a co-resident grid.  A cluster of 16 SMs meets in about 0.5 us
// where a grid meets in 1.5 us or more, but it streams the matrices and the
// basis through 16 SMs only, whose share of the work weighs more in double.
// Measured (us per iteration, cluster / grid): MGS single, 3D pattern(A^2),
// n = 8000: 16.1 / 17.9, 12696: 19.3 / 19.2, 17576: 23.9 / 20.4; MGS double n = 4096:
// 27.2 / 33.0 (2D pattern(A): 35.9 / 42.0), 8000: 40.9 / 35.8, 2D n = 10000: 51.5 / 44.8;
// one-reduction single n = 10648: 21.8 / 22.6, 17576: 24.3 / 23.0; double n = 4096:
// 28.0 / 31.0, 10648: 37.5 / 31.6.
int64_t cluster_rows(bool dbl) { return dbl ? 6144 : 12288; }

// A launch of `grid` blocks in clusters of T blocks (T > 1).
struct ClusterLaunch {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    ClusterLaunch(int grid, int T, int threads, size_t smem, cudaStream_t s)
    {
        memset(&cfg, 0, sizeof(cfg));
        memset(&at, 0, sizeof(at));
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        if (T > 1) {
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = (unsigned)T;
            at.val.clusterDim.y = 1;
            at.val.clusterDim.z = 1;
            cfg.attrs = &at;
            cfg.numAttrs = 1;
        }
    }
};

// The largest cluster, of at most MAX_CLUSTER blocks, that the device can run `kern`
// in with the most threads and shared memory a launch takes (more than eight blocks
// are not portable); asked once per kernel and device.
int max_cluster(const void* kern, size_t dyn_max)
{
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, int> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_pair(kern, dev);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    int T = MAX_CLUSTER;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) T = 8;
    for (; T > 1; T--) {
        ClusterLaunch L(T, T, IR_BT, dyn_max, nullptr);
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, kern, &L.cfg) == cudaSuccess && fit > 0) break;
    }
    cudaGetLastError();
    return known[key] = T;
}

// Launch `grid` blocks of `kern`, in clusters of T blocks when T > 1 (T <= max_cluster).
cudaError_t launch_clusters(const void* kern, int grid, int T, int threads, size_t smem, void** args, cudaStream_t s)
{
    ClusterLaunch L(grid, T, threads, smem, s);
    return cudaLaunchKernelExC(&L.cfg, kern, args);
}

// One system: on one block or one cluster (cluster_rows), or on its own grid,
// one block per SM, at least 256 rows per block, rows per block a multiple of
// 32 so that blocks own whole SELL slices.  sg = sizeof(u_g); entries: of the larger
// SELL matrix.
int launch_ir(IrArgs& a, const IrKernels& K, int sg, int sp, bool scattered, int64_t entries, int num_sms, cudaStream_t s,
              int* grid_out)
{
    size_t dyn_max = 0;
    a.scat = scattered ? 1 : 0;
    auto take = [&](const IrSmem& m) {
        a.jl = m.jl;
        a.nq = m.nq;
        a.xcap = m.xcap;
        a.xs_off = (int)m.xs_off;
    };
    if (a.n <= cluster_rows(sg == 8 || sp == 8)) {
        int64_t G = std::min<int64_t>((a.n + 63) / 64, MAX_CLUSTER);
        a.sblock = a.orth == 2 && a.gpub && G >= 9 ? 1 : 0;
        if (a.sblock && G == MAX_CLUSTER) G--;
        a.rb = ((a.n + G - 1) / G + 31) & ~int64_t(31);
        G = (a.n + a.rb - 1) / a.rb + a.sblock;
        a.g2 = 0;
        SPAI_CUDA_TRY(allow_max_dynamic_smem_ptr(K.local, &dyn_max));
        const IrSmem m = ir_pick_smem(a.rb, a.kmax, 0, a.orth, dyn_max, sg, sp, scattered ? a.n : 0);
        if (m.bytes <= dyn_max && G <= max_cluster(K.local, dyn_max)) {
            take(m);
            const IrArgs* none = nullptr;
            int T = (int)G;
            void* args[] = {(void*)&a, (void*)&none, (void*)&T};
            const cudaError_t e = launch_clusters(K.local, T, T, ir_block_threads(a.rb, a.orth), m.bytes, args, s);
            if (e == cudaSuccess) {
                *grid_out = (int)G;
                return 0;
            }
            cudaGetLastError();
            // (a size that is refused all the same: the grid)
            if (e != cudaErrorInvalidClusterSize && e != cudaErrorInvalidConfiguration && e != cudaErrorLaunchOutOfResources) {
                spai_set_last_cuda_error(e);
                return SPAI_ERR_CUDA;
            }
        }
    }
    const void* one = entries > IR_WIDE ? K.wide : K.one;
    SPAI_CUDA_TRY(allow_max_dynamic_smem_ptr(one, &dyn_max));
    // the one-reduction MGS on grids of 8 or more row blocks adds a block without
    // rows that runs the Givens rotations (FP64 work beside the other blocks'
    // inner products slowed both)
    const bool sblock = a.orth == 2 && a.gpub && std::min<int64_t>((a.n + 255) / 256, std::min(num_sms, MAX_GRID)) >= 9;
    int64_t G = std::min<int64_t>((a.n + 255) / 256, std::min(num_sms, MAX_GRID) - (sblock ? 1 : 0));
    if (G < 1) G = 1;
    a.rb = ((a.n + G - 1) / G + 31) & ~int64_t(31);
    G = (a.n + a.rb - 1) / a.rb;
    a.sblock = sblock ? 1 : 0;
    if (sblock) G += 1;
    // Gram-Schmidt group: on large grids the rounds run among half the blocks
    // (each over two blocks' rows), where an exchange takes less than among all; that
    // has to outweigh the extra barrier that publishes w once per iteration
    // (mgs_group_min_grid), and a thread's prefetched rows have to cover
    // the double range (else, n = 175616: 45.9 us per iteration in single against
    // 42.2 among all blocks, 136.8 / 126.3 in double; n = 262144: 75.5 / 51.5, 192.6 /
    // 156.8).  CGS2 and the one-reduction MGS have no such rounds.
    a.g2 = (!a.orth && G >= mgs_group_min_grid(sg) && 2 * a.rb <= PF * ir_block_threads(a.rb, 0)) ? (int)((G + 1) / 2) : 0;
    IrSmem m = ir_pick_smem(a.rb, a.kmax, a.g2, a.orth, dyn_max, sg, sp, 0, scattered && sg == 8);
    if (a.g2 && m.bytes > dyn_max) {  // the doubled row range does not fit
        a.g2 = 0;
        m = ir_pick_smem(a.rb, a.kmax, 0, a.orth, dyn_max, sg, sp, 0);
    }
    take(m);
    const size_t smem = m.bytes;
    if (smem > dyn_max) return SPAI_ERR_UNSUPPORTED;
    int occ = 0;
    SPAI_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, one, ir_block_threads(a.rb, a.orth), smem));
    if ((int64_t)occ * num_sms < G) return SPAI_ERR_UNSUPPORTED;
    void* args[] = {(void*)&a};
    SPAI_CUDA_TRY(cudaLaunchCooperativeKernel(one, dim3((unsigned)G), dim3(ir_block_threads(a.rb, a.orth)), args, smem, s));
    *grid_out = (int)G;
    return 0;
}

int prec_bytes(int p) { return p == SPAI_HALF ? 2 : (p == SPAI_SINGLE ? 4 : 8); }

// the preconditioner's cached SELL-32 copy in u_p
SellMat* sell_cache(spai_precond P, int up)
{
    return up == SPAI_HALF ? &P->sell_f16 : (up == SPAI_SINGLE ? &P->sell_f32 : &P->sell_f64);
}

}  // namespace

// SELL-32 copy of a CSR matrix with values rounded to `prec` (half, single or double),
// in two halves: sell_begin computes the slice offsets (the entry count stays
// on the device at off[nslices]); sell_finish allocates and fills once that
// count is known on the host.
int sell_begin(int64_t n, const int64_t* rp, int num_sms, cudaStream_t s, SellMat* out, int* launches)
{
    const int64_t nsl = (n + 31) >> 5;
    int32_t* w32 = nullptr;
    int rc = dev_alloc((void**)&w32, sizeof(int32_t) * nsl, s);
    if (rc) return rc;
    rc = dev_alloc((void**)&out->off, sizeof(int64_t) * (nsl + 1), s);
    if (rc) { dev_free(w32, s); return rc; }
    const int tb = 256;
    const int gb = (int)std::max<int64_t>(1, std::min<int64_t>((nsl * 32 + tb - 1) / tb, (int64_t)num_sms * 16));
    k_sell_width<<<gb, tb, 0, s>>>(n, rp, w32);
    rc = scan_counts(nsl, w32, out->off, s);
    *launches += 4;
    dev_free(w32, s);
    return rc;
}

int sell_finish(int64_t n, const int64_t* rp, const int32_t* ci, const double* val, int prec, int num_sms,
                cudaStream_t s, SellMat* out, int64_t total, int* launches)
{
    const int64_t nsl = (n + 31) >> 5;
    const int tb = 256;
    const int gb = (int)std::max<int64_t>(1, std::min<int64_t>((nsl * 32 + tb - 1) / tb, (int64_t)num_sms * 16));
    int rc;
    out->prec = prec;
    out->nnz = total;
    if ((rc = dev_alloc((void**)&out->col, sizeof(int32_t) * std::max<int64_t>(total, 1), s))) return rc;
    if ((rc = dev_alloc(&out->val, (size_t)prec_bytes(prec) * std::max<int64_t>(total, 1), s))) return rc;
    if (prec == SPAI_HALF) k_sell_fill<__half><<<gb, tb, 0, s>>>(n, rp, ci, val, out->off, out->col, (__half*)out->val);
    else if (prec == SPAI_SINGLE) k_sell_fill<float><<<gb, tb, 0, s>>>(n, rp, ci, val, out->off, out->col, (float*)out->val);
    else k_sell_fill<double><<<gb, tb, 0, s>>>(n, rp, ci, val, out->off, out->col, (double*)out->val);
    *launches += 1;
    SPAI_CUDA_TRY(cudaGetLastError());
    return 0;
}

int sell_build(int64_t n, const int64_t* rp, const int32_t* ci, const double* val, int prec, int num_sms,
               cudaStream_t s, SellMat* out, int* launches)
{
    int rc = sell_begin(n, rp, num_sms, s, out, launches);
    if (rc) return rc;
    const int64_t nsl = (n + 31) >> 5;
    int64_t total = 0;
    if (cudaMemcpyAsync(&total, out->off + nsl, sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess) return SPAI_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return SPAI_ERR_CUDA;
    return sell_finish(n, rp, ci, val, prec, num_sms, s, out, total, launches);
}

void sell_free(SellMat* m, cudaStream_t s)
{
    dev_free(m->off, s);
    dev_free(m->col, s);
    dev_free(m->val, s);
    m->off = nullptr;
    m->col = nullptr;
    m->val = nullptr;
}

namespace {

// One system's refinement: buffers, the host copies of its results, and the
// kernel arguments.  gmres_ir_dev runs one job; gmres_ir_batch_dev runs the
// jobs of one team size in one launch.
// What a refinement leaves for the host, in one block of the job's buffers so that one copy brings it.
struct IrResult {
    int out[2];
    int err[2];
    int its[SPAI_IR_MAX_STEPS + 2];
    double nbe[SPAI_IR_MAX_STEPS + 2];
};

struct IrJob {
    const DevCsr* A = nullptr;
    spai_precond P = nullptr;
    const double* b = nullptr;
    double* xout = nullptr;
    int64_t n = 0;
    int kmax = 0, imax = 0;
    void *x = nullptr, *r = nullptr, *wbuf = nullptr, *tbuf = nullptr, *V = nullptr;
    double* R = nullptr;
    IrResult* res = nullptr;
    unsigned long long* msg = nullptr;
    unsigned long long* norms = nullptr;
    void* pvec = nullptr;
    unsigned* gcount = nullptr;
    void* L = nullptr;
    double* gpub = nullptr;
    void* arena = nullptr;  // one allocation holding all of the above
    SellMat As;
    const SellMat* Ps = nullptr;
    unsigned long long h_norms[3] = {0, 0, 0};
    bool scattered = false;
    size_t ctrl = 0;        // its first bytes, cleared before the solve
    IrResult h{};
    IrArgs a;
};

int ir_check_opts(const ir_opts* o)
{
    if (!o) return SPAI_ERR_INVALID_ARG;
    if (o->u != SPAI_SINGLE && o->u != SPAI_DOUBLE) return SPAI_ERR_UNSUPPORTED;
    if (o->ug != SPAI_HALF && o->ug != SPAI_SINGLE && o->ug != SPAI_DOUBLE) return SPAI_ERR_UNSUPPORTED;
    if (o->up != SPAI_HALF && o->up != SPAI_SINGLE && o->up != SPAI_DOUBLE) return SPAI_ERR_UNSUPPORTED;
    // half Krylov storage: with the one-reduction MGS, and beside single only
    if ((o->ug == SPAI_HALF || o->up == SPAI_HALF) &&
        (o->orth != 2 || o->ug == SPAI_DOUBLE || o->up == SPAI_DOUBLE))
        return SPAI_ERR_UNSUPPORTED;
    if (o->ur != SPAI_DOUBLE && o->ur != SPAI_QUAD) return SPAI_ERR_UNSUPPORTED;
    if (o->uf != SPAI_HALF && o->uf != SPAI_SINGLE && o->uf != SPAI_DOUBLE) return SPAI_ERR_UNSUPPORTED;
    if (o->ir_max_steps < 1 || o->ir_max_steps > SPAI_IR_MAX_STEPS) return SPAI_ERR_INVALID_ARG;
    if (!(o->tau >= 0.0)) return SPAI_ERR_INVALID_ARG;
    if (o->orth < 0 || o->orth > 2) return SPAI_ERR_INVALID_ARG;
    if (o->side != 0 && o->side != 1) return SPAI_ERR_INVALID_ARG;
    if (o->stop != IR_STOP_BACKWARD && o->stop != IR_STOP_FIXED && o->stop != IR_STOP_CORRECTION)
        return SPAI_ERR_INVALID_ARG;
    return 0;
}

// The stopping threshold (reading R8): the caller's, else q u for the
// backward-error rule (q the longest row of A, the limit of Theorem 2) and u
// for the correction rule.
double ir_stop_tol(const ir_opts* o, int q)
{
    const double uu = o->u == SPAI_SINGLE ? 5.9604644775390625e-08 : 1.1102230246251565e-16;
    if (o->stop_tol > 0) return o->stop_tol;
    return o->stop == IR_STOP_CORRECTION ? uu : q * uu;
}

int ir_job_kmax(int64_t n, const ir_opts* o, int* kmax)
{
    int k = o->gmres_max_it > 0 ? o->gmres_max_it : (int)std::min<int64_t>(n, 500);
    if (k > n) k = (int)n;
    if (k > KMAX_LIMIT) return SPAI_ERR_UNSUPPORTED;
    if (k < 1) k = 1;
    *kmax = k;
    return 0;
}

// The job's buffers, carved from one allocation on s (one runtime call instead
// of one per buffer: a batch prepares hundreds of jobs); the control words
// (norms, exchange slots, results, counters) come first and are cleared
// together, here or (clear = false) by the batch's k_batch_start.
int ir_job_alloc(IrJob& J, cudaStream_t s, const ir_opts* o, bool clear)
{
    const int64_t n = J.n;
    const int su = prec_bytes(o->u), sg = prec_bytes(o->ug), sp = prec_bytes(o->up);
    const int64_t ldv = (n + 31) & ~int64_t(31);
    const int kmax = J.kmax;
    size_t off = 0;
    auto place = [&](size_t bytes) {
        off = (off + 255) & ~size_t(255);
        const size_t at = off;
        off += bytes;
        return at;
    };
    // [0..2] the norms and the longest row, [3] [4] SELL entry counts of A and P, [5] the entries'
    // distance from the diagonal
    const size_t o_norms = place(sizeof(unsigned long long) * 6);
    const size_t o_msg = place(sizeof(unsigned long long) * 4 * MAX_GRID * SLOT_WORDS);
    const size_t o_res = place(sizeof(IrResult));
    const size_t o_gcount = o->orth ? place(sizeof(unsigned)) : 0;
    J.ctrl = (off + 15) & ~size_t(15);
    off = J.ctrl;
    const size_t o_x = place((size_t)su * n);
    const size_t o_r = place((size_t)su * n);
    const size_t o_wbuf = place((size_t)sg * ldv);
    const size_t o_tbuf = place((size_t)sp * n);
    const size_t o_V = place((size_t)sg * ldv * (kmax + 1));
    const size_t o_R = place(sizeof(double) * (size_t)(kmax + 1) * kmax);
    // CGS2: 2 parities x blocks x (kmax + 1) partials; one-reduction MGS: 2 (kmax + 1) values
    // x blocks, then the 2 (kmax + 1) sums of the split reduction
    const size_t o_pvec = o->orth ? place((size_t)ir_scalar_bytes(sg) * (2 * MAX_GRID + (o->orth == 2 ? 2 : 0)) * (kmax + 1)) : 0;
    const size_t o_L = o->orth == 2 ? place((size_t)ir_scalar_bytes(sg) * ((size_t)(kmax + 1) * kmax / 2 + 1)) : 0;
    const size_t o_gpub = o->orth == 2 ? place(sizeof(double) * (kmax + 2)) : 0;
    int rc = dev_alloc(&J.arena, off, s);
    if (rc) return rc;
    unsigned char* base = (unsigned char*)J.arena;
    J.norms = (unsigned long long*)(base + o_norms);
    J.msg = (unsigned long long*)(base + o_msg);
    J.res = (IrResult*)(base + o_res);
    J.gcount = o->orth ? (unsigned*)(base + o_gcount) : nullptr;
    J.x = base + o_x;
    J.r = base + o_r;
    J.wbuf = base + o_wbuf;
    J.tbuf = base + o_tbuf;
    J.V = base + o_V;
    J.R = (double*)(base + o_R);
    J.pvec = o->orth ? base + o_pvec : nullptr;
    J.L = o->orth == 2 ? base + o_L : nullptr;
    J.gpub = o->orth == 2 ? (double*)(base + o_gpub) : nullptr;
    if (clear && cudaMemsetAsync(base, 0, J.ctrl, s) != cudaSuccess) return SPAI_ERR_CUDA;
    return 0;
}

// ||A||_inf, ||b||_inf, the longest row into J.norms, and x0 = P b in u_f
// stored in u, enqueued on s.
int ir_job_norms_x0(IrJob& J, int num_sms, cudaStream_t s, const ir_opts* o, int* nl)
{
    const int64_t n = J.n;
    const int tb = 256;
    const int gb = (int)std::max<int64_t>(1, std::min<int64_t>((n + tb - 1) / tb, (int64_t)num_sms * 32));
    const DevCsr& A = *J.A;
    spai_precond P = J.P;
    k_norms<<<gb, tb, 0, s>>>(n, A.rowptr, A.col, A.val, J.b, J.norms);
    (*nl)++;
    // x0 = P b in u_f, stored in u
    const int64_t* prp = P ? P->rowptr : nullptr;
    const int32_t* pci = P ? P->col : nullptr;
    const void* pvf = P ? P->val_uf : nullptr;
#define X0(S, TU) k_x0<S, TU><<<gb, tb, 0, s>>>(n, prp, pci, (const S*)pvf, J.b, (TU*)J.x)
    if (o->u == SPAI_SINGLE) {
        if (o->uf == SPAI_HALF) X0(__half, float);
        else if (o->uf == SPAI_SINGLE) X0(float, float);
        else X0(double, float);
    } else {
        if (o->uf == SPAI_HALF) X0(__half, double);
        else if (o->uf == SPAI_SINGLE) X0(float, double);
        else X0(double, double);
    }
#undef X0
    (*nl)++;
    if (cudaGetLastError() != cudaSuccess) return SPAI_ERR_CUDA;
    return 0;
}

// Allocations, SELL-32 copies of A (and of P, cached on the handle), the norms
// and x0 = P b, enqueued on s with one synchronisation (for the SELL entry
// counts and the norms, which are on the host when it returns).
int ir_job_prepare(IrJob& J, int num_sms, cudaStream_t s, const ir_opts* o, int* nl)
{
    int rc = ir_job_alloc(J, s, o, true);
    if (rc) return rc;
    const DevCsr& A = *J.A;
    spai_precond P = J.P;
    // one host synchronisation for the SELL entry counts and the norms: the
    // counts join the norms on the device, and one copy brings all six
    const int64_t nsl = (J.n + 31) >> 5;
    SellMat* cache = nullptr;
    rc = sell_begin(J.n, A.rowptr, num_sms, s, &J.As, nl);
    if (rc) return rc;
    if (cudaMemcpyAsync(J.norms + 3, J.As.off + nsl, 8, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return SPAI_ERR_CUDA;
    if (P) {
        cache = sell_cache(P, o->up);
        if (!cache->off) {
            rc = sell_begin(J.n, P->rowptr, num_sms, s, cache, nl);
            if (rc) return rc;
            if (cudaMemcpyAsync(J.norms + 4, cache->off + nsl, 8, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
                return SPAI_ERR_CUDA;
        } else {
            cache = nullptr;  // already made
        }
        J.Ps = sell_cache(P, o->up);
    }
    rc = ir_job_norms_x0(J, num_sms, s, o, nl);
    if (rc) return rc;
    unsigned long long h[6] = {0, 0, 0, 0, 0, 0};
    if (cudaMemcpyAsync(h, J.norms, sizeof(h), cudaMemcpyDeviceToHost, s) != cudaSuccess) return SPAI_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return SPAI_ERR_CUDA;
    for (int k = 0; k < 3; k++) J.h_norms[k] = h[k];
    J.scattered = ir_scattered(J.n, A.nnz, h[5]);
    const int64_t tot[2] = {(int64_t)h[3], (int64_t)h[4]};
    rc = sell_finish(J.n, A.rowptr, A.col, A.val, o->up, num_sms, s, &J.As, tot[0], nl);
    if (rc) return rc;
    if (cache) rc = sell_finish(J.n, P->rowptr, P->col, P->val, o->up, num_sms, s, cache, tot[1], nl);
    return rc;
}

// The kernel arguments, once the norms have reached the host (after a sync).
void ir_job_args(IrJob& J, int device, const ir_opts* o)
{
    IrArgs& a = J.a;
    memset(&a, 0, sizeof(a));
    double anorm, bnorm;
    long long t0 = (long long)J.h_norms[0], t1 = (long long)J.h_norms[1];
    memcpy(&anorm, &t0, 8);
    memcpy(&bnorm, &t1, 8);
    const int q = (int)J.h_norms[2];
    const DevCsr& A = *J.A;
    a.n = J.n;
    a.A.off = J.As.off; a.A.col = J.As.col; a.A.val = J.As.val;
    if (J.Ps) { a.P.off = J.Ps->off; a.P.col = J.Ps->col; a.P.val = J.Ps->val; }
    a.arp = A.rowptr; a.aci = A.col; a.aval = A.val;
    a.b = J.b; a.x = J.x; a.r = J.r; a.wbuf = J.wbuf; a.tbuf = J.tbuf; a.V = J.V;
    a.ldv = (J.n + 31) & ~int64_t(31); a.R = J.R; a.msg = J.msg;
    a.msg2 = J.msg + 2 * MAX_GRID * SLOT_WORDS;
    a.err = J.res->err;
    int clk_khz = device_attr_cached(cudaDevAttrClockRate, device);
    if (clk_khz <= 0) clk_khz = 2000000;
    a.limit = (long long)clk_khz * 1000LL * 4;  // about four seconds per wait
    a.anorm = anorm; a.bnorm = bnorm; a.tau = o->tau;
    a.stop_tol = ir_stop_tol(o, q);
    a.kmax = J.kmax; a.imax = J.imax; a.stop_rule = o->stop;
    a.its = J.res->its; a.nbe = J.res->nbe; a.out = J.res->out;
    a.orth = o->orth; a.pvec = J.pvec; a.gcount = J.gcount; a.L = J.L; a.gpub = J.gpub; a.side = o->side;
}

// the entries of the larger SELL copy
int64_t ir_job_entries(const IrJob& J) { return std::max(J.As.nnz, J.Ps ? J.Ps->nnz : (int64_t)0); }

// x in double, enqueued on s.
void ir_job_x(IrJob& J, int num_sms, cudaStream_t s, const ir_opts* o, int* nl)
{
    const int tb = 256;
    const int gb = (int)std::max<int64_t>(1, std::min<int64_t>((J.n + tb - 1) / tb, (int64_t)num_sms * 32));
    if (o->u == SPAI_SINGLE) k_to_double<float><<<gb, tb, 0, s>>>(J.n, (const float*)J.x, J.xout);
    else k_to_double<double><<<gb, tb, 0, s>>>(J.n, (const double*)J.x, J.xout);
    (*nl)++;
}

// x in double and the result copy, enqueued on s.
int ir_job_collect(IrJob& J, int num_sms, cudaStream_t s, const ir_opts* o, int* nl)
{
    ir_job_x(J, num_sms, s, o, nl);
    if (cudaGetLastError() != cudaSuccess) return SPAI_ERR_CUDA;
    if (cudaMemcpyAsync(&J.h, J.res, sizeof(J.h), cudaMemcpyDeviceToHost, s) != cudaSuccess) return SPAI_ERR_CUDA;
    return 0;
}

// After a sync: the statistics (timings and launch counts are the caller's)
// and the return code of the job.
int ir_job_result(const IrJob& J, const ir_opts* o, ir_stats* st)
{
    if (J.h.err[0]) return J.h.err[0];
    if (st) {
        memset(st->its, 0, sizeof(st->its));
        for (int i = 0; i < J.imax; i++) st->its[i] = J.h.its[i];
        for (int i = 0; i <= SPAI_IR_MAX_STEPS; i++) st->nbe[i] = 0.0;
        st->steps = J.h.out[0];
        st->flags = J.h.out[1];
        for (int i = 0; i <= st->steps && i <= J.imax; i++) st->nbe[i] = J.h.nbe[i];
        st->total_its = 0;
        for (int i = 0; i < st->steps; i++) st->total_its += st->its[i];
        st->final_nbe = st->nbe[st->steps];
        st->nnz_P = J.P ? J.P->nnz : 0;
    }
    if (J.h.out[1] & 8) return SPAI_ERR_NONFINITE;
    if (!(J.h.out[1] & 1) && o->stop != IR_STOP_FIXED) return SPAI_WARN_NOT_CONVERGED;
    return 0;
}

void ir_job_free(IrJob& J, cudaStream_t s)
{
    sell_free(&J.As, s);
    dev_free(J.arena, s);
    J.arena = nullptr;
    J.gpub = nullptr;
    J.x = J.r = J.wbuf = J.tbuf = J.V = J.pvec = J.L = nullptr;
    J.R = nullptr;
    J.res = nullptr;
    J.msg = J.norms = nullptr;
    J.gcount = nullptr;
}

}  // namespace

int gmres_ir_dev(int device, int num_sms, cudaStream_t s, const DevCsr& A, spai_precond P,
                 const double* b, double* xout, const ir_opts* o, ir_stats* st)
{
    int rc = ir_check_opts(o);
    if (rc) return rc;
    if (P && P->uf != o->uf) return SPAI_ERR_INVALID_ARG;
    IrJob J;
    J.A = &A; J.P = P; J.b = b; J.xout = xout; J.n = A.n; J.imax = o->ir_max_steps;
    rc = ir_job_kmax(A.n, o, &J.kmax);
    if (rc) return rc;
    cudaEvent_t e0 = nullptr, e1 = nullptr, ek0 = nullptr, ek1 = nullptr;
    SPAI_CUDA_TRY(cudaEventCreate(&e0));
    SPAI_CUDA_TRY(cudaEventCreate(&e1));
    SPAI_CUDA_TRY(cudaEventCreate(&ek0));
    SPAI_CUDA_TRY(cudaEventCreate(&ek1));
    int nl = 0;  // kernels launched
    int grid = 0;
#define TRY(x) do { rc = (x); if (rc) goto done; } while (0)
#define CTRY(x) do { if ((x) != cudaSuccess) { rc = SPAI_ERR_CUDA; goto done; } } while (0)
    CTRY(cudaEventRecord(e0, s));
    TRY(ir_job_prepare(J, num_sms, s, o, &nl));  // the norms are on the host when it returns
    ir_job_args(J, device, o);
    CTRY(cudaEventRecord(ek0, s));
    {
        IrKernels K;
        TRY(ir_kernels(o->u, o->ug, o->up, o->ur, o->orth, &K));
        TRY(launch_ir(J.a, K, prec_bytes(o->ug), prec_bytes(o->up), J.scattered, ir_job_entries(J), num_sms, s,
                      &grid));
    }
    CTRY(cudaEventRecord(ek1, s));
    nl++;
    TRY(ir_job_collect(J, num_sms, s, o, &nl));
    CTRY(cudaEventRecord(e1, s));
    CTRY(cudaStreamSynchronize(s));
    rc = ir_job_result(J, o, st);
    if (rc >= 0 && st) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        st->ms_ir = ms;
        cudaEventElapsedTime(&ms, ek0, ek1);
        st->ms_kernel = ms;
        st->launches += nl;
        st->grid = grid;
    }
done:
#undef TRY
#undef CTRY
    ir_job_free(J, s);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (ek0) cudaEventDestroy(ek0);
    if (ek1) cudaEventDestroy(ek1);
    if (rc < 0) cudaStreamSynchronize(s);
    return rc;
}

// ====================================================================
// Self-test of the bounded device waits (spai_selftest_wait_timeout): the
// blocks of a small launch run one exchange round (mode 0) or one counter
// barrier (mode 1) that counts one block more than the grid holds, so they
// wait for a word or an arrival that nothing provides.  Each wait gives up
// after a.limit clock cycles, records SPAI_ERR_TIMEOUT and returns, exactly as
// in the refinement kernels.
// ====================================================================

namespace {

__global__ void k_wait_probe(IrArgs a, int mode)
{
    __shared__ IrShared shs;
    if (threadIdx.x == 0) {
        shs.bid = (int)blockIdx.x;
        shs.G = (int)gridDim.x + 1;  // a block that does not exist
        shs.epoch = 0;
        shs.epoch2 = 0;
        shs.gepoch = 0;
        shs.ok = 1;
        shs.msg = a.msg;
        shs.msg2 = a.msg;
        shs.err = a.err;
        shs.limit = a.limit;
        shs.g2 = 0;
    }
    __syncthreads();
    if (mode == 0) {
        xbar<false>(&shs);
    } else {
        const GridBarrier gb{a.gcount, a.err, a.limit, gridDim.x + 1};
        grid_sync(gb, &shs.gepoch, &shs.ok);
    }
}

}  // namespace

extern "C" int spai_selftest_wait_timeout(int device, int mode, double limit_ms)
{
    if (mode != 0 && mode != 1) return SPAI_ERR_INVALID_ARG;
    if (!(limit_ms > 0.0) || limit_ms > 10000.0) return SPAI_ERR_INVALID_ARG;
    SPAI_CUDA_TRY(cudaSetDevice(device));
    constexpr int grid = 4;
    unsigned long long* msg = nullptr;
    int* err = nullptr;
    unsigned* gcount = nullptr;
    const size_t msg_bytes = sizeof(unsigned long long) * 2 * (grid + 1) * SLOT_WORDS;
    int rc = 0;
    if (cudaMalloc((void**)&msg, msg_bytes) != cudaSuccess || cudaMalloc((void**)&err, sizeof(int)) != cudaSuccess ||
        cudaMalloc((void**)&gcount, sizeof(unsigned)) != cudaSuccess)
        rc = SPAI_ERR_NO_MEMORY;
    if (!rc && (cudaMemset(msg, 0, msg_bytes) != cudaSuccess || cudaMemset(err, 0, sizeof(int)) != cudaSuccess ||
                cudaMemset(gcount, 0, sizeof(unsigned)) != cudaSuccess))
        rc = SPAI_ERR_CUDA;
    if (!rc) {
        IrArgs a;
        memset(&a, 0, sizeof(a));
        a.msg = msg;
        a.err = err;
        a.gcount = gcount;
        int clk_khz = device_attr_cached(cudaDevAttrClockRate, device);
        if (clk_khz <= 0) clk_khz = 2000000;
        a.limit = (long long)((double)clk_khz * limit_ms);
        k_wait_probe<<<grid, 32>>>(a, mode);
        int h = 0;
        if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess ||
            cudaMemcpy(&h, err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
            rc = SPAI_ERR_CUDA;
        else
            rc = h;  // SPAI_ERR_TIMEOUT when every wait gave up as designed
    }
    cudaFree(msg);
    cudaFree(err);
    cudaFree(gcount);
    return rc;
}

// ====================================================================
// Batched refinement (gmres_ir_solve_batch): many independent systems at
// once.  Cooperative launches of separate systems hardly overlap on the GPU
// (16 solves of an n = 4096 system: 111 ms one after another, 66-70 ms from 2
// or 4 host threads), while one such system keeps only 16 of 152 SMs busy.
// So every system gets a team of blocks that is one thread-block cluster
// (k_ir_local), and the systems of one team size are one launch whose
// clusters the hardware starts as SMs come free, larger systems first; the
// team sizes' launches run side by side on streams of their own.  A system's
// team size is a function of the system and the options alone (batch_team: about
// BATCH_ROWS_PER_BLOCK rows per block, fewer for scattered matrices, raised until a block's rows fit its
// shared memory, at most 16 blocks), so its result is the same whatever
// batch it is solved in.  Systems of more than BATCH_SOLO_N rows, which fill
// the GPU alone, run on a grid of their own (the single-system path).  All
// systems of a launch are prepared before it (their buffers coexist).  64
// systems of n 2e3..5e4 (one-reduction MGS, single), batch preparation included: 55-59 ms
// against 83-96 ms when the teams shared one cooperative launch and met through L2 (with
// staged inputs and one launch for all preparation since, 28 to 30 ms).
// ====================================================================

namespace {

// Rows per block of a batched system.  A batch is bound by the bytes each
// block streams per iteration, not by its grid-wide waits, so fewer and
// fuller blocks per system solve more systems at once: the refinement of the
// 512-system batch (n 2e3..5e4, one-reduction MGS) took 0.31 s of kernel
// time at 8192 rows per block against 0.41 s at 2048 and 0.69 s at 1024
// (the textbook MGS: 0.35 s, 0.76 s, 1.39 s).
// A scattered matrix (ir_scattered) is bound by the passes over its entries
// with a part of the input staged in shared memory each: fewer rows per block
// leave room for more of the input, so both the entries of a pass and the
// passes get fewer.  64 systems of n 2e3..5e4, half of them scattered: 26.4 ms of
// kernel time at 1024 rows, 27.0 at 2048, 27.5 at 3072, 33.1 at 4096, 59.4 at 8192;
// 3072 leaves the most SMs to other systems of those.
constexpr int64_t BATCH_ROWS_PER_BLOCK = 8192;
constexpr int64_t BATCH_SCATTERED_ROWS = 3072;
constexpr int64_t BATCH_SOLO_N = 65536;

int batch_team(int64_t n, bool scattered)
{
    const int64_t per = scattered ? BATCH_SCATTERED_ROWS : BATCH_ROWS_PER_BLOCK;
    return (int)std::max<int64_t>(1, std::min<int64_t>(16, (n + per / 2) / per));
}

// The preparation and the results of a batch: one launch for all systems each.
// 64 systems of n 2e3..5e4 in launches, copies and clears of their own (840
// launches, 600 copies) spent 7.7 ms beside the refinement kernels' 27.6; in these
// 0.9 ms.
struct BatchMat {  // a SELL copy to make
    int64_t n;
    const int64_t* rp;
    const int32_t* ci;
    const double* val;
    int64_t* off;
    unsigned long long* total;  // its entries
    int32_t* scol;
    void* sval;
};
struct BatchSys {
    int64_t n;
    const int64_t* rp;
    const int32_t* ci;
    const double* val;
    const double* b;
    const int64_t* prp;  // P (null: P = I) with its u_f values
    const int32_t* pci;
    const void* pvf;
    void* x;
    unsigned long long* norms;
    const IrResult* res;
    int4* ctrl;  // nctrl 16-byte words to clear
    int64_t nctrl;
};

// the slice offsets of matrix blockIdx.x and its entry count (1024 threads)
__global__ void k_batch_slices(const BatchMat* __restrict__ mats)
{
    const BatchMat m = mats[blockIdx.x];
    __shared__ int w32[1024];
    __shared__ int64_t part[32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t nsl = (m.n + 31) >> 5;
    int64_t carry = 0;
    for (int64_t base = 0; base < nsl; base += 1024) {
        __syncthreads();  // w32 and part are read
        for (int i = wid; i < 1024 && base + i < nsl; i += 32) {
            const int len = slice_width(m.n, m.rp, base + i);
            if (lane == 0) w32[i] = len * 32;
        }
        __syncthreads();
        const int64_t v = base + tid < nsl ? w32[tid] : 0;
        int64_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) part[wid] = x;
        __syncthreads();
        int64_t before = carry, all = 0;
        for (int w = 0; w < 32; w++) {
            if (w < wid) before += part[w];
            all += part[w];
        }
        if (base + tid < nsl) m.off[base + tid] = before + x - v;
        carry += all;
    }
    if (tid == 0) {
        m.off[nsl] = carry;
        *m.total = (unsigned long long)carry;
    }
}

// system blockIdx.y: its control words cleared, its norms (k_norms) and x0 (k_x0)
template <class S, class TU>
__global__ void k_batch_start(const BatchSys* __restrict__ sys)
{
    const BatchSys y = sys[blockIdx.y];
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t i = t0; i < y.nctrl; i += (int64_t)gridDim.x * blockDim.x) y.ctrl[i] = make_int4(0, 0, 0, 0);
    if (blockIdx.x * (int64_t)blockDim.x >= y.n) return;
    norms_rows(y.n, y.rp, y.ci, y.val, y.b, y.norms);
    x0_rows<S, TU>(y.n, y.prp, y.pci, (const S*)y.pvf, y.b, (TU*)y.x);
}

template <class TP>
__global__ void k_batch_fill(const BatchMat* __restrict__ mats)
{
    const BatchMat m = mats[blockIdx.y];
    sell_fill<TP>(m.n, m.rp, m.ci, m.val, m.off, m.scol, (TP*)m.sval);
}

// the results of system blockIdx.x, side by side
__global__ void k_batch_results(const BatchSys* __restrict__ sys, IrResult* __restrict__ res)
{
    static_assert(sizeof(IrResult) % 4 == 0, "copied in words");
    const int* from = (const int*)sys[blockIdx.x].res;
    for (int i = threadIdx.x; i < (int)(sizeof(IrResult) / 4); i += blockDim.x) ((int*)&res[blockIdx.x])[i] = from[i];
}

struct BatchRun {
    int device, num_sms;
    cudaStream_t s;
    const ir_opts* o;
    std::vector<IrJob>* jobs;
    const std::vector<int>* systems;  // by decreasing order
    std::vector<int>* grid_of;
    int* nl;
    float* ms_kernel;
    IrKernels K;
    int sg, sp;                // sizeof(u_g), sizeof(u_p)

    int tmax = 16;             // max_cluster

    // the system's team size (batch_team, at most tmax, raised until a block's rows fit its
    // shared memory; tmax + 1: they do not fit) and rows per block
    int team(const IrJob& jb, bool scattered, size_t dyn_max, int64_t* rows) const
    {
        int T = std::min(batch_team(jb.n, scattered), tmax);
        for (; T <= tmax; T++) {
            *rows = std::max<int64_t>(32, ((jb.n + T - 1) / T + 31) & ~int64_t(31));
            if (ir_pick_smem(*rows, jb.kmax, 0, o->orth, dyn_max, sg, sp, 0).bytes <= dyn_max) break;
        }
        return T;
    }

    int run()
    {
        const void* kern = K.local;
        size_t dyn_max = 0;
        SPAI_CUDA_TRY(allow_max_dynamic_smem_ptr(kern, &dyn_max));
        std::vector<IrJob>& J = *jobs;
        const std::vector<int>& order = *systems;
        const int count = (int)order.size();
        int rc = 0;
        // preparation without a wait per system: buffers, SELL offsets, norms and x0
        // for all systems, then one copy of every SELL size and norm to the host,
        // then the SELL fills
        std::set<spai_precond> building;
        std::vector<BatchMat> mats;
        std::vector<BatchSys> sys(count);
        std::vector<SellMat*> sells;
        std::vector<IrResult> res(count);
        BatchMat* d_mats = nullptr;
        BatchSys* d_sys = nullptr;
        unsigned long long* d_slots = nullptr;  // per system the norms (k_norms), at 3 and 4 A's and P's SELL entries
        IrResult* d_res = nullptr;
        // (the tables on the host are sources of copies: none of them may go before a wait)
        auto release = [&]() {
            if (cudaStreamSynchronize(s) != cudaSuccess) cudaGetLastError();
            dev_free(d_mats, s);
            dev_free(d_sys, s);
            dev_free(d_slots, s);
            dev_free(d_res, s);
        };
        // a preconditioner's SELL copy counts as built once its offsets exist: on
        // failure the copies this batch started are dropped again
        auto drop_started = [&]() {
            for (spai_precond P : building) sell_free(sell_cache(P, o->up), s);
        };
        auto upload = [&](void* to, const void* from, size_t bytes) {
            if (!rc && bytes && cudaMemcpyAsync(to, from, bytes, cudaMemcpyHostToDevice, s) != cudaSuccess) rc = SPAI_ERR_CUDA;
        };
        const size_t nslot = 6 * (size_t)count;
        rc = dev_alloc((void**)&d_slots, sizeof(unsigned long long) * nslot, s);
        if (!rc) rc = dev_alloc((void**)&d_mats, sizeof(BatchMat) * 2 * count, s);
        if (!rc) rc = dev_alloc((void**)&d_sys, sizeof(BatchSys) * count, s);
        if (!rc) rc = dev_alloc((void**)&d_res, sizeof(IrResult) * count, s);
        if (!rc && cudaMemsetAsync(d_slots, 0, sizeof(unsigned long long) * nslot, s) != cudaSuccess) rc = SPAI_ERR_CUDA;
        int64_t nmax = 1;
        for (int i = 0; i < count && !rc; i++) {
            IrJob& jb = J[order[i]];
            const DevCsr& A = *jb.A;
            nmax = std::max(nmax, jb.n);
            unsigned long long* slot = d_slots + 6 * (size_t)i;
            auto start = [&](const int64_t* rp, const int32_t* ci, const double* val, SellMat* m, unsigned long long* total) {
                rc = dev_alloc((void**)&m->off, sizeof(int64_t) * (((jb.n + 31) >> 5) + 1), s);
                mats.push_back(BatchMat{jb.n, rp, ci, val, m->off, total, nullptr, nullptr});
                sells.push_back(m);
            };
            rc = ir_job_alloc(jb, s, o, false);
            if (!rc) start(A.rowptr, A.col, A.val, &jb.As, slot + 3);
            if (!rc && jb.P) {
                SellMat* cache = sell_cache(jb.P, o->up);
                if (!cache->off) {
                    building.insert(jb.P);
                    start(jb.P->rowptr, jb.P->col, jb.P->val, cache, slot + 4);
                }
                jb.Ps = cache;
            }
            sys[i] = BatchSys{jb.n, A.rowptr, A.col, A.val, jb.b, jb.P ? jb.P->rowptr : nullptr, jb.P ? jb.P->col : nullptr,
                              jb.P ? jb.P->val_uf : nullptr, jb.x, slot, jb.res, (int4*)jb.arena,
                              (int64_t)(jb.ctrl / 16)};
        }
        upload(d_mats, mats.data(), sizeof(BatchMat) * mats.size());
        upload(d_sys, sys.data(), sizeof(BatchSys) * count);
        const int nmat = (int)mats.size();
        // (blocks without rows of their system leave at once)
        const unsigned gx = (unsigned)std::min<int64_t>((nmax + 255) / 256, (int64_t)num_sms * 32);
        // systems a launch (the grid's y limit)
        constexpr int YMAX = 32768;
        if (!rc) {
            k_batch_slices<<<nmat, 1024, 0, s>>>(d_mats);
            for (int i0 = 0; i0 < count; i0 += YMAX) {
                const dim3 g(gx, (unsigned)std::min(YMAX, count - i0));
#define START(S, TU) k_batch_start<S, TU><<<g, 256, 0, s>>>(d_sys + i0)
                if (o->u == SPAI_SINGLE) {
                    if (o->uf == SPAI_HALF) START(__half, float);
                    else if (o->uf == SPAI_SINGLE) START(float, float);
                    else START(double, float);
                } else {
                    if (o->uf == SPAI_HALF) START(__half, double);
                    else if (o->uf == SPAI_SINGLE) START(float, double);
                    else START(double, double);
                }
#undef START
                (*nl)++;
            }
            (*nl)++;
            if (cudaGetLastError() != cudaSuccess) rc = SPAI_ERR_CUDA;
        }
        std::vector<unsigned long long> hs(nslot, 0);
        if (!rc && cudaMemcpyAsync(hs.data(), d_slots, sizeof(unsigned long long) * nslot, cudaMemcpyDeviceToHost, s) !=
                       cudaSuccess)
            rc = SPAI_ERR_CUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess && !rc) rc = SPAI_ERR_CUDA;
        for (int i = 0; i < count && !rc; i++) {
            IrJob& jb = J[order[i]];
            const unsigned long long* h = hs.data() + 6 * (size_t)i;
            for (int k = 0; k < 3; k++) jb.h_norms[k] = h[k];
            jb.scattered = ir_scattered(jb.n, jb.A->nnz, h[5]);
        }
        for (int i = 0; i < nmat && !rc; i++) {
            SellMat* m = sells[i];
            const int64_t total = (int64_t)hs[(size_t)(mats[i].total - d_slots)];
            m->prec = o->up;
            m->nnz = total;
            rc = dev_alloc((void**)&m->col, sizeof(int32_t) * std::max<int64_t>(total, 1), s);
            if (!rc) rc = dev_alloc(&m->val, (size_t)prec_bytes(o->up) * std::max<int64_t>(total, 1), s);
            mats[i].scol = m->col;
            mats[i].sval = m->val;
        }
        upload(d_mats, mats.data(), sizeof(BatchMat) * mats.size());
        for (int i0 = 0; i0 < nmat && !rc; i0 += YMAX) {
            const dim3 g(std::max(1u, std::min(gx, 64u)), (unsigned)std::min(YMAX, nmat - i0));
            if (o->up == SPAI_HALF) k_batch_fill<__half><<<g, 256, 0, s>>>(d_mats + i0);
            else if (o->up == SPAI_SINGLE) k_batch_fill<float><<<g, 256, 0, s>>>(d_mats + i0);
            else k_batch_fill<double><<<g, 256, 0, s>>>(d_mats + i0);
            (*nl)++;
            if (cudaGetLastError() != cudaSuccess) rc = SPAI_ERR_CUDA;
        }
        if (rc) { drop_started(); release(); return rc; }
        // classes: (team size, threads), larger teams first, systems by decreasing order
        std::map<std::pair<int, int>, std::vector<int>> byteam;
        for (int i : order) {
            int64_t rb = 0;
            const int T = team(J[i], J[i].scattered, dyn_max, &rb);
            if (T > tmax) { release(); return SPAI_ERR_INTERNAL; }  // (checked before: fewer rows per block always fit)
            byteam[{T, ir_block_threads(rb, o->orth)}].push_back(i);
            (*grid_of)[i] = T;
        }
        const std::vector<std::pair<std::pair<int, int>, std::vector<int>>> classes(byteam.rbegin(), byteam.rend());
        const int ncls = (int)classes.size();
        std::vector<int> cs(ncls + 1, 0);
        // arguments class by class, every system prepared for its class's team size
        std::vector<IrArgs> h;
        std::vector<size_t> smem(ncls, 0);
        for (int c = 0; c < ncls; c++) {
            const int T = classes[c].first.first;
            for (int i : classes[c].second) {
                IrJob& jb = J[i];
                ir_job_args(jb, device, o);
                IrArgs& a = jb.a;
                a.G = T;
                a.scat = jb.scattered ? 1 : 0;
                a.rb = std::max<int64_t>(32, ((jb.n + T - 1) / T + 31) & ~int64_t(31));
                a.g2 = 0;
                const IrSmem m = ir_pick_smem(a.rb, a.kmax, 0, a.orth, dyn_max, sg, sp, jb.scattered ? jb.n : 0);
                a.jl = m.jl;
                a.nq = m.nq;
                a.xcap = m.xcap;
                a.xs_off = (int)m.xs_off;
                smem[c] = std::max(smem[c], m.bytes);
                h.push_back(a);
            }
            cs[c + 1] = (int)h.size();
            if (smem[c] > dyn_max) { release(); return SPAI_ERR_UNSUPPORTED; }
        }
        IrArgs* d_args = nullptr;
        rc = dev_alloc((void**)&d_args, sizeof(IrArgs) * count, s);
        if (!rc && cudaMemcpyAsync(d_args, h.data(), sizeof(IrArgs) * count, cudaMemcpyHostToDevice, s) != cudaSuccess)
            rc = SPAI_ERR_CUDA;
        // one launch per class, the first (largest teams) on s, the others on streams of
        // their own between two events of s
        cudaEvent_t k0 = nullptr, k1 = nullptr, kc = nullptr;
        std::vector<cudaStream_t> side;
        if (!rc && (cudaEventCreate(&k0) != cudaSuccess || cudaEventCreate(&k1) != cudaSuccess ||
                    cudaEventCreateWithFlags(&kc, cudaEventDisableTiming) != cudaSuccess))
            rc = SPAI_ERR_CUDA;
        if (!rc && cudaEventRecord(k0, s) != cudaSuccess) rc = SPAI_ERR_CUDA;
        for (int c = 0; c < ncls && !rc; c++) {
            const int T = classes[c].first.first;
            cudaStream_t sc = s;
            if (c > 0) {
                if (cudaStreamCreateWithFlags(&sc, cudaStreamNonBlocking) != cudaSuccess) { rc = SPAI_ERR_CUDA; break; }
                side.push_back(sc);
                if (cudaStreamWaitEvent(sc, k0, 0) != cudaSuccess) { rc = SPAI_ERR_CUDA; break; }
            }
            const IrArgs* pa = d_args + cs[c];
            int Tv = T;
            void* args[] = {(void*)&h[cs[c]], (void*)&pa, (void*)&Tv};
            const cudaError_t e = launch_clusters(kern, T * (cs[c + 1] - cs[c]), T, classes[c].first.second, smem[c], args, sc);
            if (e != cudaSuccess) {
                spai_set_last_cuda_error(e);
                cudaGetLastError();
                rc = SPAI_ERR_CUDA;
            }
            (*nl)++;
        }
        for (cudaStream_t sc : side) {
            // s goes on (and frees what the launches use) only after every class
            if (cudaEventRecord(kc, sc) != cudaSuccess || cudaStreamWaitEvent(s, kc, 0) != cudaSuccess) {
                cudaStreamSynchronize(sc);
                if (!rc) rc = SPAI_ERR_CUDA;
            }
        }
        if (k1) cudaEventRecord(k1, s);
        if (!rc) {
            // (x as it is ready, a launch of its system's size each; the results together)
            for (int i = 0; i < count; i++) ir_job_x(J[order[i]], num_sms, s, o, nl);
            k_batch_results<<<count, 128, 0, s>>>(d_sys, d_res);
            (*nl)++;
            if (cudaGetLastError() != cudaSuccess) rc = SPAI_ERR_CUDA;
        }
        if (!rc && cudaMemcpyAsync(res.data(), d_res, sizeof(IrResult) * count, cudaMemcpyDeviceToHost, s) != cudaSuccess)
            rc = SPAI_ERR_CUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess && !rc) rc = SPAI_ERR_CUDA;
        for (int i = 0; i < count && !rc; i++) J[order[i]].h = res[i];
        if (!rc) {
            float ms = 0.f;
            cudaEventElapsedTime(&ms, k0, k1);
            *ms_kernel += ms;
        }
        if (k0) cudaEventDestroy(k0);
        if (k1) cudaEventDestroy(k1);
        if (kc) cudaEventDestroy(kc);
        for (cudaStream_t sc : side) cudaStreamDestroy(sc);
        dev_free(d_args, s);
        release();
        return rc;
    }
};

}  // namespace

int gmres_ir_batch_dev(int device, int num_sms, cudaStream_t s, int count, const DevCsr* A, const spai_precond* P,
                       const double* const* b, double* const* xout, const ir_opts* o, ir_stats* st, int* status)
{
    int rc = ir_check_opts(o);
    if (rc) return rc;
    if (count < 0 || (count > 0 && (!A || !b || !xout))) return SPAI_ERR_INVALID_ARG;
    std::vector<IrJob> jobs(count);
    for (int i = 0; i < count; i++) {
        spai_precond Pi = P ? P[i] : nullptr;
        if (Pi && (Pi->uf != o->uf || Pi->n != A[i].n)) return SPAI_ERR_INVALID_ARG;
        IrJob& J = jobs[i];
        J.A = &A[i]; J.P = Pi; J.b = b[i]; J.xout = xout[i]; J.n = A[i].n; J.imax = o->ir_max_steps;
        rc = ir_job_kmax(A[i].n, o, &J.kmax);
        if (rc) return rc;
    }
    std::vector<int> order(count);
    for (int i = 0; i < count; i++) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return jobs[x].n > jobs[y].n; });
    IrKernels K;
    rc = ir_kernels(o->u, o->ug, o->up, o->ur, o->orth, &K);
    if (rc) return rc;
    size_t dyn_max = 0;
    SPAI_CUDA_TRY(allow_max_dynamic_smem_ptr(K.local, &dyn_max));
    std::vector<int> grid_of(count, 0), team_run, solo;
    int nl = 0;
    float ms_kernel = 0.f;
    BatchRun B{device, num_sms, s, o, &jobs, &team_run, &grid_of, &nl, &ms_kernel, K, prec_bytes(o->ug), prec_bytes(o->up)};
    B.tmax = max_cluster(K.local, dyn_max);
    for (int i : order) {
        int64_t rb = 0;
        if (jobs[i].n > BATCH_SOLO_N || B.team(jobs[i], false, dyn_max, &rb) > B.tmax) solo.push_back(i);
        else team_run.push_back(i);
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    SPAI_CUDA_TRY(cudaEventCreate(&e0));
    SPAI_CUDA_TRY(cudaEventCreate(&e1));
    cudaEventRecord(e0, s);
    if (!rc && !team_run.empty()) rc = B.run();
    for (int i : solo) {
        if (rc) break;
        IrJob& J = jobs[i];
        rc = ir_job_prepare(J, num_sms, s, o, &nl);
        if (!rc) {
            ir_job_args(J, device, o);
            cudaEvent_t k0 = nullptr, k1 = nullptr;
            if (cudaEventCreate(&k0) != cudaSuccess || cudaEventCreate(&k1) != cudaSuccess) rc = SPAI_ERR_CUDA;
            if (!rc) cudaEventRecord(k0, s);
            if (!rc) rc = launch_ir(J.a, K, prec_bytes(o->ug), prec_bytes(o->up), J.scattered, ir_job_entries(J),
                                    num_sms, s, &grid_of[i]);
            if (!rc) {
                cudaEventRecord(k1, s);
                nl++;
                rc = ir_job_collect(J, num_sms, s, o, &nl);
            }
            if (!rc && cudaStreamSynchronize(s) != cudaSuccess) rc = SPAI_ERR_CUDA;
            if (!rc) {
                float ms = 0.f;
                cudaEventElapsedTime(&ms, k0, k1);
                ms_kernel += ms;
            }
            if (k0) cudaEventDestroy(k0);
            if (k1) cudaEventDestroy(k1);
        }
    }
    cudaEventRecord(e1, s);
    if (cudaStreamSynchronize(s) != cudaSuccess && rc >= 0) rc = SPAI_ERR_CUDA;
    float ms_all = 0.f;
    if (rc >= 0) cudaEventElapsedTime(&ms_all, e0, e1);
    int worst = 0;
    for (int i = 0; i < count; i++) {
        int ri = rc < 0 ? rc : ir_job_result(jobs[i], o, st ? &st[i] : nullptr);
        if (status) status[i] = ri;
        if (ri < 0 && worst >= 0) worst = ri;
        else if (ri > 0 && worst == 0) worst = ri;
        if (st && rc >= 0) {
            st[i].ms_ir = ms_all;
            st[i].ms_kernel = ms_kernel;
            st[i].launches = nl;
            st[i].grid = grid_of[i];
        }
        ir_job_free(jobs[i], s);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaStreamSynchronize(s);
    return rc < 0 ? rc : worst;
}

// ====================================================================
// Allocation-free refinement solve (gmres_ir_solve_noalloc).
//
// For callers that must not allocate device memory: real-time loops (the
// allocator's latency is unbounded and cudaFree synchronises the device),
// hosts that own their memory budget exactly, or runtimes that forbid the
// CUDA allocator after start-up.  The refinement
// scratch (SELL copies of A and P, the Krylov basis, the residual and
// iterate, the exchange slots) lives in one file-scope device array of
// SPAI_NOALLOC_SCRATCH_BYTES that every GPU loading this library holds
// until exit.  Host code never passes the array's name to a kernel (on the
// host it is only a stand-in symbol): its device address is looked up once
// per device with cudaGetSymbolAddress, on the first call made on that
// device.
// ====================================================================

// (beyond that, room for w's padding rows and the control words that only this build needs)
constexpr size_t NOALLOC_BYTES = (size_t)SPAI_NOALLOC_SCRATCH_BYTES + 512;
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

namespace {

std::mutex g_noalloc_mu;
unsigned char* g_noalloc_base[128] = {nullptr};

int noalloc_base(int dev, unsigned char** out)
{
    if (dev < 0 || dev >= 128) return SPAI_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_base[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            spai_set_last_cuda_error(e);
            return SPAI_ERR_CUDA;
        }
        g_noalloc_base[dev] = (unsigned char*)p;
    }
    *out = g_noalloc_base[dev];
    return 0;
}

// exclusive scan of ns counts into out[0..ns], one block
__global__ void k_scan_one_block(int64_t ns, const int32_t* __restrict__ in, int64_t* __restrict__ out)
{
    __shared__ int64_t wsum[32];
    __shared__ int64_t carry;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < ns; base += blockDim.x) {
        const int64_t i = base + threadIdx.x;
        const int64_t v = i < ns ? in[i] : 0;
        int64_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int64_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[w] = x;
        __syncthreads();
        if (w == 0) {
            int64_t t = lane < nw ? wsum[lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int64_t y = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += y;
            }
            if (lane < nw) wsum[lane] = t;
        }
        __syncthreads();
        const int64_t pre = carry + (w > 0 ? wsum[w - 1] : 0) + x - v;
        if (i < ns) out[i] = pre;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = pre + v;
        __syncthreads();
    }
    if (threadIdx.x == 0) out[ns] = carry;
}

// x0 = P b in u_f with P's float64 values rounded to u_f on the fly
template <class S, class TU>
__global__ void k_x0_dbl(int64_t n, const int64_t* __restrict__ prp, const int32_t* __restrict__ pci,
                         const double* __restrict__ pv, const double* __restrict__ b, TU* __restrict__ x)
{
    typedef typename Compute<S>::T C;
    for (int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; row < n; row += (int64_t)gridDim.x * blockDim.x) {
        C acc = C(0);
        if (prp) {
            for (int64_t q = prp[row]; q < prp[row + 1]; q++)
                acc = fma(to_c(from_d<S>(pv[q])), to_c(from_d<S>(b[pci[q]])), acc);
        } else {
            acc = to_c(from_d<S>(b[row]));
        }
        x[row] = (TU)to_c(from_d<S>((double)acc));
    }
}

struct Carve {
    unsigned char* base;
    size_t off, cap;
    void* take(size_t bytes)
    {
        off = (off + 255) & ~size_t(255);
        if (off + bytes > cap) return nullptr;
        void* p = base + off;
        off += bytes;
        return p;
    }
};

}  // namespace

extern "C" int gmres_ir_solve_noalloc(const spai_csr* A, const spai_csr* P, const double* b, double* xout,
                                      const ir_opts* o, void* cuda_stream, ir_stats* st)
{
    if (!A || !b || !xout || !o) return SPAI_ERR_INVALID_ARG;
    if (!A->on_device || (P && !P->on_device)) return SPAI_ERR_INVALID_ARG;
    if (A->n < 1 || A->nnz < 0 || !A->rowptr || !A->col || !A->val) return SPAI_ERR_INVALID_ARG;
    if (P && (P->n != A->n || P->nnz < 0 || !P->rowptr || !P->col || !P->val)) return SPAI_ERR_INVALID_ARG;
    if (A->n > INT32_MAX) return SPAI_ERR_UNSUPPORTED;
    // the options of gmres_ir_solve, less half Krylov storage
    if (o->ug == SPAI_HALF || o->up == SPAI_HALF) return SPAI_ERR_UNSUPPORTED;
    {
        const int rc = ir_check_opts(o);
        if (rc) return rc;
    }
    const int64_t n = A->n;
    int kmax = o->gmres_max_it > 0 ? o->gmres_max_it : (int)std::min<int64_t>(n, 500);
    if (kmax > n) kmax = (int)n;
    if (kmax > KMAX_LIMIT) return SPAI_ERR_UNSUPPORTED;
    if (kmax < 1) kmax = 1;
    const int imax = o->ir_max_steps;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    int device = 0, num_sms = 0;
    SPAI_CUDA_TRY(cudaGetDevice(&device));
    SPAI_CUDA_TRY(cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, device));
    unsigned char* base = nullptr;
    int rc = noalloc_base(device, &base);
    if (rc) return rc;

    const int su = prec_bytes(o->u), sg = prec_bytes(o->ug), sp = prec_bytes(o->up);
    const int64_t ldv = (n + 31) & ~int64_t(31);
    const int64_t nsl = (n + 31) >> 5;
    Carve cv{base, 0, NOALLOC_BYTES};
    const size_t msg_bytes = sizeof(unsigned long long) * 4 * MAX_GRID * SLOT_WORDS;
    // control words: err[2], out[2], the CSR check flags, its[imax + 1], nbe[imax + 1], the norms
    const size_t ctrl_bytes = sizeof(int) * 6 + sizeof(int) * (imax + 1) + sizeof(double) * (imax + 1) +
                              sizeof(unsigned long long) * 6 + 64;
    unsigned long long* msg = (unsigned long long*)cv.take(msg_bytes);
    unsigned char* ctrl = (unsigned char*)cv.take(ctrl_bytes);
    void* x = cv.take((size_t)su * n);
    void* r = cv.take((size_t)su * n);
    void* wbuf = cv.take((size_t)sg * ldv);
    void* tbuf = cv.take((size_t)sp * n);
    void* V = cv.take((size_t)sg * ldv * (kmax + 1));
    double* R = (double*)cv.take(sizeof(double) * (size_t)(kmax + 1) * kmax);
    int64_t* aoff = (int64_t*)cv.take(sizeof(int64_t) * (nsl + 1));
    int32_t* aw = (int32_t*)cv.take(sizeof(int32_t) * nsl);
    int64_t* poff = P ? (int64_t*)cv.take(sizeof(int64_t) * (nsl + 1)) : nullptr;
    int32_t* pw = P ? (int32_t*)cv.take(sizeof(int32_t) * nsl) : nullptr;
    // CGS2: the partial dot products of every block and the counter of their barrier
    // (scalars in u_g's arithmetic type, as the allocating path sizes them)
    void* pvec = o->orth ? cv.take((size_t)ir_scalar_bytes(sg) * (2 * MAX_GRID + (o->orth == 2 ? 2 : 0)) * (kmax + 1))
                         : nullptr;
    void* Lrows = o->orth == 2 ? cv.take((size_t)ir_scalar_bytes(sg) * ((size_t)(kmax + 1) * kmax / 2 + 1)) : nullptr;
    double* gpub = o->orth == 2 ? (double*)cv.take(sizeof(double) * (kmax + 2)) : nullptr;
    if (!msg || !ctrl || !x || !r || !wbuf || !tbuf || !V || !R || !aoff || !aw || (P && (!poff || !pw)) ||
        (o->orth && !pvec) || (o->orth == 2 && (!Lrows || !gpub)))
        return SPAI_ERR_UNSUPPORTED;  // the problem does not fit the fixed scratch
    int* err = (int*)ctrl;
    int* outv = err + 2;
    int* csrf = outv + 2;                   // structural check flags of A and P
    unsigned* gcount = (unsigned*)(csrf + 1);
    int* its = csrf + 2;
    double* nbe = (double*)(((uintptr_t)(its + imax + 1) + 7) & ~uintptr_t(7));
    unsigned long long* norms = (unsigned long long*)(nbe + imax + 1);
    // the array keeps the previous call's contents: clear what must start at zero
    SPAI_CUDA_TRY(cudaMemsetAsync(msg, 0, msg_bytes, s));
    SPAI_CUDA_TRY(cudaMemsetAsync(ctrl, 0, ctrl_bytes, s));
    const int tb = 256;
    const int gb = (int)std::max<int64_t>(1, std::min<int64_t>((n + tb - 1) / tb, (int64_t)num_sms * 32));
    const int gs = (int)std::max<int64_t>(1, std::min<int64_t>((nsl * 32 + tb - 1) / tb, (int64_t)num_sms * 16));
    int nl = 0;
    // the structural check of both device CSRs (rowptr order and range, columns in
    // [0, n) and ascending, no empty row of A) before any kernel indexes with them;
    // its flags come back with the SELL sizes below
    {
        const int gc = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)num_sms * 8));
        k_csr_check<<<gc, 256, 0, s>>>(n, A->nnz, A->rowptr, A->col, csrf, 0);
        nl++;
        if (P) {
            // rows of P may be empty (a zero row of P is a valid preconditioner row)
            k_csr_check<<<gc, 256, 0, s>>>(n, P->nnz, P->rowptr, P->col, csrf, 1);
            nl++;
        }
        SPAI_CUDA_TRY(cudaGetLastError());
        int h_csr = 0;
        SPAI_CUDA_TRY(cudaMemcpyAsync(&h_csr, csrf, sizeof(int), cudaMemcpyDeviceToHost, s));
        SPAI_CUDA_TRY(cudaStreamSynchronize(s));
        if (h_csr & 1) return SPAI_ERR_INVALID_ARG;
        if (h_csr & 2) return SPAI_ERR_ZERO_ROW;
    }
    k_sell_width<<<gs, tb, 0, s>>>(n, A->rowptr, aw);
    k_scan_one_block<<<1, 1024, 0, s>>>(nsl, aw, aoff);
    nl += 2;
    if (P) {
        k_sell_width<<<gs, tb, 0, s>>>(n, P->rowptr, pw);
        k_scan_one_block<<<1, 1024, 0, s>>>(nsl, pw, poff);
        nl += 2;
    }
    int64_t tot[2] = {0, 0};
    SPAI_CUDA_TRY(cudaMemcpyAsync(&tot[0], aoff + nsl, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    if (P) SPAI_CUDA_TRY(cudaMemcpyAsync(&tot[1], poff + nsl, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    SPAI_CUDA_TRY(cudaStreamSynchronize(s));
    int32_t* acol = (int32_t*)cv.take(sizeof(int32_t) * std::max<int64_t>(tot[0], 1));
    void* aval = cv.take((size_t)sp * std::max<int64_t>(tot[0], 1));
    int32_t* pcol = P ? (int32_t*)cv.take(sizeof(int32_t) * std::max<int64_t>(tot[1], 1)) : nullptr;
    void* pval = P ? cv.take((size_t)sp * std::max<int64_t>(tot[1], 1)) : nullptr;
    if (!acol || !aval || (P && (!pcol || !pval))) return SPAI_ERR_UNSUPPORTED;
    if (o->up == SPAI_SINGLE) {
        k_sell_fill<float><<<gs, tb, 0, s>>>(n, A->rowptr, A->col, A->val, aoff, acol, (float*)aval);
        if (P) k_sell_fill<float><<<gs, tb, 0, s>>>(n, P->rowptr, P->col, P->val, poff, pcol, (float*)pval);
    } else {
        k_sell_fill<double><<<gs, tb, 0, s>>>(n, A->rowptr, A->col, A->val, aoff, acol, (double*)aval);
        if (P) k_sell_fill<double><<<gs, tb, 0, s>>>(n, P->rowptr, P->col, P->val, poff, pcol, (double*)pval);
    }
    nl += P ? 2 : 1;
    k_norms<<<gb, tb, 0, s>>>(n, A->rowptr, A->col, A->val, b, norms);
    nl++;
    {
        const int64_t* prp = P ? P->rowptr : nullptr;
        const int32_t* pci = P ? P->col : nullptr;
        const double* pvd = P ? P->val : nullptr;
#define X0D(S, TU) k_x0_dbl<S, TU><<<gb, tb, 0, s>>>(n, prp, pci, pvd, b, (TU*)x)
        if (o->u == SPAI_SINGLE) {
            if (o->uf == SPAI_HALF) X0D(__half, float);
            else if (o->uf == SPAI_SINGLE) X0D(float, float);
            else X0D(double, float);
        } else {
            if (o->uf == SPAI_HALF) X0D(__half, double);
            else if (o->uf == SPAI_SINGLE) X0D(float, double);
            else X0D(double, double);
        }
#undef X0D
        nl++;
    }
    SPAI_CUDA_TRY(cudaGetLastError());
    unsigned long long h_norms[6] = {0, 0, 0, 0, 0, 0};
    SPAI_CUDA_TRY(cudaMemcpyAsync(h_norms, norms, sizeof(h_norms), cudaMemcpyDeviceToHost, s));
    SPAI_CUDA_TRY(cudaStreamSynchronize(s));
    IrArgs a;
    memset(&a, 0, sizeof(a));
    double anorm, bnorm;
    {
        long long t0 = (long long)h_norms[0], t1 = (long long)h_norms[1];
        memcpy(&anorm, &t0, 8);
        memcpy(&bnorm, &t1, 8);
    }
    const int q = (int)h_norms[2];
    const bool scattered = ir_scattered(n, A->nnz, h_norms[5]);
    a.n = n;
    a.A.off = aoff; a.A.col = acol; a.A.val = aval;
    if (P) { a.P.off = poff; a.P.col = pcol; a.P.val = pval; }
    a.arp = A->rowptr; a.aci = A->col; a.aval = A->val;
    a.b = b; a.x = x; a.r = r; a.wbuf = wbuf; a.tbuf = tbuf; a.V = V; a.ldv = ldv; a.R = R; a.msg = msg;
    a.msg2 = msg + 2 * MAX_GRID * SLOT_WORDS;
    a.err = err;
    int clk_khz = device_attr_cached(cudaDevAttrClockRate, device);
    if (clk_khz <= 0) clk_khz = 2000000;
    a.limit = (long long)clk_khz * 1000LL * 4;
    a.anorm = anorm; a.bnorm = bnorm; a.tau = o->tau;
    a.stop_tol = ir_stop_tol(o, q);
    a.kmax = kmax; a.imax = imax; a.stop_rule = o->stop;
    a.its = its; a.nbe = nbe; a.out = outv;
    a.side = o->side;
    a.orth = o->orth; a.pvec = pvec; a.gcount = gcount; a.L = Lrows; a.gpub = gpub;
    int grid = 0;
    {
        IrKernels K;
        rc = ir_kernels(o->u, o->ug, o->up, o->ur, o->orth, &K);
        if (!rc) rc = launch_ir(a, K, prec_bytes(o->ug), prec_bytes(o->up), scattered,
                                std::max(tot[0], tot[1]), num_sms, s, &grid);
    }
    if (rc) return rc;
    nl++;
    if (o->u == SPAI_SINGLE) k_to_double<float><<<gb, tb, 0, s>>>(n, (const float*)x, xout);
    else k_to_double<double><<<gb, tb, 0, s>>>(n, (const double*)x, xout);
    nl++;
    SPAI_CUDA_TRY(cudaGetLastError());
    int h_out[2] = {0, 0}, h_err = 0;
    SPAI_CUDA_TRY(cudaMemcpyAsync(h_out, outv, sizeof(h_out), cudaMemcpyDeviceToHost, s));
    SPAI_CUDA_TRY(cudaMemcpyAsync(&h_err, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    if (st) {
        memset(st, 0, sizeof(*st));
        SPAI_CUDA_TRY(cudaMemcpyAsync(st->its, its, sizeof(int) * imax, cudaMemcpyDeviceToHost, s));
        SPAI_CUDA_TRY(cudaMemcpyAsync(st->nbe, nbe, sizeof(double) * (imax + 1), cudaMemcpyDeviceToHost, s));
    }
    SPAI_CUDA_TRY(cudaStreamSynchronize(s));
    if (h_err) return h_err;
    if (st) {
        st->steps = h_out[0];
        st->flags = h_out[1];
        for (int i = 0; i < st->steps; i++) st->total_its += st->its[i];
        for (int i = st->steps + 1; i <= SPAI_IR_MAX_STEPS; i++) st->nbe[i] = 0.0;
        st->final_nbe = st->nbe[st->steps];
        st->launches = nl;
        st->grid = grid;
        st->nnz_P = P ? P->nnz : 0;
    }
    if (h_out[1] & 8) return SPAI_ERR_NONFINITE;
    if (!(h_out[1] & 1) && o->stop != IR_STOP_FIXED) return SPAI_WARN_NOT_CONVERGED;
    return 0;
}
