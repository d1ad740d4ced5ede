// The refinement kernel of Algorithm 3 (SPAI-GMRES-IR): device code shared
// by the per-precision instantiation units (gmres_ir_k_*.cu) and the host
// code in gmres_ir.cu.  The whole refinement loop of one system is ONE
// persistent kernel: k_ir on a co-resident grid, k_ir_local on one block or one
// thread-block cluster per system (small systems, and many at once).  Each block owns a contiguous slice of
// rows, keeps its slice of the Arnoldi vector w in shared memory, and meets
// the other blocks only at bounded grid-wide exchanges: for every grid-wide dot
// product the blocks leave partials and every block adds them the same way (single:
// in one order; double: as integers on one exponent, which no order changes), so all
// blocks hold bit-identical scalars and
// take identical control-flow decisions (GMRES convergence, refinement stop)
// without another barrier.  The Givens rotations, H, g and y are double
// precision in every block.
//
// Template parameters: TU, TG, TP the storage types of u, u_g, u_p (u_g and u_p
// may be half, for the one-reduction MGS only: vectors and matrix values are
// stored in half, every operation on them is binary32); RM = 2
// for the double-double residual (u_r = quad); LS selects the one-reduction
// MGS (orth 2), compiled as its own kernel so that the MGS / CGS2 kernel
// keeps its register allocation.
#pragma once

#include <algorithm>
#include <climits>
#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace spai {


constexpr int KMAX_LIMIT = 1024;
constexpr int MAX_GRID = 160;   // exchange slots are polled by one warp, SPL slots per lane
constexpr int SPL = (MAX_GRID + 31) / 32;
constexpr int MAX_CLUSTER = 16;  // blocks of a system that runs as one thread-block cluster
constexpr int SLOT_WORDS = 16;  // one 128-byte line per block and parity (up to 4 words used)
constexpr int PF = 4;           // rows per thread whose next basis entries are prefetched
// Grids from this size run the Gram-Schmidt rounds in a group.  Us per iteration, all
// blocks / group, 3D: double 96 blocks 44.0 / 46.6, 112 blocks 51.6 / 47.3, 143 blocks 53.9 / 49.2
// (2D, 77 blocks 45.9 / 48.7); single 112 blocks 23.2 / 24.2, 143 blocks 24.8 / 25.1, 150 blocks
// (n = 143350) 36.7 / 36.4.
inline int mgs_group_min_grid(int sg) { return sg == 8 ? 112 : 148; }
// one-reduction MGS: from this many partials (2 (j + 1) values x blocks) the sums over blocks are
// split among the blocks (one more exchange round) instead of every block reading all of them
constexpr int IR_DIST_MIN = 32768;

// SELL-32: rows in slices of 32; slice s stores its entries column-major
// (entry c of row 32s+l at off[s] + 32c + l), padded to the slice's longest
// row with (col = own row, val = 0).  Loads of one entry slot by a warp are
// one contiguous 128-byte line.
struct Sell {
    const int64_t* off;  // nslices + 1 element offsets
    const int32_t* col;
    const void* val;     // precision u_p
};

struct IrArgs {
    int64_t n;
    int64_t rb;                 // rows per block (multiple of 32)
    Sell A, P;                  // P.off == nullptr: P = I
    const int64_t* arp;         // A in CSR, float64 (residual)
    const int32_t* aci;
    const double* aval;
    const double* b;
    void* x;                    // n, precision u
    void* r;                    // n, precision u
    void* wbuf;                 // n, precision u_g: published w (or z)
    void* tbuf;                 // n, precision u_p: t = A v
    void* V;                    // ldv x (kmax + 1), precision u_g; a block reads back only its own rows
    int64_t ldv;
    double* R;                  // (kmax + 1) x kmax column-major, written by block 0
    unsigned long long* msg;    // [2 parities][gridDim.x][SLOT_WORDS] epoch-tagged words
    unsigned long long* msg2;   // the same for the Gram-Schmidt group's rounds
    int g2;                     // Gram-Schmidt group: blocks 0..g2-1, each over the rows of two
                                // blocks (0: every block runs the rounds on its own rows)
    int* err;
    long long limit;            // clock64 cycles a wait may take
    double anorm, bnorm, tau, stop_tol;
    int kmax, imax, stop_rule;
    int* its;                   // imax
    double* nbe;                // imax + 1
    int* out;                   // [0] steps, [1] flags
    int orth;                   // 0 modified Gram-Schmidt, 1 classical Gram-Schmidt twice (CGS2)
    int side;                   // 0 left preconditioning (P A d = P r), 1 right (A P u = r, d = P u)
    int G;                      // blocks of this system
    void* pvec;                 // CGS2: 2 parities x gridDim.x x (kmax + 1) partial dot products (u_g);
                                // one-reduction MGS: 2 (kmax + 1) values of every block, [block][value]
                                // (binary32 arithmetic) or [value][block] (double)
    unsigned* gcount;           // CGS2 / one-reduction MGS: counter of the barrier that publishes them (zeroed)
    void* L;                    // one-reduction MGS: the rows of T = (I + L)^{-1}, L the strictly
                                // lower part of Q^T Q (row i: its i entries left of the unit
                                // diagonal, packed at i (i - 1) / 2), u_g; block 0 writes them
    int jl;                     // rows 0 .. jl-1 of T are also kept in each block's shared memory
    int nq;                     // and its rows of basis vectors 0 .. nq-1
    int xcap;                   // local launches: entries of a product's input staged in shared memory
    int xs_off;                 // at a time (0: none), at this offset of the dynamic shared memory
    int scat;                   // 1 = A's entries lie far from its diagonal (ir_scattered)
    int sblock;                 // one-reduction MGS: 1 = the system's last block owns no rows and
                                // runs the Givens rotations alone, publishing R and g (gpub); its
                                // verdict on column c travels as the flag of an exchange round
    double* gpub;               // kmax + 2: g as that block leaves it
};

// Bytes of a Krylov-part scalar for sg = sizeof(u_g): binary32 when the
// vectors are stored in half.
inline int ir_scalar_bytes(int sg) { return sg == 2 ? 4 : sg; }

// one-reduction MGS: values of the reduction summed over blocks in one pass (single and half)
constexpr int SUMV = 128;
constexpr int IR_WARPS = 16;    // warps of a block, at most
// the warps' sums of a pass lie over the unit partials of c and over h (both dead then), this many
// scalars beyond them
inline __host__ __device__ int ir_psum_more(int kmax, size_t sa)
{
    const int have = 2 * kmax + 34, need = sa == 4 ? 32 * IR_WARPS : 0;
    return need > have ? need - have : 0;
}
// group partials of a row of T: 32 columns for each warp, or every column
inline __host__ __device__ int ir_tpart(int kmax)
{
    const int all = (kmax + 31) & ~31;
    return all > 32 * IR_WARPS ? all : 32 * IR_WARPS;
}

// Dynamic shared memory of the refinement kernel (ir_body's layout), sg =
// sizeof(u_g): five double arrays of kmax + 2 (Givens, g, the current column,
// y), the slice offsets of A and P, the block's rows of w (two blocks' rows
// with a Gram-Schmidt group), and for the one-reduction MGS (orth 2) the rows
// of w next to those of u, the reduced inner products, row j of L, the unit
// partials (later the newest row of T and the warps' sums over blocks), h,
// rows 0 .. jl-1 of T, the table of segments per vector, the T row's group
// partials, and the block's rows of the first nq basis vectors.  What this
// takes beside the block's rows bounds the order that a grid solves.
inline size_t ir_smem_bytes(int64_t rb, int kmax, int g2, int orth, int jl, int nq, int sg, size_t xbytes = 0)
{
    const int64_t nsl = (rb + 31) >> 5;
    size_t b = sizeof(double) * 5 * (kmax + 2) + sizeof(int64_t) * 2 * (nsl + 1) + (g2 ? 2 : 1) * rb * sg + 64;
    if (orth == 2) {
        const size_t sa = (size_t)ir_scalar_bytes(sg);
        b += (size_t)sg * rb +
             sa * (2 * (kmax + 1) + 2 * (kmax + 1) + 2 * (kmax + 1 + 32) + ir_psum_more(kmax, sa) +
                   (size_t)jl * (jl - 1) / 2) +
             sizeof(int) * (kmax + 2) + 16 +  // the unit-count table
             sa * ir_tpart(kmax) + 16 +       // the T row's group partials
             (size_t)nq * rb * sg;
    }
    return xbytes ? ((b + 15) & ~size_t(15)) + xbytes : b;
}

// Whether A's entries lie far from the diagonal, so that a product's gathers
// hit a sector each: a mean distance of more than 1/16 of the order (a random
// matrix: 1/3; a 2D grid of n = 2000: 1/60).
inline bool ir_scattered(int64_t n, int64_t nnz, unsigned long long dist)
{
    return n > 256 && (double)dist * 16.0 > (double)n * (double)nnz;
}

// What a launch keeps in shared memory beside the rest.
struct IrSmem {
    int jl = 0, nq = 0;   // rows of T, basis vectors
    int xcap = 0;         // staged entries of a product's input
    size_t xs_off = 0, bytes = 0;
};

// Scattered matrices on a grid, double: basis vectors are kept in shared memory only
// as far as the block leaves the L1 cache its share; past 196 of the SM's 256 KB it falls
// from 60 to 28 KB, and the loads in flight of the products, their gathers and T's rows
// land there.  Us per iteration with 28 / 60 / 92 KB of L1, random matrices with 500
// vectors: n = 20000 172 / 164 / 165, n = 100000 290 / 278 / 277, n = 300000 567 / 521 / 515.  (Not
// on a cluster, whose 16 SMs wait for the basis from L2: n = 6000 196 / 229.  Stencils with
// double vectors lose 2 to 4%.)
constexpr size_t IR_SMEM_L1 = (size_t)192 << 10;  // (beside static and system shares)

// n_staged > 0 (local launches of scattered matrices: ir_scattered): room for the
// whole input of a product, of n_staged entries, or, when both Krylov types are the same (partial sums then stay in `out`), for at least
// a quarter of it.  One-reduction MGS: rows of T, as many as fit, at most kmax + 1,
// within 40 KiB (24 KiB beside staged inputs, 64 KiB in double), and the block's rows of the
// first basis vectors (both passes over the basis read these without a trip to
// L2).
inline IrSmem ir_pick_smem(int64_t rb, int kmax, int g2, int orth, size_t dyn_max, int sg, int sp, int64_t n_staged,
                           bool keep_l1 = false)
{
    IrSmem s;
    const size_t sa = (size_t)ir_scalar_bytes(sg);
    const size_t lim = dyn_max - 1024;
    const size_t base = ir_smem_bytes(rb, kmax, g2, orth, 0, 0, sg);
    s.bytes = base;
    if (base > lim) return s;
    const size_t tmax = orth == 2 ? (sa == 4 ? (n_staged > 0 ? 24 << 10 : 40 << 10) : 64 << 10) : 0;
    if (n_staged > 0 && n_staged <= (1 << 22)) {
        const size_t room = (lim - base > tmax + 64 ? (lim - base - tmax - 64) / sp : 0) & ~size_t(31);
        const size_t whole = ((size_t)n_staged + 31) & ~size_t(31);
        const size_t passes = room ? (whole + room - 1) / room : 0;
        if (passes == 1 || (sg == sp && sg != 2 && passes >= 1 && passes <= 4))
            s.xcap = (int)(((whole + passes - 1) / passes + 31) & ~size_t(31));
    }
    const size_t xb = (size_t)s.xcap * sp;
    if (orth == 2) {
        const size_t room = std::min(lim - base - (xb ? xb + 16 : 0), tmax) / sa;
        while (s.jl < kmax + 1 && (size_t)(s.jl + 1) * s.jl / 2 <= room) s.jl++;
        const size_t used = ir_smem_bytes(rb, kmax, g2, orth, s.jl, 0, sg, xb);
        const size_t lq = keep_l1 ? std::min<size_t>(lim, IR_SMEM_L1) : lim;
        if (used < lq) s.nq = (int)std::min<size_t>((lq - used) / ((size_t)rb * sg), (size_t)kmax + 1);
    }
    s.bytes = ir_smem_bytes(rb, kmax, g2, orth, s.jl, s.nq, sg, xb);
    s.xs_off = s.bytes - xb;
    return s;
}

struct IrShared {
    int bid;          // the block's rank within its system
    int G;            // the system's block count
    unsigned epoch;
    unsigned epoch2;  // rounds of the Gram-Schmidt group
    unsigned gepoch;  // CGS2 barrier count
    int ok;
    // the exchange slots of the grid (IrArgs), the group's size and the wait limit
    unsigned long long* msg;
    unsigned long long* msg2;
    int* err;
    long long limit;
    int g2;
    unsigned long long res[4];  // a round's result
    double resid;
    double ibeta;  // 1 / ||z||, thread 0's (MGS and CGS2)
    double dmax;   // this block's largest |d| of the last correction (as added to x, in u)
    double qprev;  // ||d_{i-2}|| / ||x_{i-1}|| (the stagnation test of the stop rules)
};
struct IrSharedLoc : IrShared {
    // a system whose blocks are one thread-block cluster: the words of every block's
    // exchange rounds, written by the blocks themselves (two parities)
    unsigned long long cslot[2][MAX_CLUSTER][3];
};

__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// two words, each a single-copy-atomic load of its own
__device__ __forceinline__ void ld_relaxed_2u64(const unsigned long long* p, unsigned long long& a, unsigned long long& b)
{
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// What a round combines, over its blocks in a fixed order: the OR of a flag,
// a sum, or three maxima of bit patterns (abs_key).
// X_VECF and X_VECD: MGS_N sums.
enum { X_FLAG = 0, X_SUMF = 1, X_SUMD = 2, X_MAX3 = 3, X_VECF = 4, X_VECD = 5 };
template <class T> struct XSum { static constexpr int K = sizeof(T) == 8 ? X_SUMD : X_SUMF; };
// Vectors of a modified Gram-Schmidt round: as many sums as four payload words hold
template <class T> struct XVec {
    static constexpr int K = sizeof(T) == 8 ? X_VECD : X_VECF, N = sizeof(T) == 8 ? 2 : 4;
};
// 32-bit words of a block's payload
template <int K> constexpr int x_words() { return K == X_MAX3 ? 6 : (K >= X_VECF ? 4 : (K == X_SUMD ? 2 : 1)); }

// The lanes' shares of a round: add() takes one block's words, reduce() leaves
// the result of all lanes in every lane.
template <int K> struct XAcc {
    unsigned long long m[4];
    double d, dv[2];
    float f, fv[4];
    __device__ __forceinline__ void reset()
    {
        m[0] = m[1] = m[2] = 0;
        d = dv[0] = dv[1] = 0.0;
        f = fv[0] = fv[1] = fv[2] = fv[3] = 0.f;
    }
    __device__ __forceinline__ void add(const uint32_t* w)
    {
        if (K == X_FLAG) m[0] |= w[0];
        else if (K == X_SUMF) f += __uint_as_float(w[0]);
        else if (K == X_SUMD) d += __longlong_as_double((long long)(((unsigned long long)w[0] << 32) | w[1]));
        else if (K == X_VECF) {
#pragma unroll
            for (int k = 0; k < 4; k++) fv[k] += __uint_as_float(w[k]);
        } else if (K == X_VECD) {
#pragma unroll
            for (int k = 0; k < 2; k++)
                dv[k] += __longlong_as_double((long long)(((unsigned long long)w[2 * k] << 32) | w[2 * k + 1]));
        } else {
#pragma unroll
            for (int k = 0; k < 3; k++) m[k] = max(m[k], ((unsigned long long)w[2 * k] << 32) | w[2 * k + 1]);
        }
    }
    __device__ __forceinline__ void reduce(unsigned G)
    {
        if (K == X_FLAG) m[0] = __reduce_or_sync(0xffffffffu, (unsigned)m[0]);
        else if (K == X_SUMF) m[0] = __float_as_uint(G > 1 ? wsum(f) : __shfl_sync(0xffffffffu, f, 0));
        else if (K == X_SUMD)
            m[0] = (unsigned long long)__double_as_longlong(G > 1 ? wsum(d) : __shfl_sync(0xffffffffu, d, 0));
        else if (K == X_VECF) {
#pragma unroll
            for (int k = 0; k < 4; k++)
                m[k] = __float_as_uint(G > 1 ? wsum(fv[k]) : __shfl_sync(0xffffffffu, fv[k], 0));
        } else if (K == X_VECD) {
#pragma unroll
            for (int k = 0; k < 2; k++)
                m[k] = (unsigned long long)__double_as_longlong(G > 1 ? wsum(dv[k]) : __shfl_sync(0xffffffffu, dv[k], 0));
        } else {
#pragma unroll
            for (int k = 0; k < 3; k++) m[k] = warp_max_key(m[k]);
        }
    }
};
template <class T> __device__ __forceinline__ T x_value(unsigned long long m)
{
    if (sizeof(T) == 8) return (T)__longlong_as_double((long long)m);
    return (T)__uint_as_float((unsigned)m);
}
// a value as payload words
__device__ __forceinline__ void x_pay(float v, uint32_t* w) { w[0] = __float_as_uint(v); }
__device__ __forceinline__ void x_pay(double v, uint32_t* w)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    w[0] = (uint32_t)(u >> 32);
    w[1] = (uint32_t)u;
}

// One exchange round among all blocks of the co-resident grid (grp: among the
// Gram-Schmidt group, blocks 0..g2-1, with its own slots and epoch; only its
// blocks may call).  Thread 0 publishes the block's words, each tagged with
// the round's epoch in the upper 32 bits (one single-copy-atomic 64-bit store
// per word), with `data` after a fence that orders everything the block wrote
// before the preceding __syncthreads.  Each block's slot is a 128-byte line of
// its own: blocks sharing a line made every round measurably slower (the
// polls of all blocks and the stores of the line's owners queue on the same
// L2 line), while more polling warps or a denser layout made it slower still.
// Warp 0 then polls every block's words of that epoch (lane l owns blocks l,
// l+32, ...) until one pass sees every word carry the epoch, combines them in
// that fixed order and leaves the result in sh->res.  Slots alternate between
// two parities, so a block can only overwrite a slot after every block has
// read it.  The wait is bounded: on expiry SPAI_ERR_TIMEOUT goes to *err,
// sh->ok is 0 and every block leaves.
template <int K>
__device__ __forceinline__ void x_publish(IrShared* sh, bool data, bool grp, const uint32_t* pay)
{
    const unsigned G = grp ? (unsigned)sh->g2 : (unsigned)sh->G;
    const unsigned ep = (grp ? sh->epoch2 : sh->epoch) + 1u;
    unsigned long long* base = (grp ? sh->msg2 : sh->msg) + ((size_t)(ep & 1u) * G + sh->bid) * SLOT_WORDS;
    if (data) __threadfence();
#pragma unroll
    for (int k = 0; k < x_words<K>(); k++) st_relaxed_u64(base + k, ((unsigned long long)ep << 32) | pay[k]);
}

template <int K>
__device__ __forceinline__ void x_poll(IrShared* sh, bool data, bool grp)
{
    constexpr int NW = x_words<K>();
    const unsigned lane = threadIdx.x & 31;
    const unsigned G = grp ? (unsigned)sh->g2 : (unsigned)sh->G;
    unsigned* epoch = grp ? &sh->epoch2 : &sh->epoch;
    const unsigned ep = *epoch + 1u;
    const unsigned long long* base = (grp ? sh->msg2 : sh->msg) + (size_t)(ep & 1u) * G * SLOT_WORDS;
    XAcc<K> acc;
    const long long t0 = clock64();
    int ok = 1;
#pragma unroll 1
    for (unsigned spins = 1;; spins++) {
        bool all = true;
        acc.reset();
        if constexpr (K == X_MAX3) {
            // (once per refinement step: a loop, few registers)
#pragma unroll 1
            for (unsigned i = lane; i < G; i += 32u) {
                uint32_t wv[NW];
#pragma unroll
                for (int k = 0; k < NW; k++) {
                    const unsigned long long w = ld_relaxed_u64(base + (size_t)i * SLOT_WORDS + k);
                    all = all && (unsigned)(w >> 32) == ep;
                    wv[k] = (uint32_t)w;
                }
                acc.add(wv);
            }
        } else {
            uint32_t wv[SPL][NW];
#pragma unroll
            for (int u = 0; u < SPL; u++) {
                const unsigned i = lane + 32u * u;
                if (i < G) {
#pragma unroll
                    for (int k = 0; k < NW; k++) {
                        const unsigned long long w = ld_relaxed_u64(base + (size_t)i * SLOT_WORDS + k);
                        all = all && (unsigned)(w >> 32) == ep;
                        wv[u][k] = (uint32_t)w;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < SPL; u++)
                if (lane + 32u * u < G) acc.add(wv[u]);
        }
        if (__all_sync(0xffffffffu, all)) break;
        if ((spins & 31u) == 0u) {
            int bad = 0;
            if (lane == 0) {
                if (ld_relaxed_i32(sh->err) != 0) bad = 1;
                else if (clock64() - t0 > sh->limit) { atomicCAS(sh->err, 0, SPAI_ERR_TIMEOUT); bad = 1; }
            }
            if (__shfl_sync(0xffffffffu, bad, 0)) { ok = 0; break; }
        }
    }
    if (data) __threadfence();
    acc.reduce(G);
    __syncwarp();
    if (lane == 0) {
        sh->res[0] = acc.m[0];
        if (K == X_MAX3) { sh->res[1] = acc.m[1]; sh->res[2] = acc.m[2]; }
        sh->ok = ok;
        *epoch = ep;
    }
}

// x_poll for a Gram-Schmidt round's sums (XVec<T>::N of them in four words, read
// two at a time): SL blocks a lane at a time, doubles added on the integer pipe.
template <class T, int SL>
__device__ __forceinline__ void x_poll_vec(IrShared* sh, bool data, bool grp)
{
    constexpr int N = XVec<T>::N;
    const unsigned lane = threadIdx.x & 31;
    const unsigned G = grp ? (unsigned)sh->g2 : (unsigned)sh->G;
    unsigned* epoch = grp ? &sh->epoch2 : &sh->epoch;
    const unsigned ep = *epoch + 1u;
    const unsigned long long* base = (grp ? sh->msg2 : sh->msg) + (size_t)(ep & 1u) * G * SLOT_WORDS;
    T sum[N];
#pragma unroll
    for (int e = 0; e < N; e++) sum[e] = T(0);
    const long long t0 = clock64();
    int ok = 1;
#pragma unroll 1
    for (unsigned b0 = 0; b0 < G && ok; b0 += 32u * SL) {
        uint32_t wv[SL][4];
#pragma unroll 1
        for (unsigned spins = 1;; spins++) {
            bool all = true;
#pragma unroll
            for (int u = 0; u < SL; u++) {
                const unsigned i = b0 + lane + 32u * u;
#pragma unroll
                for (int k = 0; k < 4; k += 2) {
                    unsigned long long x = (unsigned long long)ep << 32, y = x;
                    if (i < G) ld_relaxed_2u64(base + (size_t)i * SLOT_WORDS + k, x, y);
                    all = all && (unsigned)(x >> 32) == ep && (unsigned)(y >> 32) == ep;
                    wv[u][k] = (uint32_t)x;
                    wv[u][k + 1] = (uint32_t)y;
                }
            }
            if (__all_sync(0xffffffffu, all)) break;
            if ((spins & 31u) == 0u) {
                int bad = 0;
                if (lane == 0) {
                    if (ld_relaxed_i32(sh->err) != 0) bad = 1;
                    else if (clock64() - t0 > sh->limit) { atomicCAS(sh->err, 0, SPAI_ERR_TIMEOUT); bad = 1; }
                }
                if (__shfl_sync(0xffffffffu, bad, 0)) { ok = 0; break; }
            }
        }
#pragma unroll
        for (int e = 0; e < N; e++) {
            T v[SL];
#pragma unroll
            for (int u = 0; u < SL; u++) {
                if constexpr (sizeof(T) == 8)
                    v[u] = __longlong_as_double((long long)(((unsigned long long)wv[u][2 * e] << 32) | wv[u][2 * e + 1]));
                else v[u] = __uint_as_float(wv[u][e]);
            }
            if constexpr (sizeof(T) == 8) {
                const T t = warp_sum_fx_n<SL>(v);
                sum[e] = b0 ? sum[e] + t : t;
            } else {
                T t = v[0];
#pragma unroll
                for (int u = 1; u < SL; u++) t += v[u];
                sum[e] += warp_sum(t);
            }
        }
    }
    if (data) __threadfence();
    __syncwarp();
    if (lane == 0) {
#pragma unroll
        for (int e = 0; e < N; e++)
            sh->res[e] = sizeof(T) == 8 ? (unsigned long long)__double_as_longlong((double)sum[e])
                                        : (unsigned long long)__float_as_uint((float)sum[e]);
        sh->ok = ok;
        *epoch = ep;
    }
}

// The cluster-wide barrier in its two halves: every thread of the cluster's
// blocks arrives (its earlier writes, global and shared, released to the
// cluster) and waits (the others' acquired).  A block that has left counts as
// arrived.
__device__ __forceinline__ void cluster_arrive()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait()
{
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// *p (in this block's shared memory) of the cluster's block `rank` = v
__device__ __forceinline__ void st_cluster_u64(unsigned long long* p, unsigned rank, unsigned long long v)
{
    const uint32_t at = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t to;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(at), "r"(rank));
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(to), "l"(v) : "memory");
}

// The round of a system that runs on one block or on one thread-block
// cluster: no polling through L2.  Warp 0 stores the block's words into every
// block's shared memory and the cluster barrier publishes them (with
// everything the blocks wrote before); every warp then combines the words of
// all blocks itself, in block order, so no block barrier follows.  The slots
// alternate between two parities (lep counts the rounds): a block writes the
// next round's words of a parity only after a barrier that follows every read
// of the last ones.  Measured on 16 blocks: 640 cycles for the barrier against
// 3000 to 4000 for a round through L2.
template <int K>
__device__ __forceinline__ void xl_send(IrShared* sh, unsigned lep, const uint32_t* pay)
{
    constexpr int NW = x_words<K>(), NU = (NW + 1) / 2;
    const unsigned G = (unsigned)sh->G, lane = threadIdx.x & 31;
    if (threadIdx.x < 32 && lane < G) {
#pragma unroll
        for (int u = 0; u < NU; u++) {
            const unsigned long long w = ((unsigned long long)pay[2 * u] << 32) | (2 * u + 1 < NW ? pay[2 * u + 1] : 0u);
            IrSharedLoc* sl = static_cast<IrSharedLoc*>(sh);
            if (G == 1) sl->cslot[lep & 1u][0][u] = w;
            else st_cluster_u64(&sl->cslot[lep & 1u][sh->bid][u], lane, w);
        }
    }
    if (G > 1) cluster_arrive();
}
template <int K>
__device__ __forceinline__ void xl_take(IrShared* sh, unsigned lep, XAcc<K>& acc)
{
    constexpr int NW = x_words<K>(), NU = (NW + 1) / 2;
    const unsigned G = (unsigned)sh->G, lane = threadIdx.x & 31;
    if (G > 1) cluster_wait();
    else __syncthreads();
    acc.reset();
    if (lane < G) {
        uint32_t wv[2 * NU];
#pragma unroll
        for (int u = 0; u < NU; u++) {
            const unsigned long long w = static_cast<IrSharedLoc*>(sh)->cslot[lep & 1u][lane][u];
            wv[2 * u] = (uint32_t)(w >> 32);
            wv[2 * u + 1] = (uint32_t)w;
        }
        acc.add(wv);
    }
    acc.reduce(G);
}

// Sum over all blocks of a per-thread value, in a fixed order; the result
// is identical in every block.  In two halves: between them thread 0 may run
// short serial work, which hides in the wait for the other blocks (their
// words take about a microsecond to arrive on a grid).  nw: the warps that may
// hold a value other than zero (the first ones).  data: the round also
// publishes the global writes made before it; without it only the scalar
// travels, in the same single-copy-atomic word as its epoch.
template <bool LOC, class T>
__device__ __forceinline__ void xsum_begin(IrShared* sh, unsigned lep, int nw, T* red, T v, bool data, bool grp)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid < nw) {
        v = wsum(v);
        if (lane == 0) red[wid] = v;
    }
    __syncthreads();
    uint32_t pay[2] = {0u, 0u};
    if (wid == 0) {
        T t = lane < nw ? red[lane] : T(0);
        if (nw > 1) t = wsum(t);
        else t = __shfl_sync(0xffffffffu, t, 0);
        x_pay(t, pay);
        if (!LOC && lane == 0) x_publish<XSum<T>::K>(sh, data, grp, pay);
    }
    if (LOC) xl_send<XSum<T>::K>(sh, lep, pay);
}
// the sum; on a grid sh->ok tells whether the wait ended well
template <bool LOC, class T>
__device__ __forceinline__ T xsum_end(IrShared* sh, unsigned lep, bool data, bool grp)
{
    if (LOC) {
        XAcc<XSum<T>::K> acc;
        xl_take(sh, lep, acc);
        return x_value<T>(acc.m[0]);
    }
    __syncwarp();
    if (threadIdx.x < 32) x_poll<XSum<T>::K>(sh, data, grp);
    __syncthreads();
    return x_value<T>(sh->res[0]);
}

// The same for the XVec<T>::N sums of a Gram-Schmidt round; red holds 32 values
// per sum.
template <bool LOC, class T, int N>
__device__ __forceinline__ void xvec_begin(IrShared* sh, unsigned lep, int nw, T* red, const T (&v)[N], bool data, bool grp)
{
    constexpr int K = XVec<T>::K;
    static_assert(N == XVec<T>::N, "sums of a round");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid < nw) {
        T t[N];
#pragma unroll
        for (int e = 0; e < N; e++) t[e] = wsum(v[e]);
        if (lane == 0) {
#pragma unroll
            for (int e = 0; e < N; e++) red[32 * e + wid] = t[e];
        }
    }
    __syncthreads();
    uint32_t pay[x_words<K>()] = {};
    if (wid == 0) {
#pragma unroll
        for (int e = 0; e < N; e++) {
            T t = lane < nw ? red[32 * e + lane] : T(0);
            if (nw > 1) t = wsum(t);
            else t = __shfl_sync(0xffffffffu, t, 0);
            x_pay(t, pay + e * (int)(sizeof(T) / 4));
        }
        if (!LOC && lane == 0) x_publish<K>(sh, data, grp, pay);
    }
    if (LOC) xl_send<K>(sh, lep, pay);
}
// out: the sums; with gam the Gram-Schmidt coefficients of a round's cnt vectors
// instead: h_e = c_e - sum_{m < e} (v_e . v_m) h_m, gam[e (e - 1) / 2 + m] = v_e . v_m
// (SL: x_poll_vec)
template <bool LOC, int SL, class T, int N>
__device__ __forceinline__ void xvec_end(IrShared* sh, unsigned lep, bool data, bool grp, const T* gam, int cnt, T (&out)[N])
{
    constexpr int K = XVec<T>::K;
    auto solve = [&]() {
#pragma unroll
        for (int e = 1; e < N; e++)
            if (e < cnt) {
#pragma unroll
                for (int m = 0; m < e; m++) out[e] = fma(-gam[e * (e - 1) / 2 + m], out[m], out[e]);
            }
    };
    if (LOC) {
        XAcc<K> acc;
        xl_take(sh, lep, acc);
#pragma unroll
        for (int e = 0; e < N; e++) out[e] = x_value<T>(acc.m[e]);
        if (gam) solve();
        return;
    }
    __syncwarp();
    if (threadIdx.x < 32) {
        x_poll_vec<T, SL>(sh, data, grp);
        // (by one thread: a double operation of every warp would hold the FP64 pipe)
        if (gam && cnt > 1 && threadIdx.x == 0) {
#pragma unroll
            for (int e = 0; e < N; e++) out[e] = x_value<T>(sh->res[e]);
            solve();
#pragma unroll
            for (int e = 1; e < N; e++)
                sh->res[e] = sizeof(T) == 8 ? (unsigned long long)__double_as_longlong((double)out[e])
                                            : (unsigned long long)__float_as_uint((float)out[e]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < N; e++) out[e] = x_value<T>(sh->res[e]);
}

// Max of three non-negative doubles (bit patterns) over all blocks, to o; red
// holds 96 words.
template <bool LOC>
__device__ __forceinline__ bool xmax3(IrShared* sh, unsigned lep, unsigned long long* red, unsigned long long v0,
                                   unsigned long long v1, unsigned long long v2, double* o)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned long long v[3] = {v0, v1, v2};
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const unsigned long long t = warp_max_key(v[k]);
        if (lane == 0) red[32 * k + wid] = t;
    }
    __syncthreads();
    uint32_t pay[6] = {0u, 0u, 0u, 0u, 0u, 0u};
    if (wid == 0) {
#pragma unroll
        for (int k = 0; k < 3; k++) x_pay(key_value(warp_max_key(lane < nw ? red[32 * k + lane] : 0ull)), pay + 2 * k);
    }
    if (LOC) {
        XAcc<X_MAX3> acc;
        xl_send<X_MAX3>(sh, lep, pay);
        xl_take(sh, lep, acc);
#pragma unroll
        for (int k = 0; k < 3; k++) o[k] = key_value(acc.m[k]);
        return true;
    }
    if (wid == 0) {
        if (lane == 0) x_publish<X_MAX3>(sh, true, false, pay);
        __syncwarp();
        x_poll<X_MAX3>(sh, true, false);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 3; k++) o[k] = key_value(sh->res[k]);
    return sh->ok != 0;
}

// plain barrier (no payload)
template <bool LOC>
__device__ __forceinline__ bool xbar(IrShared* sh)
{
    if (LOC) {
        if (sh->G > 1) {
            cluster_arrive();
            cluster_wait();
        } else {
            __syncthreads();
        }
        return true;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const uint32_t pay[1] = {0u};
        if (threadIdx.x == 0) x_publish<X_FLAG>(sh, true, false, pay);
        __syncwarp();
        x_poll<X_FLAG>(sh, true, false);
    }
    __syncthreads();
    return sh->ok != 0;
}

// Barrier with a flag: *flag becomes the OR of the blocks' `mine` (thread 0's).
// `idle` runs on every warp but the first while the block waits, its results
// visible to the block afterwards.
template <bool LOC, class Idle>
__device__ __forceinline__ bool xbar_flag(IrShared* sh, unsigned lep, unsigned mine, unsigned* flag, const Idle& idle)
{
    const uint32_t pay[1] = {mine};
    if (LOC) {
        // (what the block wrote before, for the idle work)
        __syncthreads();
        xl_send<X_FLAG>(sh, lep, pay);
        if (threadIdx.x >= 32) idle();
        XAcc<X_FLAG> acc;
        xl_take(sh, lep, acc);
        *flag = (unsigned)acc.m[0];
        // (the warps arrived before their idle work: its results need a barrier of their own)
        __syncthreads();
        return true;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        if (threadIdx.x == 0) x_publish<X_FLAG>(sh, true, false, pay);
        __syncwarp();
        x_poll<X_FLAG>(sh, true, false);
    } else {
        idle();
    }
    __syncthreads();
    *flag = (unsigned)sh->res[0];
    return sh->ok != 0;
}

// A thread's sum over its rows in two chains, taken in turn: half as many roundings, so
// binary32 sums of a block's rows over 512 threads round no more often than over 896.
// (Double: these blocks always had 512.)
template <class T> __device__ __forceinline__ void in_turn(T& a, T& b)
{
    if constexpr (sizeof(T) == 4) {
        const T t = a;
        a = b;
        b = t;
    }
}
template <class T> __device__ __forceinline__ T both(T a, T b) { return sizeof(T) == 4 ? a + b : a; }

// v 2^e, exact (reading R17: the residual scaling of half-precision Krylov
// parts); the identity when HK is false
template <bool HK, class T> __device__ __forceinline__ T scale2(T v, int e)
{
    if constexpr (HK) return (T)ldexp((double)v, e);
    else return v;
}

// How a product reads its input x_c: as it is, as the quotient x_c / d (by
// its reciprocal y, or by a division where the reciprocal is out of range), or
// scaled by 2^e (half storage).
enum { LD_PLAIN = 0, LD_QUOT = 1, LD_DIV = 2, LD_SCALE = 3 };
template <class TP, class TI, int LD> struct XIn {
    const TI* x;
    TI d, y;
    int e;
    __device__ __forceinline__ TP of(TI v) const
    {
        if constexpr (LD == LD_QUOT) {
            return (TP)quot_by(v, d, y);
        } else if constexpr (LD == LD_DIV) {
            return (TP)(v / d);
        } else if constexpr (LD == LD_SCALE) {
            return (TP)scale2<true>(v, e);
        } else {
            return (TP)v;
        }
    }
    __device__ __forceinline__ TP get(int c) const { return of(ldcg(x + c)); }
};

// One entry's input and value: from global memory, or (STAGED) from the inputs
// lo .. lo + cnt - 1 in shared memory (xs, already transformed; entries outside
// are left to another pass).
template <class TP> struct XStage {
    const TP* xs;
    int lo, cnt;
    bool more;  // a later pass: add to what out holds
};
template <bool STAGED, class TP, class TI, int LD, class C>
__device__ __forceinline__ void sell_gather(const XIn<TP, TI, LD>& in, const XStage<TP>& st, int c, C& g, bool& here)
{
    if constexpr (STAGED) {
        here = (unsigned)(c - st.lo) < (unsigned)st.cnt;
        g = here ? (C)st.xs[c - st.lo] : C(0);
    } else {
        here = true;
        g = c >= 0 ? (C)in.get(c) : C(0);
    }
}

// p + 32 k, multiplied in bytes: one wide multiply-add
template <class T> __device__ __forceinline__ const T* col32(const T* p, unsigned k)
{
    return reinterpret_cast<const T*>(reinterpret_cast<const char*>(p) + (uint64_t)k * (uint64_t)(32 * sizeof(T)));
}

// Products with single and half values (and staged ones): thread t takes rows
// t, t + BT, ...; R rows per thread and pass, U entries of each in flight: the
// entries of chunk c+1 load while chunk c gathers.  col, val: the block's first
// entry, soff[0] its offset in the matrix.  Places are entries in 32 bits, or (WIDE:
// matrices of 2^31 entries and more, which dense rows beside one another bring into one block)
// columns of 32 entries.  Us per iteration 32-bit / WIDE / a branch between two loops: MGS single
// n = 125000 34.0 / 34.4, n = 143350 35.8 / 36.1 / 36.2, CGS2 n = 262144 57.9 / 59.0.
template <class TP, class TI, class TO, int LD, bool STAGED, int R, int U, bool WIDE>
__device__ __forceinline__ void sell_pass(int rows, const int64_t* soff, const int32_t* __restrict__ col,
                                          const TP* __restrict__ val, const XIn<TP, TI, LD>& in, TO* out,
                                          const XStage<TP>& st)
{
    typedef typename Compute<TP>::T C;
    const int tid = threadIdx.x, BT = blockDim.x, lane = tid & 31;
    const int64_t first = soff[0];
    if (WIDE) {
        col += lane;
        val += lane;
    }
    auto cat = [&](int k) { return WIDE ? col32(col, k) : col + k; };
    auto vat = [&](int k) { return WIDE ? col32(val, k) : val + k; };
#pragma unroll 1
    for (int base = 0; base < rows; base += R * BT) {
        int o[R], w[R], wmax = 0;
        C acc[R];
#pragma unroll
        for (int i = 0; i < R; i++) {
            const int row = base + i * BT + tid;
            const int s = row < rows ? row >> 5 : 0;
            o[i] = WIDE ? (int)((soff[s] - first) >> 5) : (int)(soff[s] - first) + lane;
            w[i] = row < rows ? (int)(soff[s + 1] - soff[s]) >> 5 : 0;
            wmax = max(wmax, w[i]);
            acc[i] = STAGED && st.more && row < rows ? (C)out[row] : C(0);
        }
        int cc[R][U];
        TP xv[R][U];
#pragma unroll
        for (int i = 0; i < R; i++)
#pragma unroll
            for (int u = 0; u < U; u++) {
                cc[i][u] = u < w[i] ? __ldg(cat(o[i]) + 32 * u) : -1;
                xv[i][u] = u < w[i] ? __ldg(vat(o[i]) + 32 * u) : TP(0);
            }
#pragma unroll 1
        for (int c0 = U; c0 < wmax + U; c0 += U) {
            C g[R][U], yv[R][U];
#pragma unroll
            for (int i = 0; i < R; i++)
#pragma unroll
                for (int u = 0; u < U; u++) {
                    bool here;
                    sell_gather<STAGED>(in, st, cc[i][u], g[i][u], here);
                    if (STAGED) yv[i][u] = here ? to_c(xv[i][u]) : C(0);
                }
#pragma unroll
            for (int i = 0; i < R; i++) {
                o[i] += WIDE ? U : 32 * U;
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (!STAGED) yv[i][u] = to_c(xv[i][u]);
                    cc[i][u] = c0 + u < w[i] ? __ldg(cat(o[i]) + 32 * u) : -1;
                    xv[i][u] = c0 + u < w[i] ? __ldg(vat(o[i]) + 32 * u) : TP(0);
                }
            }
#pragma unroll
            for (int u = 0; u < U; u++)
#pragma unroll
                for (int i = 0; i < R; i++) acc[i] = fma(yv[i][u], g[i][u], acc[i]);
        }
#pragma unroll
        for (int i = 0; i < R; i++) {
            const int row = base + i * BT + tid;
            if (row < rows) out[row] = (TO)(TP)acc[i];
        }
    }
}

// Products with double values, which stream twelve bytes an entry: each warp
// takes consecutive slices, whose entries are one contiguous stream of
// 32-entry columns, and loads it U columns at a time, two steps ahead of the
// gathers and across the slices' ends (32 rows each, one per lane), so that
// the stream never waits for a row's end.  n = 1e6: 207 -> 189 us per iteration,
// n = 91125: 30.2 -> 25.8.  (Scattered matrices in the one-reduction form wait for their
// gathers instead, and take sell_pass with eight of them in flight: random n = 100000 246 -> 239,
// n = 20000 151 -> 148.  Single values are bound by the instructions of a
// step instead: 31.4 -> 34.7 at n = 262144.)
template <class TP, class TI, class TO, int LD>
__device__ __forceinline__ void sell_stream(int rows, const int64_t* soff, const int32_t* __restrict__ col,
                                            const TP* __restrict__ val, const XIn<TP, TI, LD>& in, TO* out)
{
    typedef typename Compute<TP>::T C;
    constexpr int U = 4;
    const int lane = threadIdx.x & 31, nwp = blockDim.x >> 5;
    const int ns = (rows + 31) >> 5, per = (ns + nwp - 1) / nwp;
    int sl = (threadIdx.x >> 5) * per;
    const int s1 = min(ns, sl + per);
    if (sl >= s1) return;
    const int64_t o0 = soff[sl];
    const int ke = (int)((soff[s1] - o0) >> 5);
    col += o0 - soff[0] + lane;
    val += o0 - soff[0] + lane;
    int kend = (int)((soff[sl + 1] - o0) >> 5);
    int row = 32 * sl + lane;
    C acc = C(0);
    // the end of a slice: its rows are complete, and so are those of empty slices after it
    auto close = [&](int k) {
        do {
            if (row < rows) out[row] = (TO)(TP)acc;
            row += 32;
            acc = C(0);
            sl++;
            kend = sl < s1 ? (int)((soff[sl + 1] - o0) >> 5) : INT_MAX;
        } while (kend == k);
    };
    if (kend == 0) close(0);
    auto fetch = [&](int k, int (&c)[U], TP (&v)[U]) {
#pragma unroll
        for (int u = 0; u < U; u++) {
            c[u] = k + u < ke ? __ldg(col + 32 * (int64_t)k + 32 * u) : -1;
            v[u] = k + u < ke ? __ldg(val + 32 * (int64_t)k + 32 * u) : TP(0);
        }
    };
    auto step = [&](int k, int (&c)[U], TP (&v)[U]) {
        C g[U], yv[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            g[u] = c[u] >= 0 ? (C)in.get(c[u]) : C(0);
            yv[u] = to_c(v[u]);
        }
        fetch(k + 2 * U, c, v);
#pragma unroll
        for (int u = 0; u < U; u++) {
            acc = fma(yv[u], g[u], acc);
            if (k + u + 1 == kend) close(k + u + 1);
        }
    };
    int ca[U], cb[U];
    TP va[U], vb[U];
    fetch(0, ca, va);
    fetch(U, cb, vb);
#pragma unroll 1
    for (int k = 0; k < ke; k += 2 * U) {
        step(k, ca, va);
        if (k + U < ke) step(k + U, cb, vb);
    }
}

// out = M x for the block's rows 0 .. rows-1 (SELL-32; soff: the slice offsets
// in shared memory): products and sums in the compute type of TP (binary32 for
// half values and inputs).  A thread keeps 12 entries in flight, of one, two or
// four rows: each chunk of entries costs one trip to L2 for its gathers.  (16
// and 8: 32.4 and 31.8 us per iteration of the one-reduction MGS at n = 262144
// against 31.4.)
template <class TP, class TI, class TO, int LD, bool STAGED, bool WIDE = false>
__device__ __forceinline__ void sell_mul(int rows, const int64_t* soff, const int32_t* __restrict__ col,
                                         const TP* __restrict__ val, const XIn<TP, TI, LD>& in, TO* out,
                                         const XStage<TP>& st, bool stream)
{
    const int BT = blockDim.x;
    col += soff[0];
    val += soff[0];
    if (sizeof(TP) == 8 && !STAGED && stream) {
        sell_stream(rows, soff, col, val, in, out);
    } else {
        constexpr int N = sizeof(TP) == 8 ? 8 : 12;
        if (rows <= BT) sell_pass<TP, TI, TO, LD, STAGED, 1, N, WIDE>(rows, soff, col, val, in, out, st);
        else if (rows <= 2 * BT) sell_pass<TP, TI, TO, LD, STAGED, 2, N / 2, WIDE>(rows, soff, col, val, in, out, st);
        else sell_pass<TP, TI, TO, LD, STAGED, 4, N / 4, WIDE>(rows, soff, col, val, in, out, st);
    }
}

template <bool WIDE, class TP, class TI, class TO, int LD>
__device__ __forceinline__ void sell_mul_direct(int rows, const int64_t* soff, const int32_t* __restrict__ col,
                                                const TP* __restrict__ val, const XIn<TP, TI, LD>& in, TO* out,
                                                bool stream)
{
    sell_mul<TP, TI, TO, LD, false, WIDE>(rows, soff, col, val, in, out, XStage<TP>{nullptr, 0, 0, false}, stream);
}

// The same with the input staged through shared memory, xcap entries at a
// time (local launches, scattered matrices): every entry is read from L2 and
// transformed once, coalesced.  A scattered gather through L2 costs a sector
// per entry, 1.5 cycles of the SM each; from shared memory it is a few cycles a
// warp.  Called by all threads.
template <class TP, class TI, class TO, int LD>
__device__ __forceinline__ void sell_staged(int n, int rows, const int64_t* soff, const int32_t* __restrict__ col,
                                            const TP* __restrict__ val, const XIn<TP, TI, LD>& in, TO* out, TP* xs,
                                            int xcap)
{
#pragma unroll 1
    for (int lo = 0; lo < n; lo += xcap) {
        const int cnt = min(xcap, n - lo), BT = blockDim.x;
        constexpr int V4 = 8;
        if (lo > 0) __syncthreads();  // every warp is done with the last entries
#pragma unroll 1
        for (int i0 = threadIdx.x; i0 < cnt; i0 += V4 * BT) {
            TI t[V4];
#pragma unroll
            for (int e = 0; e < V4; e++) t[e] = ldcg(in.x + lo + min(i0 + e * BT, cnt - 1));
#pragma unroll
            for (int e = 0; e < V4; e++)
                if (i0 + e * BT < cnt) xs[i0 + e * BT] = in.of(t[e]);
        }
        __syncthreads();
        sell_mul<TP, TI, TO, LD, true>(rows, soff, col, val, in, out, XStage<TP>{xs, lo, cnt, lo > 0}, false);
    }
}

// A column's Givens rotations by one warp (one-reduction MGS): rotations
// 0..c-1 and the new rotation c on column h (entries 0..c+1); g; the residual
// estimate.  The products of 32 rotations with their entries at once, the
// chain one FMA a rotation (a thread alone needed four FP64 instructions, 64
// cycles each, for every rotation).  store: this block writes R's column;
// pub (a rotating block): g is published through gpub, which the other blocks
// read after the next exchange round (whose flag carries the stop test).
__device__ __forceinline__ void givens_warp(IrShared* sh, double* cs, double* sn, double* g, const double* h, double* Rc,
                                         double* gpub, int c, int kmax, double beta, bool store, bool pub)
{
    const int ln = threadIdx.x & 31;
    double x = h[0];
#pragma unroll 1
    for (int q0 = 0; q0 < c; q0 += 32) {
        const int q = q0 + ln, nq = min(32, c - q0);
        const double csq = q < c ? cs[q] : 0.0, snq = q < c ? sn[q] : 0.0, hq = q < c ? h[q + 1] : 0.0;
        const double ph = csq * hq;
        double xin = 0.0;
#pragma unroll 4
        for (int t = 0; t < nq; t++) {
            const double st = __shfl_sync(0xffffffffu, snq, t), pt = __shfl_sync(0xffffffffu, ph, t);
            if (ln == t) xin = x;
            x = fma(-st, x, pt);
        }
        if (q < c && store) Rc[q] = fma(csq, xin, snq * hq);
    }
    if (ln == 0) {
        const double hs = h[c + 1];
        const double dn = sqrt(x * x + hs * hs);
        double cc = 1.0, ss = 0.0;
        if (dn != 0.0) {
            const Quot<double> qd(dn);
            cc = qd(x);
            ss = qd(hs);
        }
        cs[c] = cc;
        sn[c] = ss;
        const double gc = g[c];
        const double g1 = -ss * gc, g0 = cc * gc;
        g[c + 1] = g1;
        g[c] = g0;
        const double res = fabs(g1) / beta;
        sh->resid = res;
        if (store) Rc[c] = dn;
        if (pub) {
            gpub[c] = g0;
            gpub[c + 1] = g1;
        }
    }
    __syncwarp();
}

// y = R^{-1} g by blocks of 32 columns, the last first: lane t of warp 0 holds
// y of row c0 + t scaled by 1 / R(t, t) (one division per lane and block
// instead of one per column on the chain, which then is a shuffle and one FMA
// a column), columns loaded CB ahead; then every thread takes the block's
// columns off one row above.  (A division, two L2 loads and three warp
// barriers on the chain of every column took 2800 cycles a column.)  g is
// overwritten.
__device__ __forceinline__ void back_substitute(const double* R, double* g, double* yv, int k, int kmax)
{
    const int tid = threadIdx.x, BT = blockDim.x;
#pragma unroll 1
    for (int c1 = k; c1 > 0;) {
        const int c0 = (c1 - 1) & ~31, nb = c1 - c0;
        if (tid < 32) {
            constexpr int CB = 4;
            const int t = c0 + tid;
            const double rd = tid < nb ? __ldcg(&R[(size_t)t * (kmax + 1) + t]) : 0.0;
            auto colv = [&](int c) -> double {
                return c >= 0 && tid < c ? __ldcg(&R[(size_t)(c0 + c) * (kmax + 1) + t]) : 0.0;
            };
            double nx[CB];
#pragma unroll
            for (int u = 0; u < CB; u++) nx[u] = colv(nb - 1 - u);
            const double ri = rd != 0.0 ? 1.0 / rd : 0.0;
            double y = tid < nb && rd != 0.0 ? g[t] / rd : 0.0;
#pragma unroll 1
            for (int cb = nb - 1; cb >= 0; cb -= CB) {
                double cv[CB];
#pragma unroll
                for (int u = 0; u < CB; u++) {
                    cv[u] = nx[u] * ri;
                    nx[u] = colv(cb - CB - u);
                }
#pragma unroll
                for (int u = 0; u < CB; u++)
                    if (cb - u >= 0) y = fma(-cv[u], __shfl_sync(0xffffffffu, y, cb - u), y);
            }
            if (tid < nb) yv[t] = y;
        }
        __syncthreads();
#pragma unroll 1
        for (int t = tid; t < c0; t += BT) {
            double acc = g[t];
#pragma unroll 8
            for (int c = c0; c < c1; c++) acc = fma(-__ldcg(&R[(size_t)c * (kmax + 1) + t]), yv[c], acc);
            g[t] = acc;
        }
        __syncthreads();
        c1 = c0;
    }
}

// d = V_k y for one row, the basis loads BV at a time
template <class TG, class AG>
__device__ __forceinline__ AG basis_dot(const TG* V, int64_t ldv, const AG* ya, int k)
{
    constexpr int BV = 16;
    AG acc = AG(0);
#pragma unroll 1
    for (int i0 = 0; i0 < k; i0 += BV) {
        TG t[BV];
#pragma unroll
        for (int u = 0; u < BV; u++) t[u] = i0 + u < k ? ldcg(V + (int64_t)(i0 + u) * ldv) : TG(0);
#pragma unroll
        for (int u = 0; u < BV; u++)
            if (i0 + u < k) acc = fma((AG)t[u], ya[i0 + u], acc);
    }
    return acc;
}

// Threads per block of the refinement kernel, at most: 512, so 128 registers a
// thread.  The straight-line parts of an iteration are issued by every warp
// (28 warps made each of their instructions seven cycles), and no instantiation
// spills its loads in flight: 16 values of a sparse product, eight 16-byte
// basis loads.  Launches take fewer threads where a block has few rows
// (ir_block_threads).
constexpr int IR_BT = 512;

// Threads of a launch whose blocks own `rows` rows: enough for one row each (the
// one-reduction MGS, whose inner products spread vectors over the warps, takes
// a third more).  Measured us per iteration at 128 / 256 / 384 / 512 threads: MGS
// single, 192 rows (a cluster) 14.3 / 13.1 / 13.5 / 14.2, 256 rows 26.9 / 24.3 / 24.7 / 25.2, 424
// rows 34.2 / 30.5 / 30.8 / 28.9; one-reduction single, 256 rows 19.3 / 16.6 / 16.3 / 16.4; double, 96
// rows (a cluster) 18.8 / 18.9 / 19.8 / 21.2.
inline int ir_block_threads(int64_t rows, int orth)
{
    if (orth == 2) return rows <= 128 ? 256 : (rows <= 512 ? 384 : 512);
    return rows <= 384 ? 256 : 512;
}

// The refinement of one system by its G blocks; `bid` is this block's rank.  LOC:
// the blocks are one block or one thread-block cluster (xl_send, xl_take).
template <class TU, class TG, class TP, int RM, bool LS, bool LOC, bool WIDE = false>
__device__ __forceinline__ void ir_body(const IrArgs& a, const int bid, const int G)
{
    // AG, AP: the arithmetic types of u_g and u_p (binary32 for half storage)
    typedef typename Compute<TG>::T AG;
    typedef typename Compute<TP>::T AP;
    // half storage in the Krylov part: the residual is scaled (reading R17)
    constexpr bool HK = sizeof(TG) == 2 || sizeof(TP) == 2;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ typename std::conditional<LOC, IrSharedLoc, IrShared>::type shs;
    // the warps' words of a round: of maxima, or of at most four sums
    __shared__ unsigned long long redd[96];
    AG* const redg = reinterpret_cast<AG*>(redd);
    IrShared* sh = &shs;
    const int kmax = a.kmax;
    const int tid = threadIdx.x, BT = blockDim.x;
    const int64_t r0 = min(a.n, (int64_t)bid * a.rb);  // a block past the last row owns none
    const int rows = (int)(min(a.n, r0 + a.rb) - r0);
    // the block's rows rounded up to whole slices: the basis, w and u are kept zero in the
    // padding rows (only the last block has any), so vector loads need no tails
    const int rowsp = (rows + 31) & ~31;
    // modified Gram-Schmidt rows m0 .. m0 + mrows - 1: the block's own rows, or with a
    // Gram-Schmidt group the rows of blocks 2b and 2b+1 (none outside it)
    const bool sub = !LOC && a.g2 > 0;
    const bool gs = !sub || (int)bid < a.g2;
    const int nsl = (int)((a.rb + 31) >> 5);
    double* cs = (double*)smem;            // kmax + 2
    double* sn = cs + (kmax + 2);          // kmax + 2
    double* g = sn + (kmax + 2);           // kmax + 2
    double* hc = g + (kmax + 2);           // kmax + 2
    double* yv = hc + (kmax + 2);          // kmax + 2
    int64_t* soa = (int64_t*)(yv + (kmax + 2));  // nsl + 1 slice offsets of A
    int64_t* sop = soa + (nsl + 1);        // nsl + 1 slice offsets of P
    // w for the Gram-Schmidt rows (rb, or 2 rb with a group), 16-byte aligned
    TG* ws = (TG*)(((uintptr_t)(sop + (nsl + 1)) + 15) & ~(uintptr_t)15);
    constexpr int VN = 16 / (int)sizeof(TG);
    typedef typename std::conditional<sizeof(TG) == 8, double2, float4>::type TV;  // 16 bytes
    TU* x = (TU*)a.x;
    TU* r = (TU*)a.r;
    TG* wbuf = (TG*)a.wbuf;
    TP* tbuf = (TP*)a.tbuf;
    TG* V = (TG*)a.V;
    const bool hasP = a.P.off != nullptr;
    // the Arnoldi product w = second(first(v)): left P (A v), right A (P v)
    const bool rightP = hasP && a.side == 1;
    {
        const int64_t s0 = r0 >> 5, nslg = (a.n + 31) >> 5;
        for (int i = tid; i <= nsl; i += BT) {
            const int64_t sg = min(s0 + i, nslg);
            soa[i] = a.A.off[sg];
            sop[i] = hasP ? a.P.off[sg] : 0;
        }
        // the padding rows of u and w
        if (rowsp > rows) {
            for (int i = rows + tid; i < rowsp; i += BT) {
                wbuf[r0 + i] = TG(0);
                ws[i] = TG(0);
                if (LS) ws[a.rb + i] = TG(0);
            }
        }
    }
    if (tid == 0) {
        sh->bid = bid; sh->G = G; sh->epoch = 0; sh->epoch2 = 0; sh->gepoch = 0; sh->ok = 1;
        sh->msg = a.msg; sh->msg2 = a.msg2; sh->err = a.err; sh->limit = a.limit; sh->g2 = a.g2;
        sh->dmax = 0.0; sh->qprev = 0.0;
    }
    __syncthreads();
    unsigned lep = 0;  // rounds of xl_send so far
    // warps that own rows
    auto nwr = [&]() -> int { return LOC ? min(BT >> 5, max(1, rowsp >> 5)) : BT >> 5; };
    // a product with A or P (useP) by whichever way the launch has room for
    TP* xs = reinterpret_cast<TP*>(smem + a.xs_off);
    auto product = [&](bool useP, const auto& in, auto* out) {
        const int64_t* so = useP ? sop : soa;
        const int32_t* sc = useP ? a.P.col : a.A.col;
        const TP* sv = (const TP*)(useP ? a.P.val : a.A.val);
        if (rows == 0) return;
        if (LOC && a.xcap > 0) {
            __syncthreads();  // (the staged entries of the last product are read)
            sell_staged((int)a.n, rows, so, sc, sv, in, out, xs, a.xcap);
        } else {
            sell_mul_direct<WIDE>(rows, so, sc, sv, in, out, !LS || a.scat == 0);
        }
    };
    // the two products of an iteration, by their place: the first reads wbuf, the second tbuf
    auto first = [&](auto* out) { product(rightP, XIn<TP, TG, LD_PLAIN>{wbuf, TG(0), TG(0), 0}, out); };
    auto second = [&](TG* out) { product(!rightP, XIn<TP, TP, LD_PLAIN>{tbuf, TP(0), TP(0), 0}, out); };

    int steps = 0, flags = 0;
#pragma unroll 1
    for (int it = 0; it <= a.imax; it++) {
        // ---------------- residual r = b - A x in u_r, stored in u
        // (maxima by bit pattern; a NaN counts as infinite: a non-finite residual or iterate
        // must not pass for a small one in the stopping rule)
        decltype(abs_key(TU(0))) rmax = 0, xmax = 0;
#pragma unroll 1
        for (int64_t row = r0 + tid; row < r0 + rows; row += BT) {
            double hi = a.b[row], lo = 0.0;
            const int64_t qe = a.arp[row + 1];
#pragma unroll 4
            for (int64_t q = a.arp[row]; q < qe; q++) {
                const double xv = (double)ldcg(&x[a.aci[q]]);
                if (RM == 2) dd_sub_prod(hi, lo, a.aval[q], xv);
                else hi = fma(-a.aval[q], xv, hi);
            }
            const TU rv = (TU)(hi + lo);
            r[row] = rv;
            rmax = max(rmax, abs_key(rv));
            xmax = max(xmax, abs_key(ldcg(&x[row])));
        }
        double mx[3];
        if (!xmax3<LOC>(sh, lep++, redd, abs_key(key_value(rmax)), abs_key(key_value(xmax)), abs_key(sh->dmax), mx)) return;
        const double rn = mx[0], xn = mx[1], dn = mx[2];
        const double den = a.anorm * xn + a.bnorm;
        const double nb = den > 0.0 ? rn / den : 0.0;
        if (bid == 0 && tid == 0) a.nbe[it] = nb;
        if (!isfinite(nb)) { flags |= 8; break; }
        // the stopping rules (identical decisions in every block: the maxima are exchanged)
        const double q = xn > 0.0 ? dn / xn : (dn > 0.0 ? INFINITY : 0.0);
        if (a.stop_rule == IR_STOP_BACKWARD && nb <= a.stop_tol) { flags |= 1; break; }
        if (a.stop_rule == IR_STOP_CORRECTION && it >= 1 && q <= a.stop_tol) { flags |= 1; break; }
        if (it == a.imax) { flags |= 2; break; }
        if (a.stop_rule != IR_STOP_FIXED && it >= 2 && q >= 0.5 * sh->qprev) { flags |= 16; break; }
        __syncthreads();  // every thread has read sh->qprev and sh->dmax
        if (tid == 0) { sh->qprev = q; sh->dmax = 0.0; }
        // R17: GMRES takes r 2^-esc with ||r||_inf = m 2^esc, m in [0.5, 1), and the
        // correction is scaled back (half storage only)
        int esc = 0;
        if (HK && rn > 0.0) frexp(rn, &esc);

        // ---------------- z = P r (left) or r (right) in u_p, stored in u_g; beta = ||z||
        if (hasP && !rightP) {
            product(true, XIn<TP, TU, HK ? LD_SCALE : LD_PLAIN>{r, TU(0), TU(0), -esc}, ws);
            __syncthreads();
        }
        AG part = AG(0), part2 = AG(0);
#pragma unroll 1
        for (int i = tid; i < rows; i += BT) {
            const TG z = hasP && !rightP ? ws[i] : (TG)(TP)scale2<HK>(r[r0 + i], -esc);
            ws[i] = z;
            wbuf[r0 + i] = z;
            part = fma((AG)z, (AG)z, part);
            in_turn(part, part2);
        }
        part = both(part, part2);
        xsum_begin<LOC, AG>(sh, lep, nwr(), redg, part, true, false);
        const AG beta = sqrt(xsum_end<LOC, AG>(sh, lep++, true, false));
        if (!LOC && !sh->ok) return;
        int k = 0;
        if constexpr (LS) {
        if (beta > AG(0)) {
            // ---- GMRES with MGS in its one-reduction form (inverse compact WY, lagged
            // normalisation; Swirydowicz et al. 2020): one vector reduction per
            // iteration gives Q_j^T u_j, ||u_j||^2, Q_j^T w and u_j^T w for the not yet
            // normalised u_j and w = op(u_j); then r = ||u_j|| is h_{j,j-1}, q_j = u_j / r,
            // row j of L = (q_i^T q_k)_{i>k} is Q_j^T u_j / r, and the MGS coefficients of
            // column j are h = (I + L)^{-1} [Q_j^T w / r ; u_j^T w / r^2].  Three grid-wide
            // waits per iteration (after the first product, the reduction, and the
            // update that publishes u_{j+1}) instead of j + 3.
            //
            // The Givens rotations of column c (complete once iteration c+1 has
            // r_{c+1} = h_{c+1,c}) run on warp 0 during iteration c+2's inner
            // products, which the other warps compute; the stop test follows them, so a
            // solve that converges at column c has done one more product and inner-
            // product pass than it uses.  The columns alternate between two buffers
            // (hc, and yv until the back substitution).
            const int nwp = BT >> 5, lane = tid & 31, wid = tid >> 5;
            // (rows in u_g; the scalars, partials and T in its arithmetic type)
            TG* wsm = ws + a.rb;                 // w for the block's rows
            AG* sred = (AG*)(wsm + a.rb);        // 2 (kmax + 1) inner products, summed over blocks
            AG* lrow = sred + 2 * (kmax + 1);    // row j of L (kmax + 1)
            AG* upa = lrow + (kmax + 1);         // unit partials (kmax + 33 each)
            AG* upc = upa + (kmax + 33);
            AG* hout = upc + (kmax + 33);        // h (kmax + 1)
            // between the unit partials' sums and h: the newest row of T and the warps' sums over blocks
            AG* tnew = upa;
            AG* psum = upc;
            AG* ttri = hout + (kmax + 1) + ir_psum_more(kmax, sizeof(AG));  // rows 0 .. jl-1 of T = (I + L)^{-1}, packed
            AG* Tg = (AG*)a.L;                   // every row of T, packed (block 0 writes)
            AG* pv2 = (AG*)a.pvec;               // block partials: [block][value] (single), [value][block] (double)
            const int pvs = 2 * (kmax + 1);
            double* colb[2] = {hc, yv};          // column c of H (entries 0..c+1) in colb[c & 1]
            auto tri = [](int i) -> int { return i * (i - 1) / 2; };
            // (row i of T, T(i, m) for m < i: rows jl.. from global memory once a barrier has
            // followed block 0's store)
            // with a rotating block (sblock) only it runs the rotations, and the row blocks'
            // warp 0 joins the inner products
            const bool sblock = a.sblock != 0;
            const bool rotates = !sblock || bid == G - 1;
            auto givens = [&](int c) {
                givens_warp(sh, cs, sn, g, colb[c & 1], a.R + (size_t)c * (kmax + 1), a.gpub, c, kmax, (double)beta,
                            bid == 0 || sblock, sblock);
            };
            if (tid == 0) g[0] = (double)beta;
            // units of the inner products: S row segments per vector, whole multiples of 32 VN
            // rows (chunks), S chosen so that the busiest of the nwu warps finishes first, a
            // unit costing its chunks plus about four chunks for its two warp reductions (at
            // most kmax + 33 units: the partials' storage).  stab[nv] for nv = 1..kmax+1
            // vectors, made once per solve (32-bit arithmetic; 64-bit division is slow here).
            int* stab = reinterpret_cast<int*>(ttri + (size_t)a.jl * (a.jl - 1) / 2);
            // partial sums of the T row's column groups
            AG* tpart = reinterpret_cast<AG*>(((uintptr_t)(stab + kmax + 2) + 15) & ~(uintptr_t)15);
            // the block's rows of basis vectors 0 .. nq-1
            TG* qc = reinterpret_cast<TG*>(tpart + ir_tpart(kmax));
            const int nq = a.nq, rbq = (int)a.rb;
            constexpr int CK = 32 * VN;
            const int nwu = sblock ? nwp : nwp - 1;
            if (it == 0) {
                const int smax = rows > 0 ? (rows + CK - 1) / CK : 1;
#pragma unroll 1
                for (int nv = 1 + tid; nv <= kmax + 1; nv += BT) {
                    int best = INT_MAX, sb = 1;
#pragma unroll 1
                    for (int s2 = 1; s2 <= smax && nv * s2 <= kmax + 33; s2++) {
                        const int segc = ((rows + s2 - 1) / s2 + CK - 1) / CK;
                        const int cost = ((nv * s2 + nwu - 1) / nwu) * (segc + 4);
                        if (cost < best) { best = cost; sb = s2; }
                    }
                    stab[nv] = sb;
                }
            }
#pragma unroll 1
            for (int j = 0; j <= kmax; j++) {
                const bool prod = j < kmax;
                // w = P (A u_j) (left) or A (P u_j) (right) in u_p, stored in u_g; u_j is read
                // from the published wbuf (the first u_0 is z).  (Running the second product
                // on warps 1.. beside the rotations slowed both: the FP64 instructions hold
                // up their sub-partition.)
                if (prod) {
                    if (hasP) {
                        first(tbuf + r0);
                        if (!xbar<LOC>(sh)) return;
                        second(wsm);
                    } else {
                        first(wsm);
                    }
                }
                __syncthreads();
                const int nv = j + 1;
                const int S = stab[nv];
                if (wid == 0 && j >= 2 && rotates) givens(j - 2);
                if (sblock || wid > 0) {
                    // ---- block partials: units (vector i, row segment), vector j being u_j
                    // itself; a_i = q_i . u_j (a_j = ||u_j||^2), c_i = q_i . w (c_j = u_j . w).
                    // Each lane reads VN consecutive rows per 16-byte load
                    const int segr = ((rows + S - 1) / S + CK - 1) / CK * CK;
#pragma unroll 1
                    for (int unit = wid - (sblock ? 0 : 1); unit < nv * S; unit += nwu) {
                        const int i = unit / S, e0 = (unit - i * S) * segr, e1 = min(rowsp, e0 + segr);
                        // (binary32: four partial sums, so that a lane's chains are no longer than when the
                        // block had 28 warps to split a vector over)
                        constexpr int NA = sizeof(AG) == 4 ? 4 : 1;
                        AG sa[NA], sc[NA];
#pragma unroll
                        for (int e = 0; e < NA; e++) sa[e] = sc[e] = AG(0);
                        auto take = [&](const TV q4, int row) {
                            const TV u4 = *reinterpret_cast<const TV*>(ws + row);
                            const TV w4 = *reinterpret_cast<const TV*>(wsm + row);
                            TG qe[VN], ue[VN], we[VN];
                            memcpy(qe, &q4, sizeof(TV));
                            memcpy(ue, &u4, sizeof(TV));
                            memcpy(we, &w4, sizeof(TV));
#pragma unroll
                            for (int e = 0; e < VN; e++) {
                                sa[e % NA] = fma((AG)qe[e], (AG)ue[e], sa[e % NA]);
                                sc[e % NA] = fma((AG)qe[e], (AG)we[e], sc[e % NA]);
                            }
                        };
                        if (i == j || i < nq) {
                            // u_j, or a basis vector whose rows are in shared memory
                            const TG* qs = i == j ? ws : qc + i * rbq;
#pragma unroll 2
                            for (int row = e0 + VN * lane; row < e1; row += CK) {
                                const TV q4 = *reinterpret_cast<const TV*>(qs + row);
                                take(q4, row);
                            }
                        } else {
                            // IQ 16-byte loads of q issued together, then consumed in row order
                            constexpr int IQ = 8;
                            const TG* qb = V + (int64_t)i * a.ldv + r0;
#pragma unroll 1
                            for (int rq = e0 + VN * lane; rq < e1; rq += IQ * CK) {
                                TV q4[IQ];
#pragma unroll
                                for (int uu = 0; uu < IQ; uu++)
                                    // (clamped, not predicated: under one condition with its use
                                    // a load is not issued ahead)
                                    q4[uu] = __ldcg(reinterpret_cast<const TV*>(qb + min(rq + uu * CK, e1 - VN)));
#pragma unroll
                                for (int uu = 0; uu < IQ; uu++)
                                    if (rq + uu * CK < e1) take(q4[uu], rq + uu * CK);
                            }
                        }
                        if constexpr (sizeof(AG) == 4) {
                            const AG sv = warp_sum2(tree_sum(sa), tree_sum(sc));
                            if (lane == 0) upa[unit] = sv;
                            if (lane == 16) upc[unit] = sv;
                        } else {
                            const AG va = wsum(sa[0]), vc = wsum(sc[0]);
                            if (lane == 0) { upa[unit] = va; upc[unit] = vc; }
                        }
                    }
                }
                __syncthreads();
                // column j-2 converged: k = j-1 columns (this iteration's products are unused);
                // with a rotating block its verdict comes with the exchange round below
                if (!sblock && j >= 2 && sh->resid <= a.tau) { k = j - 1; break; }
#pragma unroll 1
                for (int v = tid; v < 2 * nv; v += BT) {
                    const AG* src = v < nv ? upa + v * S : upc + (v - nv) * S;
                    AG acc = AG(0);
#pragma unroll 1
                    for (int sg = 0; sg < S; sg++) acc += src[sg];
                    if (sizeof(AG) == 4) pv2[(size_t)bid * pvs + v] = acc;
                    else pv2[(size_t)v * G + bid] = acc;
                }
                // ---- the reduction over blocks (the partials published by an exchange round).
                // While the block waits, its other warps form row r = j-1 of T = (I + L)^{-1},
                // t_r = -l_r^T T (row r of (I + L) T = I), which h needs below: column by column,
                // t_{r,m} = -(l_{r,m} + sum_{m < k < r} l_{r,k} T(k, m)), a warp per 32 columns and
                // chunk of the rows k, so the reads T(k, m) of one row k are consecutive over the
                // lanes; the chunks' partials are added in order afterwards.
                const int tr = j - 1;
                const int tch = (max(tr, 1) + 31) >> 5;           // 32-column chunks of row r
                const int tgr = max(1, min((nwp - 1) / tch, 8));  // row groups
                auto trow = [&]() {
                    if (tr < 1) return;
                    const int kc = (tr + tgr - 1) / tgr;
#pragma unroll 1
                    for (int u = wid - 1; u < tch * tgr; u += nwp - 1) {
                        const int gq = u / tch, ch = u - gq * tch, m = 32 * ch + lane;
                        AG acc = AG(0);
                        const int kb = max(m + 1, gq * kc), ke = min(tr, (gq + 1) * kc);
                        if (m < tr) {
                            int k2 = kb;
                            const int kn = min(ke, a.jl);
#pragma unroll 4
                            for (; k2 < kn; k2++) acc = fma(lrow[k2], ttri[tri(k2) + m], acc);
                            // (rows from L2, sixteen loads in flight: with many columns a warp has
                            // every row of its 32)
                            constexpr int UQ = 16;
#pragma unroll 1
                            for (; k2 < ke; k2 += UQ) {
                                AG tv[UQ];
#pragma unroll
                                for (int e = 0; e < UQ; e++) tv[e] = ldcg(&Tg[tri(min(k2 + e, ke - 1)) + m]);
#pragma unroll
                                for (int e = 0; e < UQ; e++)
                                    if (k2 + e < ke) acc = fma(lrow[k2 + e], tv[e], acc);
                            }
                        }
                        tpart[gq * (32 * tch) + m] = acc;
                    }
                };
                unsigned done = 0;
                if (!xbar_flag<LOC>(sh, lep++, sblock && bid == G - 1 && j >= 2 && sh->resid <= a.tau ? 1u : 0u, &done, trow))
                    return;
                if (done) {
                    k = j - 1;
                    break;
                }
                for (int m = tid; m < tr; m += BT) {
                    AG acc = AG(0);
#pragma unroll 1
                    for (int gq = 0; gq < tgr; gq++) acc += tpart[gq * (32 * tch) + m];
                    const AG t = -(lrow[m] + acc);
                    tnew[m] = t;
                    if (tr < a.jl) ttri[tri(tr) + m] = t;
                    if (bid == 0) Tg[tri(tr) + m] = t;
                }
                // the sums over blocks of the 2 nv partials, each in the same order: every block
                // sums them all, or, when that would read many partials (2 nv G >= IR_DIST_MIN),
                // block b sums the values b, b + G, ... and publishes them for one more exchange
                // round.  Single: [block][value], the warps split into one part per 32 values and
                // each part's warps over the blocks, lanes over the values, then the warps' sums
                // in order (the blocks' stores are whole lines, and one trip to L2 serves every
                // value); double: [value][block], lanes over the blocks, on the integer pipe.
                if (2 * nv * G < IR_DIST_MIN) {
                    if constexpr (sizeof(AG) == 4) {
                        // (at most nine roundings a sum: 152 blocks on four warps make six in a lane and two
                        // over the warps; a lane for five blocks and a shuffle tree made nine too)
#pragma unroll 1
                        for (int v0 = 0; v0 < 2 * nv; v0 += SUMV) {
                            const int sv = min(SUMV, 2 * nv - v0);
                            const int nc = (sv + 31) >> 5, nws = nwp / nc;
                            const int v = 32 * (wid / nws) + lane, wsb = wid % nws;
                            if (v < sv) {
                                const AG* src = pv2 + wsb * pvs + v0 + v;
                                const int step = nws * pvs;
                                psum[wsb * 32 * nc + v] = strided_sum<12, AG>(
                                    (G - wsb + nws - 1) / nws, [&](int k) { return ldcg(src + k * step); });
                            }
                            __syncthreads();
                            const int nsum = min(nws, G);
                            for (int v2 = tid; v2 < sv; v2 += BT) {
                                sred[v0 + v2] = strided_sum<4, AG>(nsum, [&](int w) { return psum[w * 32 * nc + v2]; });
                            }
                            __syncthreads();
                        }
                    } else {
#pragma unroll 1
                        for (int v0 = wid; v0 < 2 * nv; v0 += nwp) {
                            AG x0[SPL];
#pragma unroll
                            for (int e = 0; e < SPL; e++) {
                                const int b = lane + 32 * e;
                                x0[e] = b < G ? ldcg(&pv2[(size_t)v0 * G + b]) : AG(0);
                            }
                            const AG acc = warp_sum_fx_n<SPL>(x0);
                            if (lane == 0) sred[v0] = acc;
                        }
                        __syncthreads();
                    }
                } else {
                    AG* tot = (AG*)a.pvec + (size_t)2 * MAX_GRID * (kmax + 1);
#pragma unroll 1
                    for (int t = wid; bid + t * G < 2 * nv; t += nwp) {
                        const int v0 = bid + t * G;
                        AG acc0 = AG(0);
#pragma unroll
                        for (int e = 0; e < SPL; e++) {
                            const int b = lane + 32 * e;
                            if (b < G) acc0 += ldcg(&pv2[sizeof(AG) == 4 ? (size_t)b * pvs + v0 : (size_t)v0 * G + b]);
                        }
                        acc0 = wsum(acc0);
                        if (lane == 0) tot[v0] = acc0;
                    }
                    if (!xbar<LOC>(sh)) return;
                    for (int v = tid; v < 2 * nv; v += BT) sred[v] = ldcg(&tot[v]);
                    __syncthreads();
                }
                const AG rr = j == 0 ? beta : sqrt(sred[j]);
                if (j >= 1 && tid == 0) colb[(j - 1) & 1][j] = (double)rr;  // h_{j,j-1}
                if (j >= 1 && (rr == AG(0) || !prod)) {
                    // breakdown or the iteration cap: column j-1 is the last one
                    __syncwarp();
                    if (wid == 0 && rotates) givens(j - 1);
                    __syncthreads();
                    k = j;
                    if (rr == AG(0)) flags |= 4;
                    break;
                }
                if (!prod) break;  // kmax = 0
                // ---- row j of L, l_j = a / r, and h = (I + L)^{-1} [c / r ; (u_j . w / r) / r], the
                // same in every block: h_i = (c_i + sum_{m < i} T(i, m) c_m) / r for i < j (a warp
                // per row), then h_j = b_j - l_j . h (in every warp: no barrier for one value), so
                // row j of T is not needed before the next column.
                for (int i = tid; i < j; i += BT) lrow[i] = sred[i] / rr;
                // (lane t keeps the sum of the warp's t-th row: one division for 32 rows, in double
                // a third of the time of this part with many columns)
                AG mine = AG(0);
#pragma unroll 1
                for (int i = wid, t = 0; i < j; i += nwp, t++) {
                    const AG* ti = i == tr ? tnew : (i < a.jl ? ttri + tri(i) : Tg + tri(i));
                    const bool near = i == tr || i < a.jl;
                    AG acc = AG(0);
                    if (near) {
#pragma unroll 2
                        for (int m = lane; m < i; m += 32) acc = fma(ti[m], sred[nv + m], acc);
                    } else {
                        constexpr int UQ = 8;
#pragma unroll 1
                        for (int m = lane; m < i; m += 32 * UQ) {
                            AG tv[UQ];
#pragma unroll
                            for (int e = 0; e < UQ; e++) tv[e] = ldcg(ti + min(m + 32 * e, i - 1));
#pragma unroll
                            for (int e = 0; e < UQ; e++)
                                if (m + 32 * e < i) acc = fma(tv[e], sred[nv + m + 32 * e], acc);
                        }
                    }
                    acc = wsum(acc);
                    const int tl = t & 31;
                    if (lane == tl) mine = sred[nv + i] + acc;
                    if (tl == 31 || i + nwp >= j) {
                        if (lane <= tl) hout[i - nwp * (tl - lane)] = mine / rr;
                    }
                }
                __syncthreads();
                AG hjj = AG(0);
#pragma unroll 1
                for (int m = lane; m < j; m += 32) hjj = fma(lrow[m], hout[m], hjj);
                hjj = (sred[2 * nv - 1] / rr) / rr - wsum(hjj);
                if (rotates) {
                    double* hj = colb[j & 1];
                    for (int i = tid; i < j; i += BT) hj[i] = (double)hout[i];
                    if (tid == 0) hj[j] = (double)hjj;
                }
                // ---- q_j = u_j / r into V, and u_{j+1} = w / r - Q_{j+1} h (the block's rows,
                // published for the next product)
                // (a thread takes VN consecutive rows, UB basis vectors at a time: 16-byte loads;
                // basis vectors 0 .. nq-1 from shared memory)
                TG* Vj = V + (int64_t)j * a.ldv + r0;
                const Quot<AG> qr(rr);
                const int jq = min(j, nq);
#pragma unroll 1
                for (int ra = VN * tid; ra < rowsp; ra += VN * BT) {
                    AG acc[VN];
                    TG qs[VN], t[VN];
                    auto get = [](TG* to, const TG* from) {
                        const TV v = *reinterpret_cast<const TV*>(from);
                        memcpy(to, &v, sizeof(TV));
                    };
                    auto put = [](TG* to, const TG* from) {
                        TV v;
                        memcpy(&v, from, sizeof(TV));
                        *reinterpret_cast<TV*>(to) = v;
                    };
                    get(qs, ws + ra);
                    get(t, wsm + ra);
#pragma unroll
                    for (int e = 0; e < VN; e++) {
                        // q_j as stored (in u_g) is the vector the update subtracts
                        qs[e] = (TG)qr((AG)qs[e]);
                        acc[e] = fma(-hjj, (AG)qs[e], qr((AG)t[e]));
                    }
                    put(Vj + ra, qs);
                    if (j < nq) put(qc + j * rbq + ra, qs);
#pragma unroll 2
                    for (int i = 0; i < jq; i++) {
                        const AG h = hout[i];
                        get(t, qc + i * rbq + ra);
#pragma unroll
                        for (int e = 0; e < VN; e++) acc[e] = fma(-h, (AG)t[e], acc[e]);
                    }
                    constexpr int UB = 8;
                    const TG* Vi = V + r0 + ra;
#pragma unroll 1
                    for (int i0 = jq; i0 < j; i0 += UB) {
                        TV tv[UB];
#pragma unroll
                        for (int u = 0; u < UB; u++)
                            tv[u] = __ldcg(reinterpret_cast<const TV*>(Vi + (int64_t)min(i0 + u, j - 1) * a.ldv));
#pragma unroll
                        for (int u = 0; u < UB; u++) {
                            const AG h = i0 + u < j ? hout[i0 + u] : AG(0);
                            memcpy(t, &tv[u], sizeof(TV));
#pragma unroll
                            for (int e = 0; e < VN; e++) acc[e] = fma(-h, (AG)t[e], acc[e]);
                        }
                    }
#pragma unroll
                    for (int e = 0; e < VN; e++) t[e] = (TG)acc[e];
                    put(ws + ra, t);
                    put(wbuf + r0 + ra, t);
                }
                if (!xbar<LOC>(sh)) return;
            }
        }
        } else {
        if (beta > TG(0)) {
            // Gram-Schmidt rows of this thread: PF rows as UV vectors of VN consecutive
            // rows, vector u = rows vrow(u) .. vrow(u) + VN - 1 of the range, then rows
            // PF BT + tid (step BT); the group's load, the first partial and every round use it
            constexpr int UV = PF / VN;
            const int64_t m0 = sub ? min(a.n, (int64_t)bid * 2 * a.rb) : r0;
            const int mrows = sub ? (gs ? (int)(min(a.n, m0 + 2 * a.rb) - m0) : 0) : rows;
            const int mrowsp = (mrows + 31) & ~31;  // (V, wbuf and ws are zero in the padding rows)
            const int mfar = PF * BT + tid;
            auto vrow = [&](int u) -> int { return VN * (tid + u * BT); };
            // the prefetch set of basis vector Vb: out[u VN + e] = Vb[m0 + vrow(u) + e]
            auto vload = [&](const TG* Vb, TG* out) {
#pragma unroll
                for (int u = 0; u < UV; u++) {
                    if (vrow(u) < mrowsp) {
                        const TV t = __ldcg(reinterpret_cast<const TV*>(Vb + m0 + vrow(u)));
                        memcpy(out + u * VN, &t, sizeof(TV));
                    }
                }
            };
            TG hdiv = beta;
            if (tid == 0) {
                g[0] = (double)beta;
                sh->ibeta = 1.0 / (double)beta;
            }
            {
                const Quot<TG> qd(hdiv);
#pragma unroll 1
                for (int i = tid; i < rowsp; i += BT) V[r0 + i] = qd(ws[i]);
            }
            __syncthreads();  // (the prefetch below reads other threads' rows)
            // Modified Gram-Schmidt in rounds of MB vectors v_i .. v_{i+MB-1}: one exchange
            // gives c_e = v_{i+e} . w for the w that all earlier rounds have left, and the
            // coefficients MGS forms one after another follow from the inner products among
            // the round's vectors (gam, a few units in the last place), h_e = c_e - sum_{m<e}
            // (v_{i+e} . v_{i+m}) h_m: the inverse compact WY form of the one-reduction MGS
            // (Swirydowicz et al. 2020), MB columns at a time.  Those inner products are
            // v_m . w / ||w|| of the vector's own last round, summed beside ||w||^2.  An
            // exchange takes 1.2 to 2 us whatever it sums, the updates of a vector 0.2: a
            // round per vector (j + 1 exchanges) was most of an iteration.
            // Us per iteration at one / MB vectors a round: single n = 143350 52.6 / 35.5, double
            // (2D) n = 19650 52.1 / 46.0, n = 1024 on a cluster 30.4 / 30.2.
            constexpr int MB = XVec<TG>::N;
            // (gam: MG of them a round, in y's place, which is free until the back substitution:
            // single 24 (kmax / 4 + 1) bytes, double 8 (kmax / 2 + 1), of 8 (kmax + 2))
            TG* gam = reinterpret_cast<TG*>(yv);
            constexpr int MG = MB * (MB - 1) / 2;
            // the padding rows of the group's double range
            if (sub)
                for (int i = mrows + tid; i < mrowsp; i += BT) ws[i] = TG(0);
            bool done = false;
#pragma unroll 1
            for (int j = 0; j < kmax && !done; j++) {
                // ---- t = A v_j (left) or P v_j (right) in u_p; v_j formed from the
                // published w: w / h
                {
                    const Quot<TG> qd(hdiv);
                    if (qd.fast) product(rightP, XIn<TP, TG, LD_QUOT>{wbuf, hdiv, qd.y, 0}, tbuf + r0);
                    else product(rightP, XIn<TP, TG, LD_DIV>{wbuf, hdiv, qd.y, 0}, tbuf + r0);
                }
                // prefetch v_0 for the first Gram-Schmidt dot while the barrier runs
                // (with a group the range holds other blocks' rows of v_0, which are
                // published by this barrier when j = 0: the load waits for it)
                TG vc[MB][PF];
                auto vfirst = [&]() {
#pragma unroll
                    for (int e = 0; e < MB; e++)
                        if (e <= j) vload(V + e * a.ldv, vc[e]);
                };
                if (!sub && !a.orth) vfirst();
                if (!xbar<LOC>(sh)) return;
                if (sub && !a.orth) vfirst();
                // ---- w = P t (left) or A t (right) in u_p, stored in u_g (own rows, shared
                // memory); first MGS partial
                if (hasP) {
                    second(sub ? wbuf + r0 : ws);
                } else {
#pragma unroll 1
                    for (int i = tid; i < rows; i += BT) {
                        const TG v = (TG)ldcg(&tbuf[r0 + i]);
                        if (sub) wbuf[r0 + i] = v;
                        else ws[i] = v;
                    }
                }
                if (sub) {
                    // the group's blocks read their double range of the published w = P t
                    if (!xbar<LOC>(sh)) return;
#pragma unroll
                    for (int u = 0; u < UV; u++)
                        if (vrow(u) < mrowsp)
                            *reinterpret_cast<TV*>(ws + vrow(u)) = __ldcg(reinterpret_cast<const TV*>(wbuf + m0 + vrow(u)));
#pragma unroll 1
                    for (int i = mfar; i < mrows; i += BT) ws[i] = ldcg(&wbuf[m0 + i]);
                }
                part = AG(0);
                TG hn;
                if (a.orth) {
                    // ---- classical Gram-Schmidt applied twice in u_g: each pass forms all
                    // j+1 projections of the same w (one vector exchange), then subtracts them
                    TG* cvec = reinterpret_cast<TG*>(yv);  // free until the back substitution
                    const int lane = tid & 31, wid = tid >> 5, nwp = BT >> 5;
                    const GridBarrier gbar{a.gcount, a.err, a.limit, (unsigned)G};
                    __syncthreads();
#pragma unroll 1
                    for (int pass = 0; pass < 2; pass++) {
                        // (two parities of the partials: pass 0 and pass 1)
                        TG* pbase = (TG*)a.pvec + (size_t)pass * G * (kmax + 1);
#pragma unroll 1
                        for (int i = wid; i <= j; i += nwp) {
                            // (16-byte loads, eight or (double: fewer rows a lane) four in flight; the
                            // padding rows are zero)
                            constexpr int IQ = sizeof(TG) == 8 ? 4 : 8, CK = 32 * VN;
                            const TG* Vi = V + (int64_t)i * a.ldv + r0;
                            TG acc = TG(0);
#pragma unroll 1
                            for (int rq = VN * lane; rq < rowsp; rq += IQ * CK) {
                                TV q4[IQ];
#pragma unroll
                                for (int e = 0; e < IQ; e++)
                                    q4[e] = __ldcg(reinterpret_cast<const TV*>(Vi + min(rq + e * CK, rowsp - VN)));
#pragma unroll
                                for (int e = 0; e < IQ; e++)
                                    if (rq + e * CK < rowsp) {
                                        const TV w4 = *reinterpret_cast<const TV*>(ws + rq + e * CK);
                                        TG qe[VN], we[VN];
                                        memcpy(qe, &q4[e], sizeof(TV));
                                        memcpy(we, &w4, sizeof(TV));
#pragma unroll
                                        for (int t = 0; t < VN; t++) acc = fma(qe[t], we[t], acc);
                                    }
                            }
                            acc = wsum(acc);
                            if (lane == 0) pbase[(size_t)bid * (kmax + 1) + i] = acc;
                        }
                        if (LOC ? !xbar<LOC>(sh) : !grid_sync(gbar, &sh->gepoch, &sh->ok)) return;
#pragma unroll 1
                        for (int i = wid; i <= j; i += nwp) {
                            TG x0[SPL];
#pragma unroll
                            for (int e = 0; e < SPL; e++) {
                                const int b = lane + 32 * e;
                                x0[e] = b < G ? ldcg(&pbase[(size_t)b * (kmax + 1) + i]) : TG(0);
                            }
                            TG acc;
                            if constexpr (sizeof(TG) == 8) {
                                acc = warp_sum_fx_n<SPL>(x0);
                            } else {
                                acc = x0[0];
#pragma unroll
                                for (int e = 1; e < SPL; e++) acc += x0[e];
                                acc = wsum(acc);
                            }
                            if (lane == 0) cvec[i] = acc;
                        }
                        __syncthreads();
                        if (tid == 0)
                            for (int i = 0; i <= j; i++) hc[i] = pass == 0 ? (double)cvec[i] : (double)((TG)hc[i] + cvec[i]);
#pragma unroll 1
                        for (int ra = VN * tid; ra < rowsp; ra += VN * BT) {
                            constexpr int UB = 8;
                            const TG* Vr = V + r0 + ra;
                            TV t = *reinterpret_cast<const TV*>(ws + ra);
                            TG acc[VN];
                            memcpy(acc, &t, sizeof(TV));
#pragma unroll 1
                            for (int i0 = 0; i0 <= j; i0 += UB) {
                                TV tv[UB];
#pragma unroll
                                for (int e = 0; e < UB; e++)
                                    tv[e] = __ldcg(reinterpret_cast<const TV*>(Vr + (int64_t)min(i0 + e, j) * a.ldv));
#pragma unroll
                                for (int e = 0; e < UB; e++) {
                                    const TG h = i0 + e <= j ? cvec[i0 + e] : TG(0);
                                    TG q[VN];
                                    memcpy(q, &tv[e], sizeof(TV));
#pragma unroll
                                    for (int v = 0; v < VN; v++) acc[v] = fma(-h, q[v], acc[v]);
                                }
                            }
                            memcpy(&t, acc, sizeof(TV));
                            *reinterpret_cast<TV*>(ws + ra) = t;
                        }
                        __syncthreads();
                    }
                    part2 = AG(0);
                    for (int i = tid; i < rows; i += BT) {
                        const TG wv = ws[i];
                        wbuf[r0 + i] = wv;
                        part = fma(wv, wv, part);
                        in_turn(part, part2);
                    }
                    part = both(part, part2);
                    if (tid == 0) {
                        // rotations 0..j-1 on the new column
#pragma unroll 1
                        for (int q2 = 0; q2 < j; q2++) {
                            const double t0 = cs[q2] * hc[q2] + sn[q2] * hc[q2 + 1];
                            hc[q2 + 1] = -sn[q2] * hc[q2] + cs[q2] * hc[q2 + 1];
                            hc[q2] = t0;
                            if (bid == 0) a.R[(size_t)j * (kmax + 1) + q2] = hc[q2];
                        }
                    }
                } else {
                // the group's load gives each thread its Gram-Schmidt rows; without a
                // group the product wrote w in its own row order.  Basis entries are read
                // through L2 (ld.cg): with a group they include rows that other blocks
                // wrote
                if (!sub) __syncthreads();
                TG* wp = ws + vrow(0);
                TG c[MB];
                {
                    const int cnt = min(MB, j + 1);
#pragma unroll
                    for (int e = 0; e < MB; e++) {
                        c[e] = TG(0);
                        if (e < cnt) {
#pragma unroll
                            for (int u = 0; u < UV; u++)
                                if (vrow(u) < mrowsp) {
#pragma unroll
                                    for (int q = 0; q < VN; q++) c[e] = fma(vc[e][u * VN + q], wp[(size_t)u * VN * BT + q], c[e]);
                                }
                            TG c2 = TG(0);
#pragma unroll 1
                            for (int i = mfar; i < mrows; i += BT) {
                                c[e] = fma(ldcg(&V[e * a.ldv + m0 + i]), ws[i], c[e]);
                                in_turn(c[e], c2);
                            }
                            if (mfar < mrows) c[e] = both(c[e], c2);
                        }
                    }
                }
                // ---- modified Gram-Schmidt in u_g (blocks outside the group skip it)
                const TG* gr = gam;  // the round's
#pragma unroll 1
                for (int i = 0; i <= j && gs; i += MB, gr += MG) {
                    // prefetch the next round's vectors before waiting for this one's coefficients
                    const TG* Vi = V + (int64_t)i * a.ldv;
                    const TG* Vn = Vi + MB * a.ldv;
                    const int cnt = min(MB, j + 1 - i), nxt = min(MB, j + 1 - i - MB);
                    const bool last = nxt <= 0;
                    TG vn[MB][PF];
#pragma unroll
                    for (int e = 0; e < MB; e++)
                        if (e < nxt) vload(Vn + e * a.ldv, vn[e]);
                    xvec_begin<LOC, TG, MB>(sh, lep, nwr(), redg, c, false, sub);
                    // Givens, pipelined with the rounds: rotation q needs h_{q+1}; thread 0
                    // applies those that the rounds before this one completed, between
                    // publishing and polling
                    if (tid == 0) {
#pragma unroll 1
                        for (int pq = max(0, i - MB - 1); pq <= i - 2; pq++) {
                            const double c1 = cs[pq], s1 = sn[pq], ha = hc[pq], hb = hc[pq + 1];
                            const double t0 = c1 * ha + s1 * hb;
                            hc[pq + 1] = -s1 * ha + c1 * hb;
                            hc[pq] = t0;
                            if (bid == 0) a.R[(size_t)j * (kmax + 1) + pq] = t0;
                        }
                    }
                    TG h[MB];
                    xvec_end<LOC, 3, TG, MB>(sh, lep++, false, sub, gr, cnt, h);
                    if (!LOC && !sh->ok) return;
                    if (tid == 0) {
#pragma unroll
                        for (int e = 0; e < MB; e++)
                            if (e < cnt) hc[i + e] = (double)h[e];
                    }
                    // c: the next round's inner products, or after the last round ||w||^2 and,
                    // where v_{j+1} joins this round's vectors, w . v_{i+e}
#pragma unroll
                    for (int e = 0; e < MB; e++) c[e] = TG(0);
#pragma unroll
                    for (int u = 0; u < UV; u++) {
                        if (vrow(u) < mrowsp) {
                            TV t = *reinterpret_cast<TV*>(wp + (size_t)u * VN * BT);
                            TG wv[VN];
                            memcpy(wv, &t, sizeof(TV));
#pragma unroll
                            for (int e = 0; e < MB; e++)
                                if (e < cnt) {
#pragma unroll
                                    for (int q = 0; q < VN; q++) wv[q] = fma(-h[e], vc[e][u * VN + q], wv[q]);
                                }
                            if (last) {
#pragma unroll
                                for (int q = 0; q < VN; q++) c[0] = fma(wv[q], wv[q], c[0]);
#pragma unroll
                                for (int e = 0; e + 1 < MB; e++)
                                    if (e < cnt && cnt < MB) {
#pragma unroll
                                        for (int q = 0; q < VN; q++) c[e + 1] = fma(vc[e][u * VN + q], wv[q], c[e + 1]);
                                    }
                            } else {
#pragma unroll
                                for (int e = 0; e < MB; e++)
                                    if (e < nxt) {
#pragma unroll
                                        for (int q = 0; q < VN; q++) c[e] = fma(vn[e][u * VN + q], wv[q], c[e]);
                                    }
                            }
                            memcpy(&t, wv, sizeof(TV));
                            *reinterpret_cast<TV*>(wp + (size_t)u * VN * BT) = t;
                            if (last) *reinterpret_cast<TV*>(wbuf + m0 + vrow(u)) = t;
                        }
                    }
#pragma unroll
                    for (int e = 0; e < MB; e++)
#pragma unroll
                        for (int q = 0; q < PF; q++) vc[e][q] = vn[e][q];
                    TG c2[MB];
#pragma unroll
                    for (int e = 0; e < MB; e++) c2[e] = TG(0);
#pragma unroll 1
                    for (int r2 = mfar; r2 < mrows; r2 += BT) {
                        TG wv = ws[r2], ve[MB];
#pragma unroll
                        for (int e = 0; e < MB; e++)
                            if (e < cnt) {
                                ve[e] = ldcg(&Vi[e * a.ldv + m0 + r2]);
                                wv = fma(-h[e], ve[e], wv);
                            }
                        ws[r2] = wv;
                        if (last) {
                            wbuf[m0 + r2] = wv;
                            c[0] = fma(wv, wv, c[0]);
#pragma unroll
                            for (int e = 0; e + 1 < MB; e++)
                                if (e < cnt && cnt < MB) c[e + 1] = fma(ve[e], wv, c[e + 1]);
                        } else {
#pragma unroll
                            for (int e = 0; e < MB; e++)
                                if (e < nxt) c[e] = fma(ldcg(&Vn[e * a.ldv + m0 + r2]), wv, c[e]);
                        }
#pragma unroll
                        for (int e = 0; e < MB; e++) in_turn(c[e], c2[e]);
                    }
                    if (mfar < mrows) {
#pragma unroll
                        for (int e = 0; e < MB; e++) c[e] = both(c[e], c2[e]);
                    }
                }
                // the rotations that the rounds left
                if (gs && tid == 0) {
#pragma unroll 1
                    for (int q2 = max(0, j / MB * MB - 1); q2 < j; q2++) {
                        const double t0 = cs[q2] * hc[q2] + sn[q2] * hc[q2 + 1];
                        hc[q2 + 1] = -sn[q2] * hc[q2] + cs[q2] * hc[q2 + 1];
                        hc[q2] = t0;
                        if (bid == 0) a.R[(size_t)j * (kmax + 1) + q2] = t0;
                    }
                }
                // outside the group the sums are 0; block 0 stores the rotated diagonal
                // entry h_jj (rotations 0..j-1 applied) in the unused last row of R's
                // column j for the blocks outside the group
                if (!gs) {
#pragma unroll
                    for (int e = 0; e < MB; e++) c[e] = TG(0);
                }
                if (sub && bid == 0 && tid == 0) a.R[(size_t)j * (kmax + 1) + kmax] = hc[j];
                xvec_begin<LOC, TG, MB>(sh, lep, nwr(), redg, c, true, false);
                TG hv[MB];
                xvec_end<LOC, SPL, TG, MB>(sh, lep++, true, false, (const TG*)nullptr, 0, hv);
                if (!LOC && !sh->ok) return;
                hn = sqrt(hv[0]);
                // v_{j+1} . v_m for the vectors of its round (a warp whose FP64 work does not hold up thread 0's)
                if (tid == 32 && hn > TG(0)) {
                    const int q = (j + 1) % MB;
                    TG* gq = gam + (j + 1) / MB * MG + q * (q - 1) / 2;
#pragma unroll
                    for (int e = 0; e + 1 < MB; e++)
                        if (e < q) gq[e] = hv[e + 1] / hn;
                }
                }
                if (a.orth) {
                    xsum_begin<LOC, TG>(sh, lep, nwr(), redg, part, true, false);
                    hn = sqrt(xsum_end<LOC, TG>(sh, lep++, true, false));
                    if (!LOC && !sh->ok) return;
                }
                if (sub && !a.orth && !gs && tid == 0) hc[j] = __ldcg(&a.R[(size_t)j * (kmax + 1) + kmax]);
                // ---- v_{j+1} = w / h_{j+1,j} (own rows; with a group from the published w)
                if (hn > TG(0)) {
                    TG* Vn = V + (int64_t)(j + 1) * a.ldv + r0;
                    const Quot<TG> qd(hn);
#pragma unroll 1
                    for (int i = tid; i < rowsp; i += BT) Vn[i] = qd(sub ? ldcg(&wbuf[r0 + i]) : ws[i]);
                }
                // ---- the new Givens rotation in double (identical in every block);
                // rotations 0..j-1 were applied to this column during the rounds
                if (tid == 0) {
                    const double ha = hc[j], hs = (double)hn;
                    double dnj = sqrt(ha * ha + hs * hs);
                    double cj = 1.0, sj = 0.0;
                    if (dnj != 0.0) {
                        const Quot<double> qd(dnj);
                        cj = qd(ha);
                        sj = qd(hs);
                    }
                    cs[j] = cj;
                    sn[j] = sj;
                    hc[j] = dnj;
                    hc[j + 1] = hs;
                    const double gj = g[j];
                    g[j + 1] = -sj * gj;
                    g[j] = cj * gj;
                    sh->resid = fabs(g[j + 1]) * sh->ibeta;
                    if (bid == 0) a.R[(size_t)j * (kmax + 1) + j] = dnj;
                }
                __syncthreads();
                k = j + 1;
                hdiv = hn;
                if (hn == TG(0)) { flags |= 4; done = true; }
                else if (sh->resid <= a.tau) done = true;
            }
        }
        }
        if (beta > AG(0)) {
            // ---- y = R^{-1} g (double), d = V y in u_g, x = x + d in u
            if (!xbar<LOC>(sh)) return;  // R columns from block 0 (or the rotating block)
            if (LS && a.sblock)
                for (int t = tid; t <= k; t += BT) g[t] = __ldcg(&a.gpub[t]);
            __syncthreads();
            back_substitute(a.R, g, yv, k, kmax);
            // y in u_g's arithmetic, rounded once (a conversion holds the FP64 pipe as an
            // FP64 instruction does)
            AG* ya = reinterpret_cast<AG*>(hc);
            for (int t = tid; t < k; t += BT) ya[t] = (AG)yv[t];
            __syncthreads();
            decltype(abs_key(TU(0))) dkey = 0;  // this thread's largest |d| (as added to x, in u)
            if (rightP) {
                // right preconditioning: d = P (V_k y), the product in u_p stored in u_g
#pragma unroll 1
                for (int i = tid; i < rows; i += BT) wbuf[r0 + i] = (TG)basis_dot<TG, AG>(V + r0 + i, a.ldv, ya, k);
                if (!xbar<LOC>(sh)) return;
                first(tbuf + r0);
                __syncthreads();
            }
#pragma unroll 1
            for (int i = tid; i < rows; i += BT) {
                const TU d = rightP ? (TU)(TG)(TP)ldcg(&tbuf[r0 + i]) : (TU)basis_dot<TG, AG>(V + r0 + i, a.ldv, ya, k);
                const TU du = scale2<HK>(d, esc);
                dkey = max(dkey, abs_key(du));
                x[r0 + i] = (TU)(x[r0 + i] + du);
            }
            const unsigned long long kw = warp_max_key(abs_key(key_value(dkey)));
            if ((tid & 31) == 0) redd[tid >> 5] = kw;
            __syncthreads();
            if (tid < 32) {
                const unsigned long long kb = warp_max_key(tid < (BT >> 5) ? redd[tid] : 0ull);
                if (tid == 0) sh->dmax = key_value(kb);
            }
            __syncthreads();
        }
        if (bid == 0 && tid == 0) a.its[it] = k;
        steps = it + 1;
        // x must be complete before the next residual
        if (!xbar<LOC>(sh)) return;
    }
    if (bid == 0 && tid == 0) {
        a.out[0] = steps;
        a.out[1] = flags;
    }
}

// One system on its own grid, its blocks co-resident (a cooperative launch).
template <class TU, class TG, class TP, int RM, bool LS>
__global__ void __launch_bounds__(IR_BT, 1) k_ir(IrArgs a)
{
    ir_body<TU, TG, TP, RM, LS, false>(a, (int)blockIdx.x, (int)gridDim.x);
}

// The same for matrices whose entries (padding included) 32 bits may not count.
constexpr int64_t IR_WIDE = INT_MAX - 4096;
template <class TU, class TG, class TP, int RM, bool LS>
__global__ void __launch_bounds__(IR_BT, 1) k_ir_wide(IrArgs a)
{
    ir_body<TU, TG, TP, RM, LS, false, true>(a, (int)blockIdx.x, (int)gridDim.x);
}

// Systems of T blocks each, a thread-block cluster when T > 1: the one system
// `one` (args null), or the systems args[0 ..] of one team size of a batch
// (gmres_ir_solve_batch), blocks T i .. T i + T - 1 solving system i.  The
// hardware starts a cluster as soon as T SMs of one GPC are free, so a system
// with many iterations holds only its own SMs, and no block waits for one
// outside its cluster.
template <class TU, class TG, class TP, int RM, bool LS>
__global__ void __launch_bounds__(IR_BT, 1) k_ir_local(const __grid_constant__ IrArgs one,
                                                                     const IrArgs* __restrict__ args, int T)
{
    __shared__ IrArgs a;
    const int sys = (int)blockIdx.x / T;
    const uint32_t* from = reinterpret_cast<const uint32_t*>(args ? args + sys : &one);
    for (unsigned i = threadIdx.x; i < sizeof(IrArgs) / 4; i += blockDim.x) reinterpret_cast<uint32_t*>(&a)[i] = from[i];
    __syncthreads();
    if (T > 1) {
        // the blocks have all started (their shared memory may be written) once this returns
        cluster_arrive();
        cluster_wait();
    }
    ir_body<TU, TG, TP, RM, LS, true>(a, (int)blockIdx.x - sys * T, T);
}

// The kernels of one precision tuple, for run-time dispatch: `one` is
// k_ir, `wide` k_ir_wide, `local` k_ir_local.
struct IrKernels {
    const void* one = nullptr;
    const void* wide = nullptr;
    const void* local = nullptr;
};

template <class TU, class TG, class TP, int RM, bool LS>
void ir_kernels_set(IrKernels* k)
{
    k->one = (const void*)k_ir<TU, TG, TP, RM, LS>;
    k->wide = (const void*)k_ir_wide<TU, TG, TP, RM, LS>;
    k->local = (const void*)k_ir_local<TU, TG, TP, RM, LS>;
}

template <class TU, class TG, class TP>
void ir_kernels_t(int rm, bool ls, IrKernels* k)
{
    if (rm == 2) {
        if (ls) ir_kernels_set<TU, TG, TP, 2, true>(k);
        else ir_kernels_set<TU, TG, TP, 2, false>(k);
    } else {
        if (ls) ir_kernels_set<TU, TG, TP, 1, true>(k);
        else ir_kernels_set<TU, TG, TP, 1, false>(k);
    }
}

// Half Krylov storage (u_g or u_p = half): the one-reduction MGS only; the
// other forms are not instantiated (k->one stays null).
template <class TU, class TG, class TP>
void ir_kernels_ls(int rm, bool ls, IrKernels* k)
{
    if (!ls) return;
    if (rm == 2) ir_kernels_set<TU, TG, TP, 2, true>(k);
    else ir_kernels_set<TU, TG, TP, 1, true>(k);
}

// defined one per (u, u_g, u_p) in gmres_ir_k_<u><u_g><u_p>.cu (f single, d double)
void ir_kernels_fff(int rm, bool ls, IrKernels* k);
void ir_kernels_ffd(int rm, bool ls, IrKernels* k);
void ir_kernels_fdf(int rm, bool ls, IrKernels* k);
void ir_kernels_fdd(int rm, bool ls, IrKernels* k);
void ir_kernels_dff(int rm, bool ls, IrKernels* k);
void ir_kernels_dfd(int rm, bool ls, IrKernels* k);
void ir_kernels_ddf(int rm, bool ls, IrKernels* k);
void ir_kernels_ddd(int rm, bool ls, IrKernels* k);
// half (h) u_g and/or u_p: gmres_ir_k_x<u_g><u_p>.cu, both u in one unit
void ir_kernels_fhh(int rm, bool ls, IrKernels* k);
void ir_kernels_dhh(int rm, bool ls, IrKernels* k);
void ir_kernels_fhf(int rm, bool ls, IrKernels* k);
void ir_kernels_dhf(int rm, bool ls, IrKernels* k);
void ir_kernels_ffh(int rm, bool ls, IrKernels* k);
void ir_kernels_dfh(int rm, bool ls, IrKernels* k);

}  // namespace spai
