// SPAI column kernel for adaptive patterns (Grote-Huckle), one CTA of 16 warps
// per column: the steps and the arithmetic of k_spai_cta<S, true, 16>
// (spai_cta.cuh), bit for bit, with the index work done another way.  That
// kernel spent 230k cycles a step on random matrices of 16 entries per column:
// half in rho, where every candidate's thread walked its row of A and looked
// each index up in a hash of the shadow; the rest in block-wide bitonic sorts
// of the shadow and of up to 8192 candidates, and in barriers of warps without
// rows.
//   - Sorted sets come from bitmaps over the n indices in shared memory: set a
//     bit per index, scan the words' population counts, and an index's place in
//     the sorted set is its word's prefix plus the bits below it.  The shadow
//     I_k and the candidate set J~ are formed this way, without a sort or a hash.
//   - rho's numerators s^T b_j run over the entries (l, j) of the column lists of
//     A with s_l != 0 (the lists that made the candidates), whose values lie next
//     to them (bT, B's entries in the order of A^T); an entry is linked to its
//     candidate, whose thread adds its few entries in ascending l, the order of
//     the row of A.  ||b_j||^2 is formed once per matrix (k_bt).
//   - Householder: only the warps that hold rows take part, on a barrier of
//     their own, one barrier a reflector (the pivot row and the partial dot
//     products alternate between two buffers); R for the back substitution from
//     shared memory.
//   - Selection: each thread keeps its best candidate as one key; a round is
//     one block minimum.
// It takes matrices whose bitmap fits beside the tile (launch_spai_adapt), finite
// B, and rho over full columns (rho_restricted = 0); the others keep
// k_spai_cta.  Which columns outgrow the kernel (more than 512 shadow rows or
// a.cmax candidate entries) is the same, so a column's result does not depend
// on which of the two ran.  Random n = 20000, 16 per column: 52.6 -> 13.1 ms
// (u_f = double, n = 7000, 13 per column: 35.2 -> 23.6, bound by the FP64 pipe in the
// reflectors).  Of a step's 56k cycles the reflectors are 24k (1200 each, with a
// barrier, a square root and a division on the chain), the selection 5.6k, rho
// 5.4k, the back substitution 4.7k.  (A second barrier for the pivot column, which each warp
// has for its own rows: 14.35 against 14.2 ms for the whole build.)
#pragma once

#include "spai_cta.cuh"

namespace spai {

// per row j of A: B's entries into the order of A^T (bt, beside ri) and
// ||b_j||^2 (den) in the compute type, added in row order; *bad is set when an
// entry of B is not finite
template <class S>
__global__ void k_bt(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                     const S* __restrict__ bval, const int64_t* __restrict__ cp, const int32_t* __restrict__ ri,
                     S* __restrict__ bt, typename Compute<S>::T* __restrict__ den, int* __restrict__ bad)
{
    typedef typename Compute<S>::T C;
    bool nf = false;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        C d = 0;
        for (int64_t q = rp[j]; q < rp[j + 1]; q++) {
            const S v = bval[q];
            const C b = bvalue<S>(v);
            nf = nf || !isfinite(b);
            d = fma(b, b, d);
            int64_t lo = cp[col[q]], hi = cp[col[q] + 1] - 1;
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (ri[mid] < (int32_t)j) lo = mid + 1;
                else hi = mid;
            }
            bt[lo] = v;
        }
        den[j] = d;
    }
    if (nf) atomicOr(bad, 1);
}

constexpr int ADAPT_NW = 16, ADAPT_MM = 32 * ADAPT_NW, ADAPT_BT = 32 * ADAPT_NW;

// shared memory of k_spai_adapt.  The original tile W is dead while the
// candidates are handled: their entries (next, p, b) lie over it, and the
// bitmap with its prefixes after them or behind everything.
template <class C> struct AdaptSmem {
    size_t w, v, P, arow, mb, R, I, J, tmp, red, key, sc, cand, rho, bits, total;
    __host__ __device__ AdaptSmem(int64_t n, int cmax)
    {
        size_t off = 0;
        auto place = [&](size_t b) {
            const size_t at = off;
            off += align16(b);
            return at;
        };
        const size_t ent = align16((size_t)cmax * (4 + sizeof(C)));
        const size_t words = (size_t)((n + 31) >> 5);
        const size_t bmp = align16(words * 4) + align16(words * 2);
        const size_t tile = align16((size_t)ADAPT_MM * SPAI_LD * sizeof(C));
        // (the bitmap is also used while the tile is built: never over it)
        w = place(tile > ent ? tile : ent);
        v = place(2 * ADAPT_MM * sizeof(C));
        P = place(2 * ADAPT_NW * 33 * sizeof(C));
        arow = place(2 * 32 * sizeof(C));
        mb = place(32 * sizeof(C));
        R = place(32 * 33 * sizeof(C));
        I = place(ADAPT_MM * 4);
        J = place(32 * 4);
        tmp = place(64 * 4);
        red = place(33 * sizeof(C));
        key = place(2 * ADAPT_NW * 16);
        sc = place(8 * 4);
        cand = place((size_t)cmax * 4);
        rho = place((size_t)cmax * sizeof(C));
        bits = place(bmp);
        total = off;
    }
};

// barrier of the warps that hold rows
__device__ __forceinline__ void bar_rows(int nthreads)
{
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

// prefix[w] = set bits in words 0 .. w-1 of the bitmap; returns the total.  All
// threads; a barrier before (the bits are set) and after.
__device__ __forceinline__ int bitmap_scan(const uint32_t* bits, uint16_t* prefix, int words, int* tmp)
{
    const int per = (words + ADAPT_BT - 1) / ADAPT_BT, w0 = threadIdx.x * per, w1 = min(words, w0 + per);
    __syncthreads();
    int c = 0;
    for (int w = w0; w < w1; w++) c += __popc(bits[w]);
    int total;
    int at = block_excl_scan(c, tmp, &total);
    for (int w = w0; w < w1; w++) {
        prefix[w] = (uint16_t)at;
        at += __popc(bits[w]);
    }
    __syncthreads();
    return total;
}
__device__ __forceinline__ int bitmap_rank(const uint32_t* bits, const uint16_t* prefix, int key)
{
    return prefix[key >> 5] + __popc(bits[key >> 5] & ((1u << (key & 31)) - 1u));
}

// the smaller of (rho, j): order of the selection.  Non-negative rho order like
// their bits.
struct SelKey {
    unsigned long long r;  // bits of rho (all ones: none)
    int j;
    __device__ __forceinline__ bool less(const SelKey& o) const { return r < o.r || (r == o.r && j < o.j); }
};
__device__ __forceinline__ unsigned long long rho_bits(float v) { return (unsigned long long)__float_as_uint(v); }
__device__ __forceinline__ unsigned long long rho_bits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ SelKey warp_min_key(SelKey k)
{
    const unsigned FULL = 0xffffffffu;
    const unsigned h = (unsigned)(k.r >> 32);
    const unsigned mh = __reduce_min_sync(FULL, h);
    const unsigned ml = __reduce_min_sync(FULL, h == mh ? (unsigned)k.r : 0xffffffffu);
    SelKey o;
    o.r = ((unsigned long long)mh << 32) | ml;
    o.j = __reduce_min_sync(FULL, k.r == o.r ? k.j : INT_MAX);
    return o;
}

template <class S>
__global__ void __launch_bounds__(ADAPT_BT, 1) k_spai_adapt(SpaiArgs a)
{
    typedef typename Compute<S>::T C;
    constexpr int MM = ADAPT_MM, BT = ADAPT_BT, NW = ADAPT_NW;
    extern __shared__ __align__(16) unsigned char smem[];
    const AdaptSmem<C> L(a.n, a.cmax);
    C* const W = (C*)(smem + L.w);
    // the candidates' entries, over W: value, next entry of the candidate, shadow position
    C* const entb = W;
    uint16_t* const entn = (uint16_t*)(smem + L.w + (size_t)a.cmax * sizeof(C));
    uint16_t* const entp = entn + a.cmax;
    C* const vbuf = (C*)(smem + L.v);
    C* const Pbuf = (C*)(smem + L.P);
    C* const abuf = (C*)(smem + L.arow);
    C* const mb = (C*)(smem + L.mb);
    C* const R = (C*)(smem + L.R);
    int32_t* const I = (int32_t*)(smem + L.I);
    int32_t* const J = (int32_t*)(smem + L.J);
    int32_t* const tmp = (int32_t*)(smem + L.tmp);
    C* const red = (C*)(smem + L.red);
    SelKey* const keys = (SelKey*)(smem + L.key);
    int* const sc = (int*)(smem + L.sc);  // [0] nj, [2] flags from warp 0, [3] nadd
    int32_t* const cand = (int32_t*)(smem + L.cand);
    C* const rho = (C*)(smem + L.rho);
    const int words = (int)((a.n + 31) >> 5);
    uint32_t* const bits = (uint32_t*)(smem + L.bits);
    uint16_t* const prefix = (uint16_t*)(smem + L.bits + align16((size_t)words * 4));
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned FULL = 0xffffffffu;
    const int F = a.F;
    const S* bv = (const S*)a.bval;
    const S* bt = (const S*)a.bt;
    const C* den = (const C*)a.den;
    C* const s = vbuf;  // the residual

    for (int w = tid; w < words; w += BT) bits[w] = 0u;
    for (int64_t k = blockIdx.x; k < a.n; k += gridDim.x) {
        if (tid == 0) { sc[0] = a.Jcnt[k]; sc[2] = 0; }
        __syncthreads();
        int nj = sc[0];
        if (tid < nj) J[tid] = a.Jidx[k * F + tid];
        __syncthreads();
        int m = 0, ns = 0, fl = 0;
        bool deferred = false;
        C snorm = 0;
        // the column outgrew the tile or the candidate list: the large-shadow
        // kernel resumes it at `step` with the pattern in J
        auto defer = [&](int step) {
            if (tid < nj) a.Jidx[k * F + tid] = J[tid];
            if (tid == 0) {
                a.Jcnt[k] = nj;
                a.nsolve[k] = step;
                a.flags[k] = fl | sc[2];
                if (a.big) a.big[atomicAdd(a.nbig, 1)] = (int32_t)k;
                else atomicCAS(a.err, 0, SPAI_ERR_INTERNAL);
            }
            deferred = true;
            __syncthreads();
        };
        for (int step = 0;; step++) {
            // ---- gather: warp t, t + 16, ... takes row J[t] of A (column of B): the bits
            // of its row indices and k, their ranks, the tile [B(I,J) | e_k]
            int gc[2];
            S gv[2];
            bool more = false;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int t = wid + NW * h;
                gc[h] = -1;
                if (t < nj) {
                    const int64_t b = a.rp[J[t]], e = a.rp[J[t] + 1];
                    if (b + lane < e) {
                        gv[h] = bv[b + lane];
                        if (!bmarked<S>(gv[h])) {
                            gc[h] = a.col[b + lane];
                            atomicOr(&bits[gc[h] >> 5], 1u << (gc[h] & 31));
                        }
                    }
                    // (rows of more than 32 entries: the rest is read again below)
                    for (int64_t q = b + 32 + lane; q < e; q += 32) {
                        more = true;
                        if (!bmarked<S>(bv[q])) atomicOr(&bits[a.col[q] >> 5], 1u << (a.col[q] & 31));
                    }
                }
            }
            if (tid == 0) atomicOr(&bits[k >> 5], 1u << (k & 31));
            m = bitmap_scan(bits, prefix, words, tmp);
            const bool fits = m <= MM;
            if (fits) {
                for (int t = tid; t < m * SPAI_LD; t += BT) W[t] = C(0);
                // I_k: every word's indices at their ranks
                const int per = (words + BT - 1) / BT, w0 = tid * per, w1 = min(words, w0 + per);
                for (int w = w0; w < w1; w++) {
                    int at = prefix[w];
                    for (uint32_t x = bits[w]; x; x &= x - 1u) I[at++] = 32 * w + __ffs(x) - 1;
                }
                __syncthreads();
#pragma unroll
                for (int h = 0; h < 2; h++)
                    if (gc[h] >= 0) W[bitmap_rank(bits, prefix, gc[h]) * SPAI_LD + wid + NW * h] = to_c(gv[h]);
                if (__any_sync(FULL, more)) {
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const int t = wid + NW * h;
                        if (t >= nj) continue;
                        const int64_t e = a.rp[J[t] + 1];
                        for (int64_t q = a.rp[J[t]] + 32 + lane; q < e; q += 32)
                            if (!bmarked<S>(bv[q])) W[bitmap_rank(bits, prefix, a.col[q]) * SPAI_LD + t] = to_c(bv[q]);
                    }
                }
                if (tid == 0) W[bitmap_rank(bits, prefix, (int)k) * SPAI_LD + nj] = C(1);
            }
            __syncthreads();
            for (int w = tid; w < words; w += BT) bits[w] = 0u;
            if (!fits) {
                __syncthreads();
                defer(step);
                break;
            }
            // ---- Householder QR, tile in registers: warp w rows [32w, 32w+32), lane t column t;
            // warps whose rows all lie beyond |I_k| wait at the barrier below
            // Warp 0's rows move down one register a step (register i holds row c + i), so the
            // pivot row is always its register 0; finished rows of R go to shared memory.  The
            // even and odd rows' partial sums are k_spai_cta's: which of the two is which
            // alternates, their sum does not.
            const int nwa = (m + 31) >> 5;
            if (wid < nwa) {
                C col[32];
#pragma unroll
                for (int r = 0; r < 32; r++) {
                    const int row = 32 * wid + r;
                    col[r] = (row < m && lane <= nj) ? W[row * SPAI_LD + lane] : C(0);
                }
                const int steps = nj < m ? nj : m;
                constexpr int NV = 16 / sizeof(C);
                typedef typename std::conditional<sizeof(C) == 8, double2, float4>::type CV;  // 16 bytes
#pragma unroll 1
                for (int c = 0; c < steps; c++) {
                    C* const v = vbuf + (c & 1) * MM;
                    C* const P = Pbuf + (c & 1) * (NW * 33);
                    C* const arow = abuf + (c & 1) * 32;
                    // the pivot column (rows >= c): each warp's own rows, so a block barrier is
                    // needed for the partial sums and the pivot row only
                    if (lane == c) {
#pragma unroll
                        for (int r = 0; r < 32; r += NV) {
                            CV t;
                            memcpy(&t, &col[r], sizeof(CV));
                            *reinterpret_cast<CV*>(v + 32 * wid + r) = t;
                        }
                    }
                    if (wid == 0) arow[lane] = col[0];
                    __syncwarp();
                    // (single: v stays in registers for the update; double: read again)
                    constexpr bool KEEP = sizeof(C) == 4;
                    C vr[KEEP ? 32 : 1];
                    if constexpr (KEEP) {
#pragma unroll
                        for (int r = 0; r < 32; r += NV) {
                            const CV t = *reinterpret_cast<const CV*>(v + 32 * wid + r);
                            memcpy(&vr[r], &t, sizeof(CV));
                        }
                    }
                    auto vat = [&](int r) -> C {
                        if constexpr (KEEP) return vr[r];
                        else return v[32 * wid + r];
                    };
                    C g0 = 0, g1 = 0;
#pragma unroll
                    for (int r = 0; r < 32; r += 2) {
                        g0 = fma(vat(r), col[r], g0);
                        g1 = fma(vat(r + 1), col[r + 1], g1);
                    }
                    P[wid * 33 + lane] = g0 + g1;
                    bar_rows(32 * nwa);
                    C g = 0;
#pragma unroll 4
                    for (int w = 0; w < nwa; w++) g += P[w * 33 + lane];
                    const C sig2 = __shfl_sync(FULL, g, c);
                    const C x0 = arow[c];
                    const C nrm = rnd<S>(sqrt(sig2));
                    const bool upd = nrm != C(0) && lane > c && lane <= nj;
                    C f = 0, v0 = 0, alpha = 0;
                    const C act = arow[lane];
                    if (nrm != C(0)) {
                        alpha = x0 >= C(0) ? -nrm : nrm;
                        v0 = rnd<S>(x0 - alpha);
                        const C vtv = C(2) * nrm * (nrm + fabs(x0));
                        const C sv = g + (v0 - x0) * act;
                        f = rnd<S>((sv + sv) / vtv);
                    }
                    if (wid == 0) {
                        // row c of R, then the rows below move down
                        R[c * 33 + lane] = upd ? rnd<S>(act - f * v0) : (lane == c && nrm != C(0) ? alpha : act);
#pragma unroll
                        for (int r = 1; r < 32; r++) col[r - 1] = upd ? rnd<S>(col[r] - f * vat(r)) : col[r];
                        col[31] = C(0);
                    } else if (upd) {
#pragma unroll
                        for (int r = 0; r < 32; r++) col[r] = rnd<S>(col[r] - f * vat(r));
                    }
                }
                // ---- back substitution (warp 0 holds R): m_c = (y_c - sum_t R(c,t) m_t) / R(c,c)
                if (wid == 0) {
#pragma unroll 1
                    for (int r = steps; r < nj; r++) R[r * 33 + lane] = C(0);  // (no more rows than columns)
                    __syncwarp();
                    int f0 = 0;
                    C mv = 0;
#pragma unroll 1
                    for (int c = nj - 1; c >= 0; c--) {
                        const C rc = R[c * 33 + lane];
                        const C yc = R[c * 33 + nj], rcc = R[c * 33 + c];
                        C part = (lane > c && lane < nj) ? rc * mv : C(0);
                        part = warp_sum(part);
                        C mc = 0;
                        if (c < m && rcc != C(0)) mc = rnd<S>(rnd<S>(yc - part) / rcc);
                        else f0 = CF_SINGULAR;
                        if (lane == c) mv = mc;
                    }
                    if (lane < nj) mb[lane] = mv;
                    if (lane == 0 && f0) sc[2] |= f0;
                }
            }
            __syncthreads();
            // ---- explicit residual from the original tile
            C part = 0;
            if (tid < m) {
                C acc = 0;
#pragma unroll 4
                for (int c = 0; c < nj; c++) acc = fma(W[tid * SPAI_LD + c], mb[c], acc);
                const C sp = rnd<S>(rnd<S>(acc) - W[tid * SPAI_LD + nj]);
                s[tid] = sp;
                part = fma(sp, sp, part);
            }
            const C s2 = block_sum_det(part, red);
            snorm = rnd<S>(sqrt(s2));
            ns++;
            if (!isfinite((double)snorm)) fl |= CF_NONFINITE;
            if (snorm <= (C)a.eps) { fl |= CF_CONVERGED; break; }
            if (step >= a.alpha) { fl |= CF_ALPHA; break; }
            if (nj >= F) { fl |= CF_FILLCAP; break; }
            // ---- candidates: the column lists of A for the rows l of I with s_l != 0, minus J.
            // Entry e of the lists one after another (in ascending l); a warp per list
            int64_t lb = 0;
            int cntp = 0;
            if (tid < m && s[tid] != C(0)) {
                lb = a.cp[I[tid]];
                cntp = (int)(a.cp[I[tid] + 1] - lb);
            }
            int total = 0;
            const int off = block_excl_scan(cntp, tmp, &total);
            if (total > a.cmax) { defer(step); break; }  // redone from this step's solve
            // (entry e belongs to row p = entp[e]; a thread takes entries tid, tid + 512, ...: a.cmax
            // <= 8192, at most 16 of them, all their loads in flight)
            int64_t* const lbase = reinterpret_cast<int64_t*>(Pbuf);
            if (wid < nwa) {
                lbase[tid] = lb - off;
                for (int q = 0; q < cntp; q++) entp[off + q] = (uint16_t)tid;
            }
            __syncthreads();
            constexpr int EX = 16;
            int jx[EX];
            S bx[EX];
#pragma unroll
            for (int x = 0; x < EX; x++) {
                const int e = tid + BT * x;
                jx[x] = -1;
                if (e < total) {
                    const int64_t q = lbase[entp[e]] + e;
                    jx[x] = a.ri[q];
                    bx[x] = bt[q];
                }
            }
#pragma unroll
            for (int x = 0; x < EX; x++)
                if (jx[x] >= 0) {
                    entb[tid + BT * x] = bvalue<S>(bx[x]);
                    atomicOr(&bits[jx[x] >> 5], 1u << (jx[x] & 31));
                }
            __syncthreads();
            if (tid < nj) atomicAnd(&bits[J[tid] >> 5], ~(1u << (J[tid] & 31)));
            const int u = bitmap_scan(bits, prefix, words, tmp);
            if (u == 0) {
                // (the bits left: none)
                fl |= CF_NOCAND;
                break;
            }
            // link every entry to its candidate (heads in rho's storage)
            int32_t* const head = reinterpret_cast<int32_t*>(rho);
            constexpr int HS = sizeof(C) / 4;  // candidate t's head lies in rho[t]
            for (int t = tid; t < u; t += BT) head[t * HS] = 0xffff;
#pragma unroll
            for (int x = 0; x < EX; x++)
                if (jx[x] >= 0)
                    jx[x] = bits[jx[x] >> 5] >> (jx[x] & 31) & 1u ? bitmap_rank(bits, prefix, jx[x]) : -1;
            __syncthreads();
#pragma unroll
            for (int x = 0; x < EX; x++)
                if (jx[x] >= 0) entn[tid + BT * x] = (uint16_t)atomicExch(&head[jx[x] * HS], tid + BT * x);
            {
                const int per = (words + BT - 1) / BT, w0 = tid * per, w1 = min(words, w0 + per);
                for (int w = w0; w < w1; w++) {
                    int at = prefix[w];
                    for (uint32_t x = bits[w]; x; x &= x - 1u) cand[at++] = 32 * w + __ffs(x) - 1;
                    bits[w] = 0u;
                }
            }
            __syncthreads();
            // ---- rho_j for every candidate: its entries in ascending l, picked from the list
            // (||b_j||^2 of EB candidates in flight)
            C rs = 0;
            constexpr int EB = 8;
#pragma unroll 1
            for (int t0 = tid; t0 < u; t0 += EB * BT) {
                C dj[EB];
#pragma unroll
                for (int x = 0; x < EB; x++) dj[x] = t0 + x * BT < u ? den[cand[t0 + x * BT]] : C(0);
#pragma unroll
                for (int x = 0; x < EB; x++) {
                    const int t = t0 + x * BT;
                    if (t >= u) break;
                    const int h0 = head[t * HS];
                    C num = 0;
                    if (entn[h0] == 0xffff) {
                        num = fma(s[entp[h0]], entb[h0], num);
                    } else {
                        int last = -1;
                        for (;;) {
                            int nx = INT_MAX;
                            for (int e = h0; e != 0xffff; e = entn[e])
                                if (e > last && e < nx) nx = e;
                            if (nx == INT_MAX) break;
                            num = fma(s[entp[nx]], entb[nx], num);
                            last = nx;
                        }
                    }
                    C r2 = s2;
                    if (dj[x] > C(0)) r2 = s2 - num * num / dj[x];
                    const C r = sqrt(r2 > C(0) ? r2 : C(0));
                    rho[t] = r;  // (over the head, this thread's)
                    rs += r;
                }
            }
            const C mean = block_sum_det(rs, red) / (C)u;
            // ---- up to min(beta, F - nj) acceptable indices with the smallest rho
            const int room = F - nj;
            const int want = a.beta < room ? a.beta : room;
            auto best = [&](const SelKey& after) {
                // this thread's smallest acceptable key beyond `after`
                SelKey b{~0ull, INT_MAX};
                for (int t = tid; t < u; t += BT) {
                    const C r = rho[t];
                    if (!(r <= mean)) continue;
                    const SelKey kk{rho_bits(r), cand[t]};
                    if (after.less(kk) && kk.less(b)) b = kk;
                }
                return b;
            };
            SelKey mine = best(SelKey{0ull, -1});
            int nadd = 0;
            for (; nadd < want; nadd++) {
                const SelKey wk = warp_min_key(mine);
                SelKey* const kb = keys + (nadd & 1) * NW;
                if (lane == 0) kb[wid] = wk;
                __syncthreads();
                const SelKey bk = warp_min_key(lane < NW ? kb[lane] : SelKey{~0ull, INT_MAX});
                if (bk.r == ~0ull) break;  // nothing was acceptable
                if (tid == 0) {
                    int pos = nj + nadd;
                    while (pos > 0 && J[pos - 1] > bk.j) { J[pos] = J[pos - 1]; pos--; }
                    J[pos] = bk.j;
                }
                if (mine.r == bk.r && mine.j == bk.j) mine = best(bk);
            }
            __syncthreads();
            if (nadd == 0) { fl |= CF_NOCAND; break; }
            nj += nadd;
        }
        if (deferred) continue;
        fl |= sc[2];
        // ---- outputs: row k of P = mbar_k * d(J_k) (entries past |J_k| are never read)
        if (tid < nj) {
            const int j = J[tid];
            const C mv = mb[tid];
            a.Jidx[k * F + tid] = j;
            a.Praw[k * F + tid] = (double)mv * a.d[j];
            if (!isfinite((double)mv)) atomicOr(&sc[2], CF_NONFINITE);
        }
        __syncthreads();
        if (tid == 0) {
            a.Jcnt[k] = nj;
            a.colres[k] = (double)snorm;
            a.flags[k] = fl | sc[2];
            a.Icnt[k] = m;
            a.nsolve[k] = ns;
        }
        __syncthreads();
    }
}

// Adaptive patterns grow, so they run 16 warps per column (tiles of 512 rows):
// this kernel, or k_spai_cta where the bitmap does not fit (n beyond 444160 in half
// and single, 101376 in double, beside the longest candidate lists), rho is restricted to the shadow or B has an infinity or NaN
// (a.bt null).  cmax is k_spai_cta's in both, so the same columns go on in the
// large-shadow kernel.
template <class S>
int launch_spai_cta_t(const SpaiArgs& a0, bool adaptive, int num_sms, size_t smem_cap, cudaStream_t s)
{
    typedef typename Compute<S>::T C;
    if (!adaptive || !a0.bt) return launch_spai_cta_nw<S, 16>(a0, adaptive, num_sms, smem_cap, s);
    SpaiArgs a = a0;
    a.mmax = ADAPT_MM;
    while (a.cmax > 512 && cta_tile_bytes<C>(a.mmax, ADAPT_NW, a.rl, a.cmax) > smem_cap) a.cmax >>= 1;
    if (cta_tile_bytes<C>(a.mmax, ADAPT_NW, a.rl, a.cmax) > smem_cap) return SPAI_ERR_UNSUPPORTED;
    size_t dyn = 0;
    SPAI_CUDA_TRY(allow_max_dynamic_smem(k_spai_adapt<S>, &dyn));
    const size_t smem = AdaptSmem<C>(a.n, a.cmax).total;
    if (smem > dyn || a.cmax > 8192) return launch_spai_cta_nw<S, 16>(a0, adaptive, num_sms, smem_cap, s);
    int occ = 0;
    SPAI_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_spai_adapt<S>, ADAPT_BT, smem));
    if (occ < 1) return SPAI_ERR_UNSUPPORTED;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>(a.n, (int64_t)num_sms * occ));
    k_spai_adapt<S><<<(unsigned)blocks, ADAPT_BT, smem, s>>>(a);
    SPAI_CUDA_TRY(cudaGetLastError());
    return 0;
}

// B in the order of A^T and its column norms (k_bt)
template <class S>
int launch_spai_bt_t(int64_t n, const int64_t* rp, const int32_t* col, const void* bval, const int64_t* cp,
                     const int32_t* ri, void* bt, void* den, int* bad, int num_sms, cudaStream_t s)
{
    const int gb = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)num_sms * 16));
    k_bt<S><<<gb, 256, 0, s>>>(n, rp, col, (const S*)bval, cp, ri, (S*)bt, (typename Compute<S>::T*)den, bad);
    SPAI_CUDA_TRY(cudaGetLastError());
    return 0;
}

}  // namespace spai
