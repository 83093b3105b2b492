// kernels.cuh -- hand-written sm_103a kernels of the nested block solver:
// block-sparse products with fused epilogues, deterministic multi-dot /
// multi-axpy for CGS2 Arnoldi, the device Givens least-squares update and the
// AMG transfer operators.  Internal header (templates), included by the
// translation units that launch them.
#pragma once

#include <cooperative_groups.h>

#include <cstring>
#include <type_traits>
#include <utility>

#include "nbp_common.cuh"

namespace nbp {

// ===================================================== block-sparse products
// y = epilogue(M x) for a block CSR matrix with BR x BC blocks.  A group of G
// lanes walks one block row's values as one flat, contiguous array (perfectly
// coalesced loads whatever the block shape), keeps BR partial sums, and
// reduces them with xor shuffles inside the group.  Epilogues:
//   EPI_SET  y = Mx (+ rank-one term, LR)      EPI_ADD  y += Mx
//   EPI_SUB  y -= Mx                           EPI_RES  y = b - Mx
//   EPI_CHEB r = b - Mx; d = c1 d + c2 Dinv r; xout = x + d   (Chebyshev step)
//   EPI_POST M = A P, x = e the coarse correction, b the residual before the
//            restriction: d = c2 Dinv (b - M e); xout = xin + P e + d, i.e. the
//            prolongation and the first post-smoothing step (c1 = 0) in one
//            (sliced kernels k_sell and k_sellm)
enum Epi { EPI_SET = 0, EPI_ADD = 1, EPI_SUB = 2, EPI_RES = 3, EPI_CHEB = 4, EPI_POST = 5 };

struct SpmvArgs {
    int nbr;
    const int *rp, *ci;
    const void *val;
    const void *x;
    void *y;
    const void *b;          // EPI_RES / EPI_CHEB
    const void *dinv;       // EPI_CHEB: BR x BR per row (same type as vectors)
    void *d;                // EPI_CHEB: Chebyshev direction (in/out)
    void *xout;             // EPI_CHEB: x + d
    const void *xin;        // EPI_POST: the iterate before the correction
    const int *agg;         // EPI_POST: aggregate of each row (-1: none)
    double c1, c2;          // EPI_CHEB coefficients (FP64 vectors)
    float c1f, c2f;         // the same, pre-rounded for FP32 vectors (no FP64 work per element)
    const int *lr_rp, *lr_k, *lr_c;   // rank-one epilogue (EPI_SET only)
    const double *lr_val, *lr_f;
    // the factors r_k (a^k . x) taken by the product's own blocks where lr_rev is
    // 0 or 1 (see lr_factors; -1: read from lr_f): the outlets' vectors and
    // weights, and whether the blocks run from the last rows (1)
    const int *lr_optr, *lr_oidx;
    const double *lr_oval, *lr_r;
    int lr_n, lr_rev;
    int nslice;                       // sliced-ELL layout (k_sell): slices of C rows
    const long long *sl_ptr;
    const int *sl_ci;
    bool d_read, d_write;             // EPI_CHEB: d is read (c1 != 0) / written (a later step reads it)
    // device-driven loops: x, b and xout are column *jp of a basis where their
    // column stride is set (0: the pointer itself)
    const int *jp;
    long long x_ld, b_ld, out_ld;
};
// a vector of the product, its basis column taken on the device
__device__ __forceinline__ long long col_off(const SpmvArgs &a, long long ld) { return ld ? (long long)*a.jp * ld : 0; }

template <int BR, int BC, int G, typename VT, typename XT, int EPI, bool LR>
__global__ void __launch_bounds__(256) k_bspmv(SpmvArgs a) {
    using AT = XT;   // accumulate in the vector type (FP64 or FP32)
    constexpr int BB = BR * BC;
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int row = (int)(gid / G);
    const int lane = (int)(gid % G);
    if (row >= a.nbr) return;   // whole groups leave together (G divides 32)
    const unsigned wl = threadIdx.x & 31u;
    const unsigned mask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << (wl & ~(unsigned)(G - 1)));
    const int e0 = __ldg(a.rp + row);
    const int cnt = (__ldg(a.rp + row + 1) - e0) * BB;
    const VT *__restrict__ val = (const VT *)a.val + (long long)e0 * BB;
    const int *__restrict__ ci = a.ci + e0;
    // the first entry's value and column before the wait
    const VT v0 = lane < cnt ? __ldg(val + lane) : VT(0.f);
    const int c0 = lane < cnt ? __ldg(ci + lane / BB) : 0;
    pdl_wait();
    const XT *x = (const XT *)a.x + col_off(a, a.x_ld);
    AT acc0 = 0, acc1 = 0, acc2 = 0;
#pragma unroll 4
    for (int v = lane; v < cnt; v += G) {
        const int e = v / BB;
        const int rc = v - e * BB;
        const int r = rc / BC;
        const int c = rc - r * BC;
        const bool first = v == lane;
        const AT p = cvt<AT>(first ? v0 : __ldg(val + v)) * x[(long long)(first ? c0 : __ldg(ci + e)) * BC + c];
        if (BR == 1) acc0 += p;
        else {
            acc0 += (r == 0) ? p : AT(0);
            acc1 += (r == 1) ? p : AT(0);
            acc2 += (r == 2) ? p : AT(0);
        }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        acc0 += __shfl_xor_sync(mask, acc0, o);
        if (BR > 1) {
            acc1 += __shfl_xor_sync(mask, acc1, o);
            acc2 += __shfl_xor_sync(mask, acc2, o);
        }
    }
    if (lane >= BR) return;
    AT s = (lane == 0) ? acc0 : (lane == 1 ? acc1 : acc2);
    const long long idx = (long long)row * BR + lane;
    XT *y = (XT *)a.y;
    if (EPI == EPI_SET) {
        if (LR) {   // FP64 only on the rows that carry rank-one entries
            const int e0 = a.lr_rp[row], e1 = a.lr_rp[row + 1];
            if (e1 > e0) {
                double t = 0.0;
                for (int q = e0; q < e1; ++q)
                    if (a.lr_c[q] == lane) t += a.lr_f[a.lr_k[q]] * a.lr_val[q];
                s = (AT)((double)s + t);
            }
        }
        y[idx] = s;
    } else if (EPI == EPI_ADD) {
        y[idx] += s;
    } else if (EPI == EPI_SUB) {
        y[idx] -= s;
    } else if (EPI == EPI_RES) {
        y[idx] = ((const XT *)a.b + col_off(a, a.b_ld))[idx] - s;
    } else {   // EPI_CHEB, BR == BC
        const XT *b = (const XT *)a.b + col_off(a, a.b_ld);
        const XT *dinv = (const XT *)a.dinv + (long long)row * BR * BR + lane * BR;
        AT t;
        if (BR == 1) {
            t = dinv[0] * (b[idx] - s);
        } else {
            const AT r0 = b[(long long)row * 3 + 0] - acc0;
            const AT r1 = b[(long long)row * 3 + 1] - acc1;
            const AT r2 = b[(long long)row * 3 + 2] - acc2;
            t = dinv[0] * r0 + dinv[1] * r1 + dinv[2] * r2;
        }
        XT *d = (XT *)a.d;
        const AT c1 = sizeof(AT) == 4 ? (AT)a.c1f : (AT)a.c1, c2 = sizeof(AT) == 4 ? (AT)a.c2f : (AT)a.c2;
        const AT dn = (a.d_read ? c1 * d[idx] : AT(0)) + c2 * t;
        if (a.d_write) d[idx] = dn;
        ((XT *)a.xout + col_off(a, a.out_ld))[idx] = x[idx] + dn;
    }
}

// What a solve writes (x, b, d, bases, ...) is read with plain loads, never
// through the read-only path: in a device-driven loop a kernel may have started
// before its predecessor wrote it (see pdl_wait).
//
// Streamed loads of matrix values and columns: each is read once per
// product, so they can bypass L1 allocation (ld.global.nc.L1::no_allocate)
// and leave L1 to the x gathers, which neighbouring rows share.
__device__ __forceinline__ float lds(const float *p) {
    float v;
    asm volatile("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ double lds(const double *p) {
    double v;
    asm volatile("ld.global.nc.L1::no_allocate.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ int lds(const int *p) {
    int v;
    asm volatile("ld.global.nc.L1::no_allocate.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ int2 lds(const int2 *p) {
    int2 v;
    asm volatile("ld.global.nc.L1::no_allocate.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ __nv_bfloat16 lds(const __nv_bfloat16 *p) {
    unsigned short v;
    asm volatile("ld.global.nc.L1::no_allocate.b16 %0, [%1];" : "=h"(v) : "l"(p));
    __nv_bfloat16 r;
    memcpy(&r, &v, 2);
    return r;
}
__device__ __forceinline__ __nv_bfloat162 lds(const __nv_bfloat162 *p) {
    unsigned v;
    asm volatile("ld.global.nc.L1::no_allocate.b32 %0, [%1];" : "=r"(v) : "l"(p));
    __nv_bfloat162 r;
    memcpy(&r, &v, 4);
    return r;
}

// Matrix loads of the sliced layouts: streamed (no L1 allocation) for
// 32-row slices, whose warps read whole 128-byte segments; 8-row slices read
// quarter segments, and there the lines that L1 keeps serve the neighbouring
// components, so those loads stay cached.
template <bool STREAM, typename P> __device__ __forceinline__ P ldm(const P *p) {
    if constexpr (STREAM) return lds(p);
    else return __ldg(p);
}

// One pair of slots of the paired BF16 layout: columns c, values m, added in
// slot order (the first slot of the pair, then the second).
template <int BS>
__device__ __forceinline__ void pair_fma(const int2 c, const __nv_bfloat162 (&m)[BS * BS], const float *x,
                                         float &acc0, float &acc1, float &acc2) {
    if (BS == 1) {
        const float2 mm = __bfloat1622float2(m[0]);
        acc0 += mm.x * x[c.x];
        acc0 += mm.y * x[c.y];
    } else {
        const float xa0 = x[3LL * c.x], xa1 = x[3LL * c.x + 1], xa2 = x[3LL * c.x + 2];
        const float xb0 = x[3LL * c.y], xb1 = x[3LL * c.y + 1], xb2 = x[3LL * c.y + 2];
        float2 mm[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) mm[q] = __bfloat1622float2(m[q]);
        acc0 += mm[0].x * xa0 + mm[1].x * xa1 + mm[2].x * xa2;
        acc1 += mm[3].x * xa0 + mm[4].x * xa1 + mm[5].x * xa2;
        acc2 += mm[6].x * xa0 + mm[7].x * xa1 + mm[8].x * xa2;
        acc0 += mm[0].y * xb0 + mm[1].y * xb1 + mm[2].y * xb2;
        acc1 += mm[3].y * xb0 + mm[4].y * xb1 + mm[5].y * xb2;
        acc2 += mm[6].y * xb0 + mm[7].y * xb1 + mm[8].y * xb2;
    }
}

// Slots p0, p0 + step, ... of the paired BF16 layout (DMat::sl2_ptr) of one
// row: per pair, one int2 of columns and one bf16x2 per component; the two
// slots are added in slot order, as the unpaired loop adds them.  Several pairs
// (PairBatch) are loaded before any is used (more loads in flight per thread);
// the pairs are still added in ascending order.  The first batch is loaded
// by sell_pairs_load, before the kernel waits for its predecessor.
// 32-row slices (the fine level, HBM-bound): two pairs per step; 8-row slices
// (coarse levels) measured faster one pair at a time.
template <int BS, int C, int K = C == 32 ? 2 : 1> struct PairBatch {
    int2 c[K];
    __nv_bfloat162 m[K][BS * BS];
};
template <int BS, int C, int K>
__device__ __forceinline__ void sell_pairs_load(PairBatch<BS, C, K> &B, const SpmvArgs &a, long long base2, int np, int t,
                                                int p, int step) {
    constexpr int BB = BS * BS;
    const __nv_bfloat162 *__restrict__ val = (const __nv_bfloat162 *)a.val;
    const int2 *__restrict__ ci = (const int2 *)a.sl_ci;
#pragma unroll
    for (int u = 0; u < K; ++u) {
        if (p + u * step >= np) break;
        const long long g = base2 + (long long)C * (p + u * step);
        B.c[u] = ldm<C == 32>(ci + g + t);
#pragma unroll
        for (int q = 0; q < BB; ++q) B.m[u][q] = ldm<C == 32>(val + g * BB + t + q * C);
    }
}
template <int BS, int C, int K>
__device__ __forceinline__ void sell_pairs(PairBatch<BS, C, K> &B, const SpmvArgs &a, long long base2, int np, int t, int p0,
                                           int step, const float *x, float &acc0, float &acc1, float &acc2) {
    for (int p = p0; p < np; p += K * step) {
        if (p != p0) sell_pairs_load(B, a, base2, np, t, p, step);
#pragma unroll
        for (int u = 0; u < K; ++u)
            if (p + u * step < np) pair_fma<BS>(B.c[u], B.m[u], x, acc0, acc1, acc2);
    }
}

// The unpaired last slot of an odd-width slice of the paired layout: its
// columns at sl_ci[g + t] and value q at val[g bb + C q + t] (int and bf16
// units), g = the slice's slot offset + C (width - 1).
template <int BS, int C>
__device__ __forceinline__ void sell_single(const SpmvArgs &a, long long g, int t, const float *x,
                                            float &acc0, float &acc1, float &acc2) {
    const __nv_bfloat16 *__restrict__ val = (const __nv_bfloat16 *)a.val + g * (BS * BS) + t;
    const int c = ldm<C == 32>(a.sl_ci + g + t);
    if (BS == 1) {
        acc0 += __bfloat162float(ldm<C == 32>(val)) * x[c];
    } else {
        const float x0 = x[3LL * c], x1 = x[3LL * c + 1], x2 = x[3LL * c + 2];
        float m[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) m[q] = __bfloat162float(ldm<C == 32>(val + q * C));
        acc0 += m[0] * x0 + m[1] * x1 + m[2] * x2;
        acc1 += m[3] * x0 + m[4] * x1 + m[5] * x2;
        acc2 += m[6] * x0 + m[7] * x1 + m[8] * x2;
    }
}

// One slot of the unpaired layouts: its column and the block's values
template <int BB, typename VT> struct SlotBatch {
    int c;
    VT m[BB];
};
template <int BB, int C, typename VT>
__device__ __forceinline__ void slot_load(SlotBatch<BB, VT> &B, const VT *__restrict__ val, const int *__restrict__ ci,
                                          long long base, int t, int k) {
    const long long g = base + (long long)C * k;
    B.c = ldm<C == 32>(ci + g + t);
#pragma unroll
    for (int q = 0; q < BB; ++q) B.m[q] = ldm<C == 32>(val + g * BB + t + q * C);
}
template <int BS, typename VT, typename AT>
__device__ __forceinline__ void slot_fma(const SlotBatch<BS * BS, VT> &B, const AT *x, AT &acc0, AT &acc1,
                                         AT &acc2) {
    if constexpr (BS == 1) {
        acc0 += cvt<AT>(B.m[0]) * x[B.c];
    } else {
        const AT x0 = x[3LL * B.c], x1 = x[3LL * B.c + 1], x2 = x[3LL * B.c + 2];
        acc0 += cvt<AT>(B.m[0]) * x0 + cvt<AT>(B.m[1]) * x1 + cvt<AT>(B.m[2]) * x2;
        acc1 += cvt<AT>(B.m[3]) * x0 + cvt<AT>(B.m[4]) * x1 + cvt<AT>(B.m[5]) * x2;
        acc2 += cvt<AT>(B.m[6]) * x0 + cvt<AT>(B.m[7]) * x1 + cvt<AT>(B.m[8]) * x2;
    }
}

// Rank-one factors f_k = r_k (a^k . x) inside the product: a block whose rows
// [r0, r1) carry outlet entries takes the inner products of their outlets
// itself (at most kLrInline in any 256 rows, a rule the host has checked), in
// the order of k_lowrank_dots, instead of a launch before every product that
// does nothing else.  The few blocks that do run first where the outlets' rows
// are last (lr_rev), so that the others hide them.  Returns the first outlet of
// fs.  All 256 threads of the block.  Not inlined: its registers would cost
// every block's occupancy.
constexpr int kLrInline = 4;
template <typename XT>
__device__ __noinline__ int lr_factors(const SpmvArgs &a, int r0, int r1, const XT *x, double (&fs)[kLrInline]) {
    __shared__ int kfirst;
    __shared__ double red[kLrInline][8];
    r0 = min(r0, a.nbr);
    r1 = min(r1, a.nbr);
    const int e0 = a.lr_rp[r0], e1 = a.lr_rp[r1];
    if (e1 <= e0) return 0;   // uniform over the block
    const int tid = threadIdx.x;
    if (tid == 0) kfirst = a.lr_n;
    __syncthreads();
    for (int e = e0 + tid; e < e1; e += 256) atomicMin(&kfirst, a.lr_k[e]);
    __syncthreads();
    const int k0 = kfirst, nk = min(kLrInline, a.lr_n - k0);
    for (int q = 0; q < nk; ++q) {
        double s = 0.0;
        for (int e = a.lr_optr[k0 + q] + tid; e < a.lr_optr[k0 + q + 1]; e += 256)
            s += a.lr_oval[e] * (double)x[a.lr_oidx[e]];
        s = warp_sum(s);
        if ((tid & 31) == 0) red[q][tid >> 5] = s;
    }
    __syncthreads();
    if (tid < nk) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[tid][w];
        fs[tid] = a.lr_r[k0 + tid] * t;
    }
    __syncthreads();
    return k0;
}
// the rank-one terms of component q of a row with entries [e0, e1)
__device__ __forceinline__ double lr_term(const SpmvArgs &a, int e0, int e1, int q, const double *fs, int k0) {
    double t = 0.0;
    for (int e = e0; e < e1; ++e)
        if (a.lr_c[e] == q) t += (a.lr_rev >= 0 ? fs[a.lr_k[e] - k0] : a.lr_f[a.lr_k[e]]) * a.lr_val[e];
    return t;
}

// A row of the paired BF16 layout by one thread, summed as k_sellm's V threads
// per row sum it: pair p into chain p % V, an odd width's last slot into the
// chain whose turn comes next, then the chains in the order of the lanes' tree.
// The same bits from fewer threads: for the instances of a batch that together
// fill the GPU, where V threads per row only add work, and whose results must
// not depend on their neighbours.  48, 57 and 75 registers for V = 2, 4 and 8.
template <int BS, int C, int K, int V>
__device__ __forceinline__ void sell_chains(const SpmvArgs &a, long long base, int w, int t, float &acc0, float &acc1,
                                            float &acc2) {
    static_assert(V % K == 0, "whole steps of loads");
    const int np = w / 2;
    float s0[V] = {}, s1[V] = {}, s2[V] = {};
    PairBatch<BS, C, K> pb;
    sell_pairs_load(pb, a, base / 2, np, t, 0, 1);
    pdl_wait();
    const float *x = (const float *)a.x + col_off(a, a.x_ld);
    for (int p = 0; p < np; p += V) {
#pragma unroll
        for (int h = 0; h < V; h += K) {
            if (p + h >= np) break;
            if (p + h > 0) sell_pairs_load(pb, a, base / 2, np, t, p + h, 1);
#pragma unroll
            for (int u = 0; u < K; ++u)
                if (p + h + u < np) pair_fma<BS>(pb.c[u], pb.m[u], x, s0[h + u], s1[h + u], s2[h + u]);
        }
    }
    if (w & 1) {
        const int last = np % V;
#pragma unroll
        for (int h = 0; h < V; ++h)
            if (h == last) sell_single<BS, C>(a, base + (long long)C * (w - 1), t, x, s0[h], s1[h], s2[h]);
    }
#pragma unroll
    for (int o = V / 2; o > 0; o >>= 1)
#pragma unroll
        for (int h = 0; h < o; ++h) {
            s0[h] += s0[h + o];
            s1[h] += s1[h + o];
            s2[h] += s2[h + o];
        }
    acc0 = s0[0];
    acc1 = s1[0];
    acc2 = s2[0];
}

// Sliced-ELL product for square BS x BS blocks: one thread per block row, C
// rows per slice (C = 32: a warp per slice; C = 8 for matrices whose row
// lengths vary, to cut padding).  Every load of values and columns by the C
// threads of a slice is one contiguous segment (C x value bytes).  Same
// epilogues as k_bspmv (a.rp unused; a.sl_* describe the slices).  V > 1: the
// sums in the order of k_sellm's V threads per row (sell_chains; BF16 values).
template <int BS, typename VT, typename XT, int EPI, bool LR, int C, int K = C == 32 ? 2 : 1, int V = 1>
__global__ void __launch_bounds__(256) k_sell(SpmvArgs a) {
    using AT = XT;
    constexpr int BB = BS * BS;
    const int bx = LR && a.lr_rev == 1 ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    const int row = bx * blockDim.x + threadIdx.x;
    const int sl = row / C, t = row % C;
    const bool live = sl < a.nslice;
    if (!LR && !live) return;   // LR: whole blocks stay for lr_factors
    const long long base = live ? a.sl_ptr[sl] : 0;
    const int w = live ? (int)((a.sl_ptr[sl + 1] - base) / C) : 0;
    const VT *__restrict__ val = (const VT *)a.val;
    const int *__restrict__ ci = a.sl_ci;
    AT acc0 = 0, acc1 = 0, acc2 = 0;
    if constexpr (V > 1) {
        sell_chains<BS, C, K, V>(a, base, w, t, acc0, acc1, acc2);
    } else if constexpr (std::is_same<VT, __nv_bfloat16>::value) {   // paired layout: w / 2 pairs, then one slot if w is odd
        PairBatch<BS, C, K> pb;
        sell_pairs_load(pb, a, base / 2, w / 2, t, 0, 1);
        pdl_wait();
        const XT *x = (const XT *)a.x + col_off(a, a.x_ld);
        sell_pairs(pb, a, base / 2, w / 2, t, 0, 1, x, acc0, acc1, acc2);
        if (w & 1) sell_single<BS, C>(a, base + (long long)C * (w - 1), t, x, acc0, acc1, acc2);
    } else {
        SlotBatch<BB, VT> sb;
        if (w > 0) slot_load<BB, C>(sb, val, ci, base, t, 0);
        pdl_wait();
        const XT *x = (const XT *)a.x + col_off(a, a.x_ld);
        if (w > 0) slot_fma<BS, VT, AT>(sb, x, acc0, acc1, acc2);
#pragma unroll 2
        for (int k = 1; k < w; ++k) {
            SlotBatch<BB, VT> u;
            slot_load<BB, C>(u, val, ci, base, t, k);
            slot_fma<BS, VT, AT>(u, x, acc0, acc1, acc2);
        }
    }
    const XT *x = (const XT *)a.x + col_off(a, a.x_ld);
    __shared__ double fs[kLrInline];
    int k0 = 0;
    if (LR && a.lr_rev >= 0) k0 = lr_factors(a, bx * 256, bx * 256 + 256, x, fs);
    if (row >= a.nbr) return;
    AT accs[3] = {acc0, acc1, acc2};
    XT *y = (XT *)a.y;
    if (EPI == EPI_POST) {
        const XT *b = (const XT *)a.b;
        const XT *dinv = (const XT *)a.dinv + (long long)row * BB;
        const XT *xi = (const XT *)a.xin;
        XT *xo = (XT *)a.xout + col_off(a, a.out_ld);
        const int g = a.agg[row];
        const AT c2 = sizeof(AT) == 4 ? (AT)a.c2f : (AT)a.c2;
        AT r[3], e[3];
#pragma unroll
        for (int q = 0; q < BS; ++q) {
            r[q] = b[(long long)row * BS + q] - accs[q];
            e[q] = xi[(long long)row * BS + q];
            if (g >= 0) e[q] += x[(long long)g * BS + q];
        }
#pragma unroll
        for (int q = 0; q < BS; ++q) {
            AT tq = 0;
#pragma unroll
            for (int c = 0; c < BS; ++c) tq += dinv[q * BS + c] * r[c];
            const long long idx = (long long)row * BS + q;
            const AT dn = c2 * tq;
            if (a.d_write) ((XT *)a.d)[idx] = dn;
            xo[idx] = e[q] + dn;
        }
        return;
    }
    const bool lr = LR && EPI == EPI_SET;
    const int lr0 = lr ? a.lr_rp[row] : 0, lr1 = lr ? a.lr_rp[row + 1] : 0;
    if (EPI == EPI_CHEB) {
        const XT *b = (const XT *)a.b + col_off(a, a.b_ld);
        const XT *dinv = (const XT *)a.dinv + (long long)row * BB;
        XT *d = (XT *)a.d;
        XT *xo = (XT *)a.xout + col_off(a, a.out_ld);
        const AT c1 = sizeof(AT) == 4 ? (AT)a.c1f : (AT)a.c1, c2 = sizeof(AT) == 4 ? (AT)a.c2f : (AT)a.c2;
        AT r[3];
#pragma unroll
        for (int q = 0; q < BS; ++q) r[q] = b[(long long)row * BS + q] - accs[q];
#pragma unroll
        for (int q = 0; q < BS; ++q) {
            AT tq = 0;
#pragma unroll
            for (int c = 0; c < BS; ++c) tq += dinv[q * BS + c] * r[c];
            const long long idx = (long long)row * BS + q;
            const AT dn = (a.d_read ? c1 * d[idx] : AT(0)) + c2 * tq;
            if (a.d_write) d[idx] = dn;
            xo[idx] = x[idx] + dn;
        }
        return;
    }
#pragma unroll
    for (int q = 0; q < BS; ++q) {
        const long long idx = (long long)row * BS + q;
        AT s = accs[q];
        if (EPI == EPI_SET) {
            // the rank-one term in FP64, only on the rows that carry its
            // entries (outlet rows): GB300's FP64 pipe would otherwise hold
            // every warp for the conversions of every row
            if (lr && lr1 > lr0) s = (AT)((double)s + lr_term(a, lr0, lr1, q, fs, k0));
            y[idx] = s;
        } else if (EPI == EPI_ADD) {
            y[idx] += s;
        } else if (EPI == EPI_SUB) {
            y[idx] -= s;
        } else {
            y[idx] = ((const XT *)a.b + col_off(a, a.b_ld))[idx] - s;
        }
    }
}

// Sliced-ELL product for the rectangular coupling blocks (B: 3x1, C: 1x3):
// T threads per block row as in k_sellm (T = 1: one), slot values
// component-major as in k_sell (value q = r BC + c of the C slots at (slot
// base) * BR BC + C q + t).  Epilogues SET / ADD / SUB; FP64 or FP32 values.
template <int BR, int BC, typename VT, typename XT, int EPI, int C, int T>
__global__ void __launch_bounds__(256) k_sellr(SpmvArgs a) {
    using AT = XT;
    constexpr int BB = BR * BC;
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int row = (int)(gid / T), h = (int)(gid % T);
    const int sl = row / C, t = row % C;
    if (T == 1 && sl >= a.nslice) return;
    const bool live = sl < a.nslice;   // T > 1: whole warps stay for the shuffles
    const long long base = live ? a.sl_ptr[sl] : 0;
    const int w = live ? (int)((a.sl_ptr[sl + 1] - base) / C) : 0;
    const VT *__restrict__ val = (const VT *)a.val;
    const int *__restrict__ ci = a.sl_ci;
    SlotBatch<BB, VT> sb;
    if (h < w) slot_load<BB, C>(sb, val, ci, base, t, h);
    pdl_wait();
    const XT *x = (const XT *)a.x + col_off(a, a.x_ld);
    AT acc[BR];
#pragma unroll
    for (int r = 0; r < BR; ++r) acc[r] = 0;
    auto add = [&](const SlotBatch<BB, VT> &s) {
        AT xs[BC];
#pragma unroll
        for (int cc = 0; cc < BC; ++cc) xs[cc] = x[(long long)BC * s.c + cc];
#pragma unroll
        for (int r = 0; r < BR; ++r) {
            AT u = 0;
#pragma unroll
            for (int cc = 0; cc < BC; ++cc) u += cvt<AT>(s.m[r * BC + cc]) * xs[cc];
            acc[r] += u;
        }
    };
    if (h < w) add(sb);
#pragma unroll 2
    for (int k = h + T; k < w; k += T) {
        SlotBatch<BB, VT> u;
        slot_load<BB, C>(u, val, ci, base, t, k);
        add(u);
    }
#pragma unroll
    for (int o = T / 2; o > 0; o >>= 1)
#pragma unroll
        for (int r = 0; r < BR; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
    if (row >= a.nbr || h != 0) return;
    XT *y = (XT *)a.y;
#pragma unroll
    for (int r = 0; r < BR; ++r) {
        const long long idx = (long long)row * BR + r;
        if (EPI == EPI_SET) y[idx] = acc[r];
        else if (EPI == EPI_ADD) y[idx] += acc[r];
        else y[idx] -= acc[r];
    }
}

// Sliced-ELL product with T threads per block row (T = 2, 4, 8: thread h
// takes slots h, h + T, ..., then an xor-shuffle tree over the T lanes), for
// levels whose rows are few, so that one thread per row leaves the SMs with
// little memory parallelism.  V > T: T threads in the sums of V, the same bits
// (see sell_chains, which is the form for one thread and BF16 values).
constexpr int kSellMT = 1000;   // DMat::tuned code kSellMT + T selects this kernel with T threads per row
__host__ __device__ inline bool is_sellm(int g) { return g == kSellMT + 2 || g == kSellMT + 4 || g == kSellMT + 8; }
template <int BS, typename VT, typename XT, int EPI, int C, int T, bool LR = false, int K = C == 32 ? 2 : 1, int V = T>
__global__ void __launch_bounds__(256) k_sellm(SpmvArgs a) {
    using AT = XT;
    constexpr int BB = BS * BS;
    const int bx = LR && a.lr_rev == 1 ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    const long long gid = (long long)bx * blockDim.x + threadIdx.x;
    const int row = (int)(gid / T), h = (int)(gid % T);
    const int sl = row / C, t = row % C;
    const bool live = sl < a.nslice;
    // everything that the solve does not write first (see pdl_wait): the slice,
    // the first slots, the block-diagonal inverse, the row's aggregate
    const bool own = h == 0 && live && row < a.nbr;
    const long long base = live ? a.sl_ptr[sl] : 0;
    const int w = live ? (int)((a.sl_ptr[sl + 1] - base) / C) : 0;
    const VT *__restrict__ val = (const VT *)a.val;
    const int *__restrict__ ci = a.sl_ci;
    constexpr bool PAIRED = std::is_same<VT, __nv_bfloat16>::value;
    PairBatch<BS, C, K> pb;
    SlotBatch<BB, VT> sb;
    if constexpr (PAIRED) sell_pairs_load(pb, a, base / 2, w / 2, t, h, T);   // the T threads take alternate pairs
    else if (h < w) slot_load<BB, C>(sb, val, ci, base, t, h);
    AT edi[BB];
    int agg = -1;
    if (own && (EPI == EPI_CHEB || EPI == EPI_POST)) {
        const XT *dv = (const XT *)a.dinv + (long long)row * BB;
#pragma unroll
        for (int q = 0; q < BB; ++q) edi[q] = dv[q];
        if (EPI == EPI_POST) agg = a.agg[row];
    }
    const int lr0 = LR && own ? a.lr_rp[row] : 0, lr1 = LR && own ? a.lr_rp[row + 1] : 0;
    pdl_wait();
    // the row's own epilogue operands are loaded before the slot loop, so that
    // their latency overlaps the gather chain (these small levels are
    // latency-bound: fewer rows than the GPU has threads in flight)
    const XT *x = (const XT *)a.x + col_off(a, a.x_ld);
    AT eb[3] = {0, 0, 0}, ed[3] = {0, 0, 0}, ex[3] = {0, 0, 0};
    if (own && (EPI == EPI_RES || EPI == EPI_CHEB || EPI == EPI_POST)) {
#pragma unroll
        for (int q = 0; q < BS; ++q) eb[q] = ((const XT *)a.b + col_off(a, a.b_ld))[(long long)row * BS + q];
    }
    if (own && EPI == EPI_CHEB) {
#pragma unroll
        for (int q = 0; q < BS; ++q) {
            if (a.d_read) ed[q] = ((const XT *)a.d)[(long long)row * BS + q];
            ex[q] = x[(long long)row * BS + q];
        }
    }
    if (own && EPI == EPI_POST) {
#pragma unroll
        for (int q = 0; q < BS; ++q) {
            ex[q] = ((const XT *)a.xin)[(long long)row * BS + q];
            if (agg >= 0) ex[q] += x[(long long)agg * BS + q];
        }
    }
    AT acc0 = 0, acc1 = 0, acc2 = 0;
    if constexpr (V > T) {
        // this thread's chains h, h + T, ... of V, added as the V lanes' tree adds them
        constexpr int Q = V / T;
        const int np = PAIRED ? w / 2 : w;
        AT s0[Q] = {}, s1[Q] = {}, s2[Q] = {};
        if constexpr (PAIRED) {
            for (int p = h; p < np; p += V) {
#pragma unroll
                for (int q = 0; q < Q; q += K) {
                    if (p + q * T >= np) break;
                    if (p + q * T != h) sell_pairs_load(pb, a, base / 2, np, t, p + q * T, T);
#pragma unroll
                    for (int u = 0; u < K; ++u)
                        if (p + (q + u) * T < np) pair_fma<BS>(pb.c[u], pb.m[u], x, s0[q + u], s1[q + u], s2[q + u]);
                }
            }
            if ((w & 1) && np % T == h) {
                const int last = np % V / T;
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if (q == last) sell_single<BS, C>(a, base + (long long)C * (w - 1), t, x, s0[q], s1[q], s2[q]);
            }
        } else {
            for (int k = h; k < w; k += V) {
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    if (k + q * T >= w) break;
                    if (k + q * T != h) slot_load<BB, C>(sb, val, ci, base, t, k + q * T);
                    slot_fma<BS, VT, AT>(sb, x, s0[q], s1[q], s2[q]);
                }
            }
        }
#pragma unroll
        for (int o = Q / 2; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < o; ++q) {
                s0[q] += s0[q + o];
                s1[q] += s1[q + o];
                s2[q] += s2[q + o];
            }
        acc0 = s0[0];
        acc1 = s1[0];
        acc2 = s2[0];
    } else if constexpr (PAIRED) {
        sell_pairs(pb, a, base / 2, w / 2, t, h, T, x, acc0, acc1, acc2);
        // an odd width's last slot goes to the thread whose turn comes next
        if ((w & 1) && h == (w / 2) % T) sell_single<BS, C>(a, base + (long long)C * (w - 1), t, x, acc0, acc1, acc2);
    } else {
        if (h < w) slot_fma<BS, VT, AT>(sb, x, acc0, acc1, acc2);
        for (int k = h + T; k < w; k += T) {
            SlotBatch<BB, VT> u;
            slot_load<BB, C>(u, val, ci, base, t, k);
            slot_fma<BS, VT, AT>(u, x, acc0, acc1, acc2);
        }
    }
#pragma unroll
    for (int o = T / 2; o > 0; o >>= 1) {
        acc0 += __shfl_xor_sync(0xffffffffu, acc0, o);
        if (BS > 1) {
            acc1 += __shfl_xor_sync(0xffffffffu, acc1, o);
            acc2 += __shfl_xor_sync(0xffffffffu, acc2, o);
        }
    }
    __shared__ double fs[kLrInline];
    int k0 = 0;
    if (LR && a.lr_rev >= 0) k0 = lr_factors(a, bx * (256 / T), (bx + 1) * (256 / T), x, fs);
    if (!own) return;
    const AT accs[3] = {acc0, acc1, acc2};
    XT *y = (XT *)a.y;
    if (EPI == EPI_CHEB || EPI == EPI_POST) {
        XT *d = (XT *)a.d;
        XT *xo = (XT *)a.xout + col_off(a, a.out_ld);
        const AT c1 = sizeof(AT) == 4 ? (AT)a.c1f : (AT)a.c1, c2 = sizeof(AT) == 4 ? (AT)a.c2f : (AT)a.c2;
        AT r[3];
#pragma unroll
        for (int q = 0; q < BS; ++q) r[q] = eb[q] - accs[q];
#pragma unroll
        for (int q = 0; q < BS; ++q) {
            AT tq = 0;
#pragma unroll
            for (int c = 0; c < BS; ++c) tq += edi[q * BS + c] * r[c];
            const long long idx = (long long)row * BS + q;
            const AT dn = (EPI == EPI_CHEB && a.d_read ? c1 * ed[q] : AT(0)) + c2 * tq;
            if (a.d_write) d[idx] = dn;
            xo[idx] = ex[q] + dn;
        }
        return;
    }
#pragma unroll
    for (int q = 0; q < BS; ++q) {
        const long long idx = (long long)row * BS + q;
        if (EPI == EPI_SET) {
            AT s = accs[q];
            // the rank-one term in FP64, on the rows that carry its entries (see k_sell)
            if (LR && lr1 > lr0) s = (AT)((double)s + lr_term(a, lr0, lr1, q, fs, k0));
            y[idx] = s;
        }
        else if (EPI == EPI_ADD) y[idx] += accs[q];
        else if (EPI == EPI_SUB) y[idx] -= accs[q];
        else y[idx] = eb[q] - accs[q];
    }
}

// ============================================ deterministic reductions
// The Arnoldi kernels run on a fixed grid of kReduceBlocks blocks; block b
// covers one fixed contiguous chunk of the vectors (a multiple of the 16-byte
// vector width), writes its partial sums to partial[col][b], and the last
// block to finish (atomic ticket) adds the partials of every column in a
// fixed order.  Results therefore do not depend on block scheduling.

// 16-byte vectors of T (float4 / double2)
template <typename T> struct Vec16;
template <> struct Vec16<float> { static constexpr int W = 4; using type = float4; };
template <> struct Vec16<double> { static constexpr int W = 2; using type = double2; };

template <typename T> __device__ __forceinline__ void vld(const T *p, T (&o)[Vec16<T>::W]) {
    const typename Vec16<T>::type u = *reinterpret_cast<const typename Vec16<T>::type *>(p);
    memcpy(o, &u, 16);
}
template <typename T> __device__ __forceinline__ void vst(T *p, const T (&o)[Vec16<T>::W]) {
    typename Vec16<T>::type u;
    memcpy(&u, o, 16);
    *reinterpret_cast<typename Vec16<T>::type *>(p) = u;
}

// This block's chunk [lo, hi) of 0..n-1; lo is a multiple of W.
__device__ __forceinline__ void block_chunk(long long n, int W, long long &lo, long long &hi) {
    const long long per = ((n + gridDim.x - 1) / gridDim.x + W - 1) / W * W;
    lo = min(n, (long long)blockIdx.x * per);
    hi = min(n, lo + per);
}

// True in the last block of the grid to get here (after every block has
// published its partials).  The last block resets the ticket before it ends.
__device__ __forceinline__ bool grid_last_block(unsigned *ticket) {
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
    __syncthreads();
    return s_last != 0;
}

// out[col] = sum_b partial[col][b] for col < ncols, run by one whole block:
// thread t adds partials b = t, t + blockDim, ... of up to 8 columns at a time
// (all loads independent), then a warp tree and a fixed sum over the warps --
// one order whatever the scheduling.
// The FP32 kernels' partials are float-float pairs (float2 in the double
// slots); those go through block_reduce_partials_ff.
__device__ __forceinline__ void block_reduce_partials(const double *partial, int nb, int ncols, double *out) {
    __shared__ double red[8][32];
    const int warp = threadIdx.x >> 5, ln = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int c0 = 0; c0 < ncols; c0 += 8) {
        double acc[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] = 0.0;
#pragma unroll 4
        for (int b = threadIdx.x; b < nb; b += blockDim.x) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (c0 + q < ncols) acc[q] += __ldcg(partial + (long long)(c0 + q) * nb + b);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const double v = warp_sum(acc[q]);
            if (ln == 0) red[q][warp] = v;
        }
        __syncthreads();
        if ((int)threadIdx.x < 8 && c0 + (int)threadIdx.x < ncols) {
            double u = 0.0;
            for (int w = 0; w < nw; ++w) u += red[threadIdx.x][w];
            out[c0 + threadIdx.x] = u;
        }
        __syncthreads();
    }
}

// out[col] = sum_b of the float-float partials of column col.  With 4, 2
// or 1 warps per column (few columns leave warps over), warp part p of a
// column adds partials b = lane + 32 p, ... in ascending order, eight loads in
// flight, then a fixed warp tree and the parts in order (one order whatever
// the scheduling).  All threads of a 256-thread block.
__device__ __forceinline__ void block_reduce_partials_ff(const double *partial, int nb, int ncols, double *out) {
    __shared__ FF red[8];
    const int warp = threadIdx.x >> 5, ln = threadIdx.x & 31;
    const int wpc = ncols <= 2 ? 4 : ncols <= 4 ? 2 : 1, step = 32 * wpc;
    for (int col = warp / wpc; col < ncols; col += 8 / wpc) {
        const float2 *p = reinterpret_cast<const float2 *>(partial + (long long)col * nb);
        FF a{0.f, 0.f};
        for (int b0 = ln + 32 * (warp % wpc); b0 < nb; b0 += 8 * step) {
            float2 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = b0 + u * step < nb ? __ldcg(p + b0 + u * step) : make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 8; ++u) a = ff_add(a, FF{v[u].x, v[u].y});
        }
        a = ff_warp_sum(a);
        if (ln == 0) {
            if (wpc == 1) out[col] = ff_to_double(a);
            else red[warp] = a;
        }
    }
    if (wpc > 1) {   // uniform over the block; one column per group of warps then
        __syncthreads();
        if ((int)threadIdx.x < ncols) {
            FF u = red[threadIdx.x * wpc];
            for (int q = 1; q < wpc; ++q) u = ff_add(u, red[threadIdx.x * wpc + q]);
            out[threadIdx.x] = ff_to_double(u);
        }
    }
}
// the last block's reduction of a T kernel's partials
template <typename T> __device__ __forceinline__ void reduce_partials(const double *partial, int nb, int ncols, double *out) {
    if constexpr (std::is_same<T, float>::value) block_reduce_partials_ff(partial, nb, ncols, out);
    else block_reduce_partials(partial, nb, ncols, out);
}

// Warp sums of NQ values (a power of two up to 16) at once by folding: in
// each of the first log2 NQ xor steps a lane keeps half of its values and
// sends the other half, so NQ - 1 adds replace the NQ per step of NQ separate
// trees (8 values: 9 adds a lane instead of 40).  On return every lane of
// group g = lane / (32 / NQ) holds the sum of value g.
template <typename V, int NQ, typename Add, typename Xor>
__device__ __forceinline__ V fold_warp(V (&v)[NQ], int ln, Add add, Xor xr) {
    int o = 16;
#pragma unroll
    for (int h = NQ / 2; h > 0; h >>= 1, o >>= 1) {
        const bool up = (ln & o) != 0;
#pragma unroll
        for (int q = 0; q < h; ++q) {
            const V keep = up ? v[q + h] : v[q], send = up ? v[q] : v[q + h];
            v[q] = add(keep, xr(send, o));
        }
    }
    V r = v[0];
    for (; o > 0; o >>= 1) r = add(r, xr(r, o));
    return r;
}

// Block stage of the grid reductions: for q < nq, the sum of acc[q] over the
// block's threads into partial[(col0 + q) * gridDim.x + blockIdx.x].  FP64
// kernels: FP64 warp trees, then the warps' sums in order; FP32 kernels: the
// same in float-float (the partial stored as a float2).  256 threads; columns
// in folded groups of up to 8 (fold_warp).  FP32 kernels give the thread's
// sums as floats or as float-float pairs.
__device__ __forceinline__ FF as_ff(float v) { return FF{v, 0.f}; }
__device__ __forceinline__ FF as_ff(FF v) { return v; }
template <typename T, int NQ, typename A>
__device__ __forceinline__ void block_partials(const A (&acc)[NQ], int nq, double *partial, int col0) {
    const int warp = threadIdx.x >> 5, ln = threadIdx.x & 31, nw = blockDim.x >> 5;
    constexpr int F = NQ < 8 ? NQ : 8;   // values folded together
    static_assert(NQ % F == 0 && (F & (F - 1)) == 0, "fold size");
    const int q_of = ln / (32 / F);      // fold_warp's value of this lane (its bits, top first)
    const bool lead = ln % (32 / F) == 0;
    if constexpr (std::is_same<T, float>::value) {
        __shared__ FF redf[NQ][8];
        auto add = [](FF a, FF b) { return ff_add(a, b); };
        auto xr = [](FF a, int o) {
            return FF{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
        };
#pragma unroll
        for (int q0 = 0; q0 < NQ; q0 += F)
            if (q0 < nq) {   // uniform over the block
                if (nq - q0 == 1) {   // one column left: a plain warp sum
                    const FF v = ff_warp_sum(as_ff(acc[q0]));
                    if (ln == 0) redf[q0][warp] = v;
                } else {
                    FF v[F];
#pragma unroll
                    for (int q = 0; q < F; ++q) v[q] = as_ff(acc[q0 + q]);
                    const FF r = fold_warp<FF, F>(v, ln, add, xr);
                    if (lead) redf[q0 + q_of][warp] = r;
                }
            }
        __syncthreads();
        if ((int)threadIdx.x < nq) {
            FF u = redf[threadIdx.x][0];
            for (int k = 1; k < nw; ++k) u = ff_add(u, redf[threadIdx.x][k]);
            *reinterpret_cast<float2 *>(partial + (long long)(col0 + threadIdx.x) * gridDim.x + blockIdx.x) =
                make_float2(u.hi, u.lo);
        }
    } else {
        __shared__ double redd[NQ][8];
        auto add = [](double a, double b) { return a + b; };
        auto xr = [](double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); };
#pragma unroll
        for (int q0 = 0; q0 < NQ; q0 += F)
            if (q0 < nq) {
                if (nq - q0 == 1) {
                    const double v = warp_sum((double)acc[q0]);
                    if (ln == 0) redd[q0][warp] = v;
                } else {
                    double v[F];
#pragma unroll
                    for (int q = 0; q < F; ++q) v[q] = (double)acc[q0 + q];
                    const double r = fold_warp<double, F>(v, ln, add, xr);
                    if (lead) redd[q0 + q_of][warp] = r;
                }
            }
        __syncthreads();
        if ((int)threadIdx.x < nq) {
            double u = 0.0;
            for (int k = 0; k < nw; ++k) u += redd[threadIdx.x][k];
            partial[(long long)(col0 + threadIdx.x) * gridDim.x + blockIdx.x] = u;
        }
    }
}

// The inner products of one step of a K-cycle (x = a1 z1 + a2 (z2 - beta z1),
// w1 = M z1, w2 = M z2, r the residual after the first step) by the launch that
// makes w1 or w2.  First step: w1.w1 and w1.b.  Second step, the direction
// made orthogonal to the first: beta = (w2.w1)/(w1.w1), w2' = w2 - beta w1,
// a2 = (w2'.r)/(w2'.w2').  The products of w2 itself give both,
//   w2'.w2' = w2.w2 - beta w2.w1,   w2'.r = w2.r - beta w1.r,
// without a pass that forms w2' and z2' (2 launches and 10 vector passes fewer
// per K-cycle than updating, reducing and then combining).  Where w2 is close
// to w1 the differences cancel: 3.6e-5 of w2.w2 was left at the least and 0.98
// of it at the median (S_hat levels of four boxes, residuals of 5 cycles).  So
// FP32 sums exact products (two-product) in float-float, and FP64, whose pipe
// is too narrow for more digits, sums over w2' itself where less than a quarter
// is left, in the last block (0 to 6 cycles in a hundred).
// Largest relative error of a2 on those levels: FP32 1e-11 (1.3e-6 with w2'
// formed first and rounded products, 1.7e-4 from rounded products and w1.r
// taken as zero), FP64 1.7e-15 (1.7e-15 and 4e-12).
template <typename T> struct GsSum { using type = double; };
template <> struct GsSum<float> { using type = FF; };
__device__ __forceinline__ FF gs_add(FF a, FF b) { return ff_add(a, b); }
__device__ __forceinline__ double gs_add(double a, double b) { return a + b; }
// a b without rounding (the product and its error by a fused multiply-add)
__device__ __forceinline__ FF gs_mul(float a, float b) {
    const float p = __fmul_rn(a, b);
    return FF{p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ double gs_mul(double a, double b) { return a * b; }
__device__ __forceinline__ void gs_set(FF &s, float v) { s = FF{v, 0.f}; }
__device__ __forceinline__ void gs_set(double &s, double v) { s = v; }

// By the last block of the launch (256 threads), s = {w.w, w.da, w.db, da.db},
// w11 = kd[0] and a1 = kd[2] as loaded beside the partials:
// the first step (da = b): kd[0] = w1.w1, kd[1] = w1.b; the second (da = w1,
// db = r): the cycle's coefficients kd[3] of z1 and kd[4] of z2.  Where nothing
// but rounding is left of w2' the second direction is dropped.
template <typename T>
__device__ __forceinline__ void kc_finish(const double (&s)[4], double w11, double a1, const T *w2, const T *w1, const T *r,
                                          long long n, double *kd) {
    if (!r) {
        if (threadIdx.x == 0) {
            kd[0] = s[0];
            kd[1] = s[1];
        }
        return;
    }
    // by one thread: a warp's FP64 operation holds the pipe for 16 clocks
    double beta = 0.0, ww = 0.0, wr = 0.0;
    if (threadIdx.x == 0) {
        beta = w11 > 0.0 ? s[1] / w11 : 0.0;
        ww = s[0] - beta * s[1];
        wr = s[2] - beta * s[3];
    }
    if constexpr (sizeof(T) == 8) {
        __shared__ double sbeta, red[2][8];
        __shared__ int direct;
        if (threadIdx.x == 0) {
            sbeta = beta;
            direct = ww < 0.25 * s[0];
        }
        __syncthreads();
        if (direct) {
            const double bt = sbeta;
            double p0 = 0.0, p1 = 0.0;
#pragma unroll 4
            for (long long i = threadIdx.x; i < n; i += 256) {
                const double v = __ldcg(w2 + i) - bt * w1[i];   // w2: written by this launch
                p0 += v * v;
                p1 += v * r[i];
            }
            p0 = warp_sum(p0);
            p1 = warp_sum(p1);
            if ((threadIdx.x & 31) == 0) {
                red[0][threadIdx.x >> 5] = p0;
                red[1][threadIdx.x >> 5] = p1;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                ww = wr = 0.0;
                for (int k = 0; k < 8; ++k) {
                    ww += red[0][k];
                    wr += red[1][k];
                }
            }
        }
    }
    if (threadIdx.x == 0) {
        const double a2 = ww <= (sizeof(T) == 4 ? 1e-10 : 1e-20) * s[0] ? 0.0 : wr / ww;   // NaN passes through
        kd[3] = a1 - a2 * beta;
        kd[4] = a2;
    }
}

// Scalar-block (Ŝ level) sliced-ELL product y = M x fused with the inner
// products the K-cycle takes of it (see kc_finish).  T threads per row as in
// k_sellm (T = 1: one thread per row); each row's sum
// is the same as the unfused kernels'.  The row products are summed per block
// (block_partials) into part, and the last block to finish (ticket kd[7])
// adds the block partials in a fixed order -- one launch instead of a product
// and a reduction, the same result whatever the order the blocks run in.
struct DotArgs {
    const void *da, *db;   // vectors the product is dotted with (same type as y); db null in the first step
    double *part;          // 4 x gridDim.x block partials
    double *kd;            // results (kc_finish); kd[7] is the ticket
};
template <typename VT, typename XT, int C, int T>
__global__ void __launch_bounds__(256) k_sell_dot(SpmvArgs a, DotArgs q) {
    using AT = XT;
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int row = (int)(gid / T), h = (int)(gid % T);
    const int sl = row / C, t = row % C;
    const bool live = sl < a.nslice;
    const long long base = live ? a.sl_ptr[sl] : 0;
    const int w = live ? (int)((a.sl_ptr[sl + 1] - base) / C) : 0;
    const VT *__restrict__ val = (const VT *)a.val;
    const XT *x = (const XT *)a.x;
    AT acc0 = 0, acc1 = 0, acc2 = 0;
    if constexpr (std::is_same<VT, __nv_bfloat16>::value) {
        PairBatch<1, C> pb;
        sell_pairs_load(pb, a, base / 2, w / 2, t, h, T);
        pdl_wait();
        sell_pairs(pb, a, base / 2, w / 2, t, h, T, x, acc0, acc1, acc2);
        if ((w & 1) && h == (w / 2) % T) sell_single<1, C>(a, base + (long long)C * (w - 1), t, x, acc0, acc1, acc2);
    } else {
        SlotBatch<1, VT> sb;
        if (h < w) slot_load<1, C>(sb, val, a.sl_ci, base, t, h);
        pdl_wait();
        if (h < w) slot_fma<1, VT, AT>(sb, x, acc0, acc1, acc2);
        for (int k = h + T; k < w; k += T) {
            SlotBatch<1, VT> u;
            slot_load<1, C>(u, val, a.sl_ci, base, t, k);
            slot_fma<1, VT, AT>(u, x, acc0, acc1, acc2);
        }
    }
#pragma unroll
    for (int o = T / 2; o > 0; o >>= 1) acc0 += __shfl_xor_sync(0xffffffffu, acc0, o);
    typename GsSum<AT>::type pp[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) gs_set(pp[k], AT(0));
    const XT *da = (const XT *)q.da, *db = (const XT *)q.db;
    if (h == 0 && live && row < a.nbr) {
        ((XT *)a.y)[row] = acc0;
        const XT u = da[row];
        pp[0] = gs_mul(acc0, acc0);
        pp[1] = gs_mul(acc0, u);
        if (db) {
            const XT v = db[row];
            pp[2] = gs_mul(acc0, v);
            pp[3] = gs_mul(u, v);
        }
    }
    const int nq = db ? 4 : 2;
    block_partials<AT>(pp, nq, q.part, 0);
    unsigned *ticket = (unsigned *)(q.kd + 7);
    if (!grid_last_block(ticket)) return;
    __shared__ double out[4];
    const double w11 = q.kd[0], a1 = q.kd[2];
    reduce_partials<AT>(q.part, gridDim.x, nq, out);
    __syncthreads();
    kc_finish<XT>(out, w11, a1, (const XT *)a.y, da, db, a.nbr, q.kd);
    if (threadIdx.x == 0) *ticket = 0;
}

// ================================================ Givens / least squares
struct GmState {
    double res;      // |g_{j+1}|
    double beta;     // h_{j+1,j}
    double inv;      // 1 / beta (0 where beta is 0): the next basis vector is w inv
    float invf;      // the same, rounded
    int nan;         // NaN/Inf met
};
__device__ __forceinline__ void gm_set_beta(GmState *st, double beta) {
    const double inv = beta == 0.0 ? 0.0 : 1.0 / beta;
    st->beta = beta;
    st->inv = inv;
    st->invf = (float)inv;
}
template <typename T> __device__ __forceinline__ T gm_inv(const GmState *st) {
    if constexpr (std::is_same<T, float>::value) return st->invf;
    else return st->inv;
}

// Loop state of one device-driven GMRES level (graph WHILE nodes).
struct GmDev {
    int j, its, m, nmax;        // column of the current cycle, iterations, restart length, iteration limit
    int conv, nan, pad0, pad1;  // pad0: restart cycles run (outer level)
    double tol, bnorm, res, rel_true;
};

// What the fused Givens update of Hessenberg column j needs (H == nullptr:
// no update).
struct GivensArgs {
    double *H = nullptr;
    int ldh = 0, j = 0;
    const double *h1 = nullptr, *h2 = nullptr;
    double *cs = nullptr, *sn = nullptr, *g = nullptr;
    GmState *st = nullptr;
    // device-driven loops: the column index is dl->j, and the update also ends
    // the iteration (givens_step): it advances dl and sets the WHILE condition
    GmDev *dl = nullptr;
    cudaGraphConditionalHandle h = 0;
};

// Operands of the Givens update staged in shared memory by the block that
// applies it (before it reduces the norm's partials, so that these loads and
// the partials' are in flight together): as a chain of dependent global loads
// in one thread they cost most of the norm pass's tail.  Bases longer than
// kGivensCols read global memory instead.
constexpr int kGivensCols = 64;
struct GivensBuf {
    double h[kGivensCols], cs[kGivensCols], sn[kGivensCols];
    double g, a;   // a: H(j, j) after the previous rotations (j < kGivensCols)
    GmDev dl;
    int j;
};
// by one warp, which also applies the previous rotations to the column: they
// do not wait for the norm
__device__ __forceinline__ void givens_stage(const GivensArgs &q, GivensBuf &B) {
    const int ln = threadIdx.x & 31, j = q.dl ? q.dl->j : q.j;
    if (ln == 0) {
        B.j = j;
        B.g = q.g[j];
        if (q.dl) B.dl = *q.dl;
    }
    if (j >= kGivensCols) return;
    for (int i = ln; i <= j; i += 32) {
        B.h[i] = q.h2 ? q.h1[i] + q.h2[i] : q.h1[i];
        if (i < j) { B.cs[i] = q.cs[i]; B.sn[i] = q.sn[i]; }
    }
    __syncwarp();
    if (ln != 0) return;
    double a = B.h[0];
    for (int i = 0; i < j; ++i) {
        const double b = B.h[i + 1], c = B.cs[i], s = B.sn[i];
        q.H[(long long)i * q.ldh + j] = c * a + s * b;
        a = -s * a + c * b;
    }
    B.a = a;
}

// Column j of the Hessenberg matrix: H(i,j) = h1_i + h2_i (i <= j; h1_i
// alone when h2 is null, a single Gram-Schmidt pass),
// H(j+1,j) = ||w|| (from ||w||^2 = nrm2); the previous rotations applied, a
// new rotation chosen to zero H(j+1,j), and the right-hand side g rotated
// (Saad 1993, FGMRES with Givens rotations).  In a device-driven loop then
// the end of the iteration: the stopping rule of the host-driven loop --
// continue while |g_{j+1}| > max(rtol ||b||, atol), h_{j+1,j} != 0, no NaN,
// j < m and its < n_max -- as the WHILE node's condition (every block has
// read j before it took its ticket, so dl may advance here).  One thread.
__device__ __forceinline__ void givens_step(const GivensArgs &q, const GivensBuf &B, double nrm2) {
    double *H = q.H;
    const long long ldh = q.ldh;
    const int j = B.j;
    double a;   // H(j, j) after the previous rotations
    if (j < kGivensCols) {
        a = B.a;
    } else {
        for (int i = 0; i <= j; ++i) H[i * ldh + j] = q.h2 ? q.h1[i] + q.h2[i] : q.h1[i];
        for (int i = 0; i < j; ++i) {
            const double u = H[i * ldh + j], b = H[(i + 1) * ldh + j];
            H[i * ldh + j] = q.cs[i] * u + q.sn[i] * b;
            H[(i + 1) * ldh + j] = -q.sn[i] * u + q.cs[i] * b;
        }
        a = H[j * ldh + j];
    }
    // Away from under- and overflow from two independent reciprocal square
    // roots: the square root, hypot and three divisions one after another took
    // about 2 us of the pass (an FP64 operation waits tens of clocks here).
    double beta, inv, den, c = 1.0, s = 0.0;
    const double sq = a * a + nrm2;
    if (nrm2 > 1e-280 && sq < 1e280) {
        inv = rsqrt(nrm2);
        const double r = rsqrt(sq);
        beta = nrm2 * inv;
        den = sq * r;
        c = a * r;
        s = beta * r;
    } else {
        beta = (nrm2 >= 0.0) ? sqrt(nrm2) : nrm2;   // NaN passes through
        inv = beta == 0.0 ? 0.0 : 1.0 / beta;
        den = hypot(a, beta);
        if (den != 0.0) { c = a / den; s = beta / den; }
    }
    q.cs[j] = c;
    q.sn[j] = s;
    H[j * ldh + j] = den;
    H[(j + 1) * ldh + j] = 0.0;
    const double g1 = -s * B.g;
    q.g[j + 1] = g1;
    q.g[j] = c * B.g;
    const double res = fabs(g1);
    const int nan = (isfinite(res) && isfinite(beta)) ? 0 : 1;
    q.st->res = res;
    q.st->nan = nan;
    q.st->beta = beta;
    q.st->inv = inv;
    q.st->invf = (float)inv;
    if (q.dl) {
        const int its = B.dl.its + 1, nan_any = B.dl.nan | nan;
        q.dl->its = its;
        q.dl->j = j + 1;
        q.dl->res = res;
        q.dl->nan = nan_any;
        const bool go = !nan_any && res > B.dl.tol && beta != 0.0 && j + 1 < B.dl.m && its < B.dl.nmax;
        cudaGraphSetConditional(q.h, go ? 1u : 0u);
    }
}

// The last block's end of a reduction kernel: the partials of ncols columns
// into out, then (gv.H set) the Givens update with out[0] = ||w||^2.
template <typename T>
__device__ __forceinline__ void finish_reduction(const double *partial, int ncols, double *out, unsigned *ticket,
                                                 const GivensArgs &gv) {
    __shared__ GivensBuf B;
    if (gv.H && threadIdx.x >> 5 == 7) givens_stage(gv, B);   // a warp that a norm's reduction leaves idle
    reduce_partials<T>(partial, gridDim.x, ncols, out);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (gv.H) givens_step(gv, B, out[0]);
        *ticket = 0;
    }
}

// out[c] = V(:, c)^T w for c < ncols (column c at V + c*ldv), over the fixed
// grid; VEC: every pointer and ldv are 16-byte aligned.  When gv.H is set
// (ncols == 1, w the new Arnoldi vector) the last block also applies the
// Givens update with out[0] = ||w||^2.
template <typename T, int CB, bool VEC>
__device__ __forceinline__ void mdot_body(const T *V, long long ldv, int ncols, const T *w,
                                          long long n, double *partial, double *out,
                                          unsigned *ticket, const GivensArgs &gv) {
    constexpr int W = VEC ? Vec16<T>::W : 1;
    long long lo, hi;
    block_chunk(n, Vec16<T>::W, lo, hi);
    const long long nv = (hi - lo) / W;
    for (int c0 = 0; c0 < ncols; c0 += CB) {
        T acc[CB];
#pragma unroll
        for (int q = 0; q < CB; ++q) acc[q] = 0;
        for (long long i = threadIdx.x; i < nv; i += blockDim.x) {
            const long long t = lo + i * W;
            if constexpr (VEC) {
                T wt[W];
                vld(w + t, wt);
#pragma unroll
                for (int q = 0; q < CB; ++q)
                    if (c0 + q < ncols) {
                        T v[W];
                        vld(V + (long long)(c0 + q) * ldv + t, v);
#pragma unroll
                        for (int e = 0; e < W; ++e) acc[q] += v[e] * wt[e];
                    }
            } else {
                const T wt = w[t];
#pragma unroll
                for (int q = 0; q < CB; ++q)
                    if (c0 + q < ncols) acc[q] += V[(long long)(c0 + q) * ldv + t] * wt;
            }
        }
        if (VEC && threadIdx.x < hi - lo - nv * W) {   // ragged end of the last chunk
            const long long t = lo + nv * W + threadIdx.x;
            const T wt = w[t];
#pragma unroll
            for (int q = 0; q < CB; ++q)
                if (c0 + q < ncols) acc[q] += V[(long long)(c0 + q) * ldv + t] * wt;
        }
        block_partials<T, CB>(acc, min(CB, ncols - c0), partial, c0);
        __syncthreads();
    }
    if (!grid_last_block(ticket)) return;
    finish_reduction<T>(partial, ncols, out, ticket, gv);
}

template <typename T, int CB, bool VEC>
__global__ void __launch_bounds__(256) k_mdot(const T *V, long long ldv, int ncols, const T *w,
                                              long long n, double *partial, double *out,
                                              unsigned *ticket, GivensArgs gv) {
    mdot_body<T, CB, VEC>(V, ldv, ncols, w, n, partial, out, ticket, gv);
}
// the same with ncols = *jp + off read on the device (device-driven loops)
template <typename T, int CB, bool VEC>
__global__ void __launch_bounds__(256) k_mdot_dl(const T *V, long long ldv, const int *jp, int off,
                                                 const T *w, long long n, double *partial,
                                                 double *out, unsigned *ticket, GivensArgs gv) {
    pdl_wait();
    mdot_body<T, CB, VEC>(V, ldv, *jp + off, w, n, partial, out, ticket, gv);
}

// w[t] += alpha * sum_j coef[j] V[j][t]  (coef on the device, FP64)
// (set: w = alpha * the sum instead)
template <typename T, bool VEC, bool SET = false>
__device__ __forceinline__ void maxpy_body(const T *V, long long ldv, int ncols, const double *coef, double alpha, T *w,
                                           long long n) {
    constexpr int W = VEC ? Vec16<T>::W : 1;
    __shared__ T cs[256];
    const long long nv = n / W;
    for (int c0 = 0; c0 < ncols || (SET && c0 == 0); c0 += 256) {
        const int cn = min(256, ncols - c0);
        __syncthreads();
        if ((int)threadIdx.x < cn) cs[threadIdx.x] = (T)(alpha * coef[c0 + threadIdx.x]);
        __syncthreads();
        for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (long long)gridDim.x * blockDim.x) {
            const long long t = i * W;
            T acc[W];
            if (SET && c0 == 0) {
#pragma unroll
                for (int e = 0; e < W; ++e) acc[e] = T(0);
            } else {
                if constexpr (VEC) vld(w + t, acc);
                else acc[0] = w[t];
            }
#pragma unroll 4
            for (int j = 0; j < cn; ++j) {
                T v[W];
                if constexpr (VEC) vld(V + (long long)(c0 + j) * ldv + t, v);
                else v[0] = V[(long long)(c0 + j) * ldv + t];
#pragma unroll
                for (int e = 0; e < W; ++e) acc[e] += cs[j] * v[e];
            }
            if constexpr (VEC) vst(w + t, acc);
            else w[t] = acc[0];
        }
        if (VEC && blockIdx.x == 0 && threadIdx.x < n - nv * W) {   // ragged end
            const long long t = nv * W + threadIdx.x;
            T acc = SET && c0 == 0 ? T(0) : w[t];
            for (int j = 0; j < cn; ++j) acc += cs[j] * V[(long long)(c0 + j) * ldv + t];
            w[t] = acc;
        }
    }
}

template <typename T, bool VEC>
__global__ void __launch_bounds__(256) k_maxpy(const T *V, long long ldv, int ncols, const double *coef, double alpha, T *w,
                                               long long n) {
    maxpy_body<T, VEC>(V, ldv, ncols, coef, alpha, w, n);
}
// w = sum_j coef[j] V[j] (set) or w += it, *jp columns
template <typename T, bool VEC, bool SET>
__global__ void __launch_bounds__(256) k_maxpy_dl(const T *V, long long ldv, const int *jp, const double *coef, T *w,
                                                  long long n) {
    pdl_wait();
    maxpy_body<T, VEC, SET>(V, ldv, *jp, coef, 1.0, w, n);
}

// Fused CGS pass for up to MAXC columns: w_new = w - sum_j coef[j] V[j], then
// the dots of the same columns with w_new (norm_only = 0) or the squared norm
// of w_new (norm_only = 1), V read once; partials reduced by the last block
// into out (and, with gv.H set, the Givens update with out[0] = ||w_new||^2).
template <typename T, int MAXC, bool VEC>
__device__ __forceinline__ void maxpy_dot_body(const T *V, long long ldv, int ncols,
                                               const double *coef, T *w, long long n,
                                               int norm_only, double *partial, double *out,
                                               unsigned *ticket, const GivensArgs &gv) {
    constexpr int W = VEC ? Vec16<T>::W : 1;
    __shared__ T cs[MAXC];
    if ((int)threadIdx.x < ncols) cs[threadIdx.x] = (T)coef[threadIdx.x];
    __syncthreads();
    long long lo, hi;
    block_chunk(n, Vec16<T>::W, lo, hi);
    const long long nv = (hi - lo) / W;
    T acc[MAXC];
#pragma unroll
    for (int q = 0; q < MAXC; ++q) acc[q] = 0;
    auto body = [&](long long t, auto wtag) {
        constexpr int L = decltype(wtag)::value;
        T v[MAXC][L], s[L];
        if constexpr (L > 1) vld(w + t, s);
        else s[0] = w[t];
#pragma unroll
        for (int q = 0; q < MAXC; ++q)
            if (q < ncols) {
                if constexpr (L > 1) vld(V + (long long)q * ldv + t, v[q]);
                else v[q][0] = V[(long long)q * ldv + t];
#pragma unroll
                for (int e = 0; e < L; ++e) s[e] -= cs[q] * v[q][e];
            }
        if constexpr (L > 1) vst(w + t, s);
        else w[t] = s[0];
        if (norm_only) {
#pragma unroll
            for (int e = 0; e < L; ++e) acc[0] += s[e] * s[e];
        } else {
#pragma unroll
            for (int q = 0; q < MAXC; ++q)
                if (q < ncols) {
#pragma unroll
                    for (int e = 0; e < L; ++e) acc[q] += v[q][e] * s[e];
                }
        }
    };
    for (long long i = threadIdx.x; i < nv; i += blockDim.x) body(lo + i * W, std::integral_constant<int, W>());
    if (VEC && threadIdx.x < hi - lo - nv * W) body(lo + nv * W + threadIdx.x, std::integral_constant<int, 1>());
    const int nout = norm_only ? 1 : ncols;
    block_partials<T, MAXC>(acc, nout, partial, 0);
    if (!grid_last_block(ticket)) return;
    finish_reduction<T>(partial, nout, out, ticket, gv);
}

template <typename T, int MAXC, bool VEC>
__global__ void __launch_bounds__(256) k_maxpy_dot(const T *V, long long ldv, int ncols,
                                                   const double *coef, T *w, long long n,
                                                   int norm_only, double *partial, double *out,
                                                   unsigned *ticket, GivensArgs gv) {
    maxpy_dot_body<T, MAXC, VEC>(V, ldv, ncols, coef, w, n, norm_only, partial, out, ticket, gv);
}

// The device-driven form of the fused pass with products, ncols = *jp + off
// read on the device.  A basis longer than MAXC takes two sweeps over the
// block's own chunk: the subtraction w -= V coef (columns in ascending order,
// each thread on the elements it owns), then mdot_body's products on the same
// elements, so no element crosses threads.
template <typename T, int MAXC, bool VEC>
__global__ void __launch_bounds__(256) k_maxpy_dot_dl(const T *V, long long ldv, const int *jp, int off,
                                                      const double *coef, T *w, long long n,
                                                      double *partial,
                                                      double *out, unsigned *ticket) {
    pdl_wait();
    const int ncols = *jp + off;
    if (ncols <= MAXC) {
        maxpy_dot_body<T, MAXC, VEC>(V, ldv, ncols, coef, w, n, 0, partial, out, ticket, GivensArgs());
        return;
    }
    constexpr int W = VEC ? Vec16<T>::W : 1;
    __shared__ T cs[256];
    long long lo, hi;
    block_chunk(n, Vec16<T>::W, lo, hi);
    const long long nv = (hi - lo) / W;
    for (int c0 = 0; c0 < ncols; c0 += 256) {
        const int cn = min(256, ncols - c0);
        __syncthreads();
        if ((int)threadIdx.x < cn) cs[threadIdx.x] = (T)coef[c0 + threadIdx.x];
        __syncthreads();
        for (long long i = threadIdx.x; i < nv; i += blockDim.x) {
            const long long t = lo + i * W;
            T a[W];
            if constexpr (VEC) vld(w + t, a);
            else a[0] = w[t];
            for (int j = 0; j < cn; ++j) {
                T v[W];
                if constexpr (VEC) vld(V + (long long)(c0 + j) * ldv + t, v);
                else v[0] = V[(long long)(c0 + j) * ldv + t];
#pragma unroll
                for (int e = 0; e < W; ++e) a[e] -= cs[j] * v[e];
            }
            if constexpr (VEC) vst(w + t, a);
            else w[t] = a[0];
        }
        if (VEC && threadIdx.x < hi - lo - nv * W) {   // ragged end, the thread mdot_body gives it
            const long long t = lo + nv * W + threadIdx.x;
            T a = w[t];
            for (int j = 0; j < cn; ++j) a -= cs[j] * V[(long long)(c0 + j) * ldv + t];
            w[t] = a;
        }
    }
    __syncthreads();
    mdot_body<T, 8, VEC>(V, ldv, ncols, w, n, partial, out, ticket, GivensArgs());
}

// The last pass of a device-driven step: w -= V coef (ncols = *jp + 1 columns),
// ||w||^2, and in the last block the Givens update and the end of the
// iteration.  Columns in groups of eight: the products' kernel above keeps
// its 16 columns in registers for the dots, which this pass does not need, and
// two blocks of it fill an SM against five of this.  cap: entries of coef.
template <typename T, bool VEC>
__global__ void __launch_bounds__(256) k_maxpy_norm_dl(const T *V, long long ldv, const int *jp, const double *coef, int cap,
                                                       T *w, long long n, double *partial, double *out, unsigned *ticket,
                                                       GivensArgs gv) {
    pdl_wait();
    constexpr int W = VEC ? Vec16<T>::W : 1;
    __shared__ T cs[256];
    const int tid = threadIdx.x;
    // the first 256 coefficients without waiting for the column count
    const double c0 = tid < cap ? coef[tid] : 0.0;
    const int ncols = *jp + 1;
    cs[tid] = (T)c0;
    __syncthreads();
    long long lo, hi;
    block_chunk(n, Vec16<T>::W, lo, hi);
    const long long nv = (hi - lo) / W;
    T nn[1] = {0};
    auto body = [&](long long t, auto wtag) {
        constexpr int L = decltype(wtag)::value;
        T s[L];
        if constexpr (L > 1) vld(w + t, s);
        else s[0] = w[t];
        for (int q0 = 0; q0 < ncols; q0 += 8) {
            T v[8][L];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q0 + q < ncols) {
                    if constexpr (L > 1) vld(V + (long long)(q0 + q) * ldv + t, v[q]);
                    else v[q][0] = V[(long long)(q0 + q) * ldv + t];
                }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q0 + q < ncols) {
                    const T k = q0 + q < 256 ? cs[q0 + q] : (T)coef[q0 + q];
#pragma unroll
                    for (int e = 0; e < L; ++e) s[e] -= k * v[q][e];
                }
        }
        if constexpr (L > 1) vst(w + t, s);
        else w[t] = s[0];
#pragma unroll
        for (int e = 0; e < L; ++e) nn[0] += s[e] * s[e];
    };
    for (long long i = tid; i < nv; i += blockDim.x) body(lo + i * W, std::integral_constant<int, W>());
    if (VEC && tid < hi - lo - nv * W) body(lo + nv * W + tid, std::integral_constant<int, 1>());
    block_partials<T, 1>(nn, 1, partial, 0);
    if (!grid_last_block(ticket)) return;
    finish_reduction<T>(partial, 1, out, ticket, gv);
}

// ------------------------------------------- Gram-Schmidt in one cluster
// The whole Arnoldi step of a device-driven loop for a short vector -- one or
// two Gram-Schmidt passes, ||w||, the Givens update and the loop's end -- in
// one cluster of kGsCluster blocks that exchange their partial sums through
// distributed shared memory: a pass costs a cluster barrier (about 1 us)
// instead of a launch, a ticket and a last block's reduction.  w stays in
// registers between the passes.  Up to kGsPieces 16-byte pieces per thread:
// 65,536 floats or 32,768 doubles, where eight SMs' share of L2 bandwidth is
// still no slower than the grid's chain; bases of up to kGsCols columns.
// Cube of 8, FP64 (2,187 components): solve 13.4 -> 11.0 ms; cube of 16, FP32: 25.3 -> 24.6 ms.
constexpr int kGsCluster = 8, kGsThreads = 512, kGsPieces = 4, kGsCols = 256, kGsRound = 64;
template <typename T> __host__ __device__ constexpr long long gs_cluster_max() {
    return (long long)kGsCluster * kGsThreads * kGsPieces * Vec16<T>::W;
}
__device__ __forceinline__ FF gs_xor(FF a, int o) {
    return FF{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}
__device__ __forceinline__ double gs_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ double gs_double(FF a) { return ff_to_double(a); }
__device__ __forceinline__ double gs_double(double a) { return a; }
template <typename T>
__global__ void __cluster_dims__(kGsCluster, 1, 1) __launch_bounds__(kGsThreads)
    k_gs_cluster(const T *V, long long ld, const int *jp, T *w, long long n, int passes, double *h1,
                 double *h2, GivensArgs gv) {
    namespace cg = cooperative_groups;
    using S = typename GsSum<T>::type;
    constexpr int W = Vec16<T>::W, P = kGsPieces, NW = kGsThreads / 32;
    __shared__ S red[8][NW + 1];
    __shared__ S part[2][kGsCluster][kGsRound];
    __shared__ S np[kGsCluster];
    __shared__ T coef[kGsCols];
    __shared__ GivensBuf B;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tid = threadIdx.x, warp = tid >> 5, ln = tid & 31;
    // every block of the cluster has to run before another writes its shared
    // memory: arrive here, wait before the first such write
    auto started = cl.barrier_arrive();
    bool waited = false;
    pdl_wait();
    const int ncols = *jp + 1;
    long long at[P];   // first element of each piece
#pragma unroll
    for (int u = 0; u < P; ++u) at[u] = ((long long)(u * kGsCluster + rank) * kGsThreads + tid) * W;
    auto piece = [&](const T *p, long long t, T (&o)[W]) {
        if (t + W <= n) vld(p + t, o);
        else {
#pragma unroll
            for (int e = 0; e < W; ++e) o[e] = t + e < n ? p[t + e] : T(0);
        }
    };
    T wr[P][W];
#pragma unroll
    for (int u = 0; u < P; ++u) piece(w, at[u], wr[u]);
    // one pass: coef = V^T w over the cluster (its own copy in every block; rank 0
    // also to h), then w -= V coef
    int buf = 0;
    auto pass = [&](double *h) {
        for (int base = 0; base < ncols; base += kGsRound, buf ^= 1) {
            const int cnt = min(kGsRound, ncols - base);
            for (int c0 = 0; c0 < cnt; c0 += 8) {
                T acc[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) acc[q] = 0;
#pragma unroll
                for (int u = 0; u < P; ++u) {
                    if (at[u] >= n) continue;
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        if (c0 + q < cnt) {
                            T v[W];
                            piece(V + (long long)(base + c0 + q) * ld, at[u], v);
#pragma unroll
                            for (int e = 0; e < W; ++e) acc[q] += v[e] * wr[u][e];
                        }
                }
                S f[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) gs_set(f[q], acc[q]);
                const S r = fold_warp<S, 8>(f, ln, [](S a, S b) { return gs_add(a, b); },
                                            [](S a, int o) { return gs_xor(a, o); });
                if (ln % 4 == 0) red[ln / 4][warp] = r;
                if (!waited) {   // uniform
                    cl.barrier_wait(std::move(started));
                    waited = true;
                }
                __syncthreads();
                if (tid < 8 * kGsCluster && c0 + tid / kGsCluster < cnt) {   // column, receiving block
                    const int q = tid / kGsCluster;
                    S s = red[q][0];
                    for (int k = 1; k < NW; ++k) s = gs_add(s, red[q][k]);
                    *cl.map_shared_rank(&part[buf][rank][c0 + q], tid % kGsCluster) = s;
                }
                __syncthreads();
            }
            cl.sync();
            if (tid < cnt) {
                S s = part[buf][0][tid];
                for (int r = 1; r < kGsCluster; ++r) s = gs_add(s, part[buf][r][tid]);
                const double d = gs_double(s);
                coef[base + tid] = (T)d;
                if (rank == 0) h[base + tid] = d;
            }
            // part[buf] is written again two rounds on, after the next round's
            // barrier, which every block reaches only past this point
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < P; ++u) {
            if (at[u] >= n) continue;
#pragma unroll 4
            for (int c = 0; c < ncols; ++c) {
                T v[W];
                piece(V + (long long)c * ld, at[u], v);
                const T k = coef[c];
#pragma unroll
                for (int e = 0; e < W; ++e) wr[u][e] -= k * v[e];
            }
        }
        __syncthreads();   // coef is rewritten by the next pass
    };
    pass(h1);
    if (passes > 1) pass(h2);
    T nn = 0;
#pragma unroll
    for (int u = 0; u < P; ++u) {
        if (at[u] + W <= n) vst(w + at[u], wr[u]);
        else {
#pragma unroll
            for (int e = 0; e < W; ++e)
                if (at[u] + e < n) w[at[u] + e] = wr[u][e];
        }
#pragma unroll
        for (int e = 0; e < W; ++e) nn += wr[u][e] * wr[u][e];
    }
    S s;
    gs_set(s, nn);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = gs_add(s, gs_xor(s, o));
    if (ln == 0) red[0][warp] = s;
    __syncthreads();
    if (tid == 0) {
        S t = red[0][0];
        for (int k = 1; k < NW; ++k) t = gs_add(t, red[0][k]);
        *cl.map_shared_rank(&np[rank], 0) = t;
    }
    if (rank == 0 && warp == 1) givens_stage(gv, B);
    cl.sync();
    if (rank != 0 || tid != 0) return;
    S t = np[0];
    for (int r = 1; r < kGsCluster; ++r) t = gs_add(t, np[r]);
    givens_step(gv, B, gs_double(t));
}

// ============================================================== vectors
template <typename T> __global__ void k_fill(T *x, T v, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) x[i] = v;
}
template <typename D, typename S> __global__ void k_convert(D *dst, const S *src, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = (D)src[i];
}
// y = a*x + b*y
template <typename T> __global__ void k_axpby(T *y, const T *x, double a, double b, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = (T)a * x[i] + (T)b * y[i];
}
// z = x - y
template <typename T> __global__ void k_sub(T *z, const T *x, const T *y, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        z[i] = x[i] - y[i];
}
// v = w / s[0] (skips when s[0] == 0); VEC: v, w 16-byte aligned
template <typename T, bool VEC> __device__ __forceinline__ void scale_inv_body(T *v, const T *w, const double *s, long long n) {
    constexpr int W = VEC ? Vec16<T>::W : 1;
    __shared__ T inv_s;
    __shared__ int zero;
    if (threadIdx.x == 0) {   // one FP64 division per block, not per element
        const double d = *s;
        zero = (d == 0.0);
        inv_s = zero ? T(0) : (T)(1.0 / d);
    }
    __syncthreads();
    if (zero) return;
    const T inv = inv_s;
    const long long nv = n / W;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (long long)gridDim.x * blockDim.x) {
        if constexpr (VEC) {
            T u[W];
            vld(w + i * W, u);
#pragma unroll
            for (int e = 0; e < W; ++e) u[e] *= inv;
            vst(v + i * W, u);
        } else {
            v[i] = w[i] * inv;
        }
    }
    if (VEC && blockIdx.x == 0 && threadIdx.x < n - nv * W) v[nv * W + threadIdx.x] = w[nv * W + threadIdx.x] * inv;
}
template <typename T, bool VEC> __global__ void k_scale_inv(T *v, const T *w, const double *s, long long n) {
    scale_inv_body<T, VEC>(v, w, s, n);
}

// v = w / sqrt(*s2) (skips when *s2 is not positive)
__global__ void k_scale_rsqrt(double *v, const double *w, const double *s2, long long n);

// ============================================= least squares (GMRES end)
// y = H(0:k,0:k)^{-1} g(0:k), upper triangular.  One warp.
__global__ void k_trisolve(const double *H, int ldh, const double *g, double *y, int k);
// g = [beta, 0, ...]; st->res = beta
__global__ void k_gm_init(double *g, int m1, const double *beta2, double *beta, GmState *st);

__global__ void k_recip(long long n, const double *a, double *b);

// ============================== device-driven Krylov loops (graph WHILE)
// Per-solve options of the device-driven solve (written before each launch).
struct DlParams {
    double rtol, rtol_A, rtol_S, rtol_I, atol;
    int m, m_A, m_S, nmax, nmax_A, nmax_S;
};
// Iteration counters of one device-driven solve.
struct DlCounters {
    long long A, S, I, nA, nS, nI;
};
__global__ void k_dl_init(GmDev *st, double *g, int m1, const double *nrm2, double *beta, GmState *gs,
                          const double *rtol, const double *atol, const int *m, const int *nmax,
                          cudaGraphConditionalHandle h);
// The start of an inner solve of a device-driven loop in one kernel: ||b||
// and, in the last block, the loop's state (k_dl_init's, which the outer level
// keeps) and the WHILE condition.
struct DlStart {
    GmDev *st;
    double *g, *beta;
    GmState *gs;
    const double *rtol, *atol;
    const int *m, *nmax;
    cudaGraphConditionalHandle h;
};
__device__ __forceinline__ void dl_start(const DlStart &q, double nrm2) {
    const double b = (nrm2 >= 0.0) ? sqrt(nrm2) : nrm2;   // NaN passes through
    q.g[0] = b;
    *q.beta = b;
    q.gs->res = b;
    gm_set_beta(q.gs, b);
    const int nan = isfinite(b) ? 0 : 1, nmax = *q.nmax;
    const double tol = fmax(*q.rtol * b, *q.atol);
    const int conv = (b <= tol) ? 1 : 0;
    q.gs->nan = nan;
    q.st->j = 0;
    q.st->its = 0;
    q.st->pad0 = 0;
    q.st->m = *q.m;
    q.st->nmax = nmax;
    q.st->bnorm = b;
    q.st->res = b;
    q.st->tol = tol;
    q.st->nan = nan;
    q.st->conv = conv;
    q.st->rel_true = b > 0.0 ? 1.0 : 0.0;
    cudaGraphSetConditional(q.h, (!conv && !nan && nmax > 0) ? 1u : 0u);
}
template <typename T, bool VEC>
__global__ void __launch_bounds__(256) k_norm_start(const T *b, long long n, double *partial, double *out, unsigned *ticket,
                                                    DlStart q) {
    pdl_wait();
    constexpr int W = VEC ? Vec16<T>::W : 1;
    long long lo, hi;
    block_chunk(n, Vec16<T>::W, lo, hi);
    const long long nv = (hi - lo) / W;
    T nn[1] = {0};
    for (long long i = threadIdx.x; i < nv; i += blockDim.x) {
        T v[W];
        if constexpr (VEC) vld(b + lo + i * W, v);
        else v[0] = b[lo + i];
#pragma unroll
        for (int e = 0; e < W; ++e) nn[0] += v[e] * v[e];
    }
    if (VEC && threadIdx.x < hi - lo - nv * W) {
        const T v = b[lo + nv * W + threadIdx.x];
        nn[0] += v * v;
    }
    block_partials<T, 1>(nn, 1, partial, 0);
    if (!grid_last_block(ticket)) return;
    reduce_partials<T>(partial, gridDim.x, 1, out);
    __syncthreads();
    if (threadIdx.x == 0) {
        dl_start(q, out[0]);
        *ticket = 0;
    }
}

// The first kernel of a device-driven iteration: basis column j = src / beta
// (beta, and its reciprocal, from the norm pass before), src = w, or b where
// the cycle starts (j = 0).  VEC: pointers and ld 16-byte aligned.
template <typename T, bool VEC>
__global__ void k_start_col(T *vbase, long long ld, const int *jp, const T *b, const T *w, const GmState *gs, long long n) {
    constexpr int W = VEC ? Vec16<T>::W : 1;
    pdl_wait();
    const int j = *jp;
    const T *src = j == 0 ? b : w;
    const T inv = gm_inv<T>(gs);
    T *v = vbase + (long long)j * ld;
    const long long nv = n / W;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (long long)gridDim.x * blockDim.x) {
        if constexpr (VEC) {
            T u[W];
            vld(src + i * W, u);
#pragma unroll
            for (int e = 0; e < W; ++e) u[e] *= inv;
            vst(v + i * W, u);
        } else {
            v[i] = src[i] * inv;
        }
    }
    if (VEC && blockIdx.x == 0 && threadIdx.x < n - nv * W) v[nv * W + threadIdx.x] = src[nv * W + threadIdx.x] * inv;
}
// k_start_col fused with the AMG cycle's first smoothing step from zero on
// that column (k_cheb_first): x = c2 Dinv v, and d = x where a later step of
// the same smoothing reads it (d may be null).  Saves a launch and a pass
// over v per iteration; 0.56M unknowns (421k components): 4.8 + 3.7 -> 4.0 us.
template <typename T>
__global__ void k_start_cheb(int nbr, int bs, const T *__restrict__ dinv, T *vbase, long long ld,
                             const int *jp, const T *b, const T *w, const GmState *gs, T c2, T *d,
                             T *x) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)nbr * bs) return;
    const int i = (int)(t / bs), a = (int)(t - (long long)i * bs);
    T di[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int c = 0; c < 3; ++c)
        if (c < bs) di[c] = dinv[(long long)i * bs * bs + a * bs + c];
    pdl_wait();
    const int j = *jp;
    const T *src = j == 0 ? b : w;
    const T inv = gm_inv<T>(gs);
    vbase[(long long)j * ld + t] = src[t] * inv;
    T s = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c)
        if (c < bs) s += di[c] * (src[(long long)i * bs + c] * inv);
    const T dn = c2 * s;
    if (d) d[t] = dn;
    x[t] = dn;
}
__global__ void k_dl_cycle_start(GmDev *st, cudaGraphConditionalHandle h);
__global__ void k_dl_end(GmDev *st, const double *H, int ldh, const double *g, double *y, long long *its_total,
                         long long *solves);
__global__ void k_dl_restart(GmDev *st, const double *nrm2, double *g, int m1, double *beta, GmState *gs,
                             cudaGraphConditionalHandle h);

// out = entries [from, from + n) of basis column *jp + off (stride ld), converted
template <typename D, typename S>
__global__ void k_col_get(D *out, const S *vbase, long long ld, const int *jp, int off, long long from, long long n) {
    const S *v = vbase + (long long)(*jp + off) * ld + from;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = (D)v[i];
}
// entries [to, to + n) of basis column *jp + off = in, converted
template <typename D, typename S>
__global__ void k_col_put(D *vbase, long long ld, const int *jp, int off, long long to, const S *in, long long n) {
    D *v = vbase + (long long)(*jp + off) * ld + to;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        v[i] = (D)in[i];
}
// out = x .* d with x basis column *jp (point Jacobi from a column)
template <typename T>
__global__ void k_mul_col(T *out, const T *vbase, long long ld, const int *jp, const T *d, long long n) {
    const T *x = vbase + (long long)(*jp) * ld;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = x[i] * d[i];
}

// ================================================================= AMG
// coarse r_c[I] = sum_{i in I} r[i], bs components: 8 lanes per aggregate
// (aggregates have at most 8 members), member loads in parallel, then a
// fixed xor-shuffle tree inside the 8 lanes
template <typename T>
__global__ void k_restrict(const int *__restrict__ mptr, const int *__restrict__ mem, int nc, int bs, const T *r,
                           T *rc) {
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int I = (int)(g >> 3), l = (int)(g & 7);
    const bool live = I < nc;
    const unsigned mask = 0xffu << (threadIdx.x & 24u);
    int q = 0, beg = 0;
    if (live) { beg = mptr[I]; q = mptr[I + 1] - beg; }
    const int m = (live && l < q) ? mem[beg + l] : -1;
    pdl_wait();
    if (__all_sync(0xffffffffu, !live)) return;   // whole warp past the end
    for (int a = 0; a < bs; ++a) {
        T s = (m >= 0) ? r[(long long)m * bs + a] : T(0);
        s += __shfl_xor_sync(mask, s, 4);
        s += __shfl_xor_sync(mask, s, 2);
        s += __shfl_xor_sync(mask, s, 1);
        if (live && l == 0) rc[(long long)I * bs + a] = s;
    }
}
// Restriction fused with the first Chebyshev step of the coarse level's
// pre-smoothing (which starts from zero): rc = R r, then d = c2 Dinv_c rc and
// x = d, as k_restrict followed by k_cheb_first on the coarse level computes
// them (same operations, same order); rcopy (optional) gets a copy of rc.
template <typename T>
__global__ void k_restrict_first(const int *__restrict__ mptr, const int *__restrict__ mem, int nc, int bs,
                                 const T *r, T *rc, const T *__restrict__ dinv, T c2,
                                 T *d, T *x, T *rcopy) {
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int I = (int)(g >> 3), l = (int)(g & 7);
    const bool live = I < nc;
    const unsigned mask = 0xffu << (threadIdx.x & 24u);
    int q = 0, beg = 0;
    if (live) { beg = mptr[I]; q = mptr[I + 1] - beg; }
    const int m = (live && l < q) ? mem[beg + l] : -1;
    T di[3] = {T(0), T(0), T(0)};   // row l of the coarse block-diagonal inverse
    if (live && l < bs) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (c < bs) di[c] = dinv[(long long)I * bs * bs + l * bs + c];
    }
    pdl_wait();
    if (__all_sync(0xffffffffu, !live)) return;
    T v[3] = {T(0), T(0), T(0)};   // bs <= 3; every lane of the group ends with the sums
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (a < bs) {
            T s = (m >= 0) ? r[(long long)m * bs + a] : T(0);
            s += __shfl_xor_sync(mask, s, 4);
            s += __shfl_xor_sync(mask, s, 2);
            s += __shfl_xor_sync(mask, s, 1);
            v[a] = s;
        }
    }
    if (!live || l >= bs) return;
    // lane l < bs finishes component l of aggregate I
    const long long t = (long long)I * bs + l;
    const T vl = (l == 0) ? v[0] : (l == 1) ? v[1] : v[2];
    rc[t] = vl;
    if (rcopy) rcopy[t] = vl;
    T s = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c)
        if (c < bs) s += di[c] * v[c];
    const T dn = c2 * s;
    if (d) d[t] = dn;   // read by a second pre-smoothing step only
    x[t] = dn;
}
// x[i] += e_c[agg[i]]
template <typename T>
__global__ void k_prolong(const int *__restrict__ agg, int n, int bs, const T *ec, T *x) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)n * bs) return;
    const int i = (int)(t / bs), a = (int)(t - (long long)i * bs);
    const int I = agg[i];
    if (I >= 0) x[t] += ec[(long long)I * bs + a];
}
// The same for blocks of BS components with W = Vec16<T>::W consecutive
// nodes per thread: their map entries and BS 16-byte pieces of x loaded at
// once (the one-component form keeps a single load chain per thread), the
// same per-element adds; the last n % W nodes one per thread.  x and agg
// 16-byte aligned.
template <typename T, int BS>
__global__ void k_prolong_v(const int *__restrict__ agg, int n, const T *ec, T *x) {
    constexpr int W = Vec16<T>::W;
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long ng = n / W;
    pdl_wait();
    if (g < ng) {
        int I[W];
#pragma unroll
        for (int e = 0; e < W; ++e) I[e] = agg[g * W + e];
        T v[BS][W];
#pragma unroll
        for (int c = 0; c < BS; ++c) vld(x + (g * BS + c) * W, v[c]);
#pragma unroll
        for (int k = 0; k < BS * W; ++k) {   // element k: node k / BS, component k % BS
            const int Ik = I[k / BS];
            if (Ik >= 0) v[k / W][k % W] += ec[(long long)Ik * BS + k % BS];
        }
#pragma unroll
        for (int c = 0; c < BS; ++c) vst(x + (g * BS + c) * W, v[c]);
    } else if (g < ng + n % W) {
        const long long i = ng * W + (g - ng);
        const int Ii = agg[i];
        if (Ii >= 0) {
#pragma unroll
            for (int a = 0; a < BS; ++a) x[i * BS + a] += ec[(long long)Ii * BS + a];
        }
    }
}
// Chebyshev first step from x = 0: d = c2 Dinv b; x = d
// (bcopy != nullptr: b is also copied there, for a cycle replayed on fixed buffers)
template <typename T>
__global__ void k_cheb_first(int nbr, int bs, const T *__restrict__ dinv, const T *b, T c2, T *d,
                             T *x, T *bcopy) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)nbr * bs) return;
    const int i = (int)(t / bs), a = (int)(t - (long long)i * bs);
    T di[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int c = 0; c < 3; ++c)
        if (c < bs) di[c] = dinv[(long long)i * bs * bs + a * bs + c];
    pdl_wait();
    if (bcopy) bcopy[t] = b[t];
    T s = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c)
        if (c < bs) s += di[c] * b[(long long)i * bs + c];
    const T dn = c2 * s;
    d[t] = dn;
    x[t] = dn;
}
// x = Cinv b, dense (coarsest level); one warp per row; the inverse is stored
// in the vector type (FP64 or FP32).  Each lane keeps four independent
// partial sums and, when rows start on 16-byte boundaries, reads 16 bytes
// at a time, so a lane has several loads in flight instead of one long
// chain of dependent adds; the partials are added in a fixed order.
template <typename T>
__global__ void k_dense_gemv(const T *__restrict__ Cinv, int n, const T *b, T *x) {
    constexpr int W = Vec16<T>::W;
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int ln = threadIdx.x & 31;
    if (row >= n) return;
    pdl_wait();
    const T *r = Cinv + (long long)row * n;
    T s[4] = {0, 0, 0, 0};
    if (n % W == 0 && ((uintptr_t)Cinv & 15u) == 0 && ((uintptr_t)b & 15u) == 0) {
        const int nv = n / W;
#pragma unroll 4
        for (int c = ln; c < nv; c += 32) {
            T a[W], v[W];
            vld(r + (long long)c * W, a);
            vld(b + (long long)c * W, v);
#pragma unroll
            for (int e = 0; e < W; ++e) s[e % 4] += a[e] * v[e];
        }
    } else {
        int c = ln;
        for (; c + 96 < n; c += 128) {
#pragma unroll
            for (int q = 0; q < 4; ++q) s[q] += r[c + 32 * q] * b[c + 32 * q];
        }
        for (; c < n; c += 32) s[0] += r[c] * b[c];
    }
    T t = (s[0] + s[1]) + (s[2] + s[3]);
    t = warp_sum(t);
    if (ln == 0) x[row] = t;
}

// The FP32 form with a block of kGemvThreads threads (four warps) per row:
// each thread keeps four partial sums over the 16-byte pieces t, t + 128, ...
// of the row, then a fixed warp tree per warp and the four warps' sums in
// order.  A row of a coarsest inverse about 1300 wide is about 330 pieces,
// three per thread, so a row's loads are in flight together instead of ten
// deep in one warp.  VEC: rows on 16-byte boundaries (n % 4 == 0, Cinv and b
// aligned); otherwise single floats c = t, t + 128, ... into the four sums in
// turn.
constexpr int kGemvThreads = 128;
template <typename T, bool VEC>   // float
__global__ void __launch_bounds__(kGemvThreads) k_dense_gemv_rows(const T *__restrict__ Cinv, int n,
                                                                  const T *b, T *x) {
    static_assert(std::is_same<T, float>::value, "FP32 form");
    __shared__ float ws[kGemvThreads / 32];
    const int row = blockIdx.x;
    const float *r = Cinv + (long long)row * n;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    if constexpr (VEC) {
        const int nv = n / 4;
        float a[4] = {0.f, 0.f, 0.f, 0.f}, v[4];
        if ((int)threadIdx.x < nv) vld(r + (long long)threadIdx.x * 4, a);
        pdl_wait();
        for (int c = threadIdx.x; c < nv; c += kGemvThreads) {
            if (c != (int)threadIdx.x) vld(r + (long long)c * 4, a);
            vld(b + (long long)c * 4, v);
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] += a[e] * v[e];
        }
    } else {
        int c = threadIdx.x;
        float a[4];   // the row's first four values of this thread
#pragma unroll
        for (int e = 0; e < 4; ++e) a[e] = c + e * kGemvThreads < n ? r[c + e * kGemvThreads] : 0.f;
        pdl_wait();
        if (n <= 4 * kGemvThreads) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (c + e * kGemvThreads < n) s[e] += a[e] * b[c + e * kGemvThreads];
            c = n;
        }
        for (; c + 3 * kGemvThreads < n; c += 4 * kGemvThreads) {
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] += r[c + e * kGemvThreads] * b[c + e * kGemvThreads];
        }
        for (int e = 0; c < n; c += kGemvThreads, ++e) s[e] += r[c] * b[c];
    }
    float t = (s[0] + s[1]) + (s[2] + s[3]);
    t = warp_sum(t);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        float u = ws[0];
#pragma unroll
        for (int w = 1; w < kGemvThreads / 32; ++w) u += ws[w];
        x[row] = u;
    }
}

// ============================================================== K-cycle
// The inner products of a K-cycle step (see kc_finish; b null in the first)
// where the level's product is the flat kernel or its blocks are 3x3.  Each
// block reduces a fixed contiguous chunk into kd[8 + blk], kd[8 + nb + blk],
// ..., and the last block to finish (ticket in kd[7]) sums the block partials
// in a fixed order: one launch, same result whatever order the blocks run in.
constexpr int kKdotBlocks = 96;
template <typename T>
__global__ void __launch_bounds__(256) k_kdots(const T *y, const T *a, const T *b, long long n, double *kd) {
    pdl_wait();
    const long long chunk = (n + gridDim.x - 1) / gridDim.x;
    const long long lo = (long long)blockIdx.x * chunk, hi = min(n, lo + chunk);
    typename GsSum<T>::type pp[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) gs_set(pp[k], T(0));
    for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        const T u = y[i], p = a[i];
        pp[0] = gs_add(pp[0], gs_mul(u, u));
        pp[1] = gs_add(pp[1], gs_mul(u, p));
        if (b) {
            const T v = b[i];
            pp[2] = gs_add(pp[2], gs_mul(u, v));
            pp[3] = gs_add(pp[3], gs_mul(p, v));
        }
    }
    const int nq = b ? 4 : 2;
    block_partials<T>(pp, nq, kd + 8, 0);
    unsigned *ticket = (unsigned *)(kd + 7);
    if (!grid_last_block(ticket)) return;
    __shared__ double out[4];
    const double w11 = kd[0], a1 = kd[2];
    reduce_partials<T>(kd + 8, gridDim.x, nq, out);
    __syncthreads();
    kc_finish<T>(out, w11, a1, y, a, b, n, kd);
    if (threadIdx.x == 0) *ticket = 0;
}
// r -= a1 w1 with a1 = (w1.r)/(w1.w1) = kd[1]/kd[0], saved in kd[2]; then, where
// the second cycle starts with a smoothing step from zero (dinv set), that
// step: x = c2 Dinv r, and d = x when d is set.  One thread per block row.
template <typename T>
__global__ void k_kupd1(T *r, const T *w1, double *kd, int nbr, int bs, const T *__restrict__ dinv, T c2, T *d, T *x) {
    __shared__ T a1s;
    pdl_wait();
    if (threadIdx.x == 0) {
        const double a1 = kd[0] > 0.0 ? kd[1] / kd[0] : 0.0;
        a1s = (T)a1;
        if (blockIdx.x == 0) kd[2] = a1;
    }
    __syncthreads();
    const T a1 = a1s;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nbr; i += gridDim.x * blockDim.x) {
        T v[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (c < bs) {
                const long long t = (long long)i * bs + c;
                v[c] = r[t] - a1 * w1[t];
                r[t] = v[c];
            }
        if (!dinv) continue;
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (a < bs) {
                T s = 0;
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    if (c < bs) s += dinv[(long long)i * bs * bs + a * bs + c] * v[c];
                const T dn = c2 * s;
                const long long t = (long long)i * bs + a;
                if (d) d[t] = dn;
                x[t] = dn;
            }
    }
}
// x = a1 z1 + a2 (z2 - beta z1), the coefficients of z1 and z2 from kc_finish
template <typename T> __global__ void k_kupd2(T *x, const T *z1, const T *z2, const double *kd, long long n) {
    pdl_wait();
    const T c1 = (T)kd[3], c2 = (T)kd[4];
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        x[i] = c1 * z1[i] + c2 * z2[i];
}

// =============================================================== rank one
// f[k] = r_k * (a^k . x), one block per outlet (fixed-order tree reduction)
template <typename T>
__global__ void k_lowrank_dots(const int *__restrict__ optr, const int *__restrict__ oidx, const double *__restrict__ oval,
                               const double *__restrict__ r, const T *x, double *f,
                               const int *jp = nullptr, long long x_ld = 0) {
    __shared__ double red[8];
    const int k = blockIdx.x;
    const int q0 = optr[k] + threadIdx.x, q1 = optr[k + 1];
    const int i0 = q0 < q1 ? oidx[q0] : 0;
    const double v0 = q0 < q1 ? oval[q0] : 0.0;
    pdl_wait();
    if (jp) x += (long long)*jp * x_ld;   // x is basis column *jp
    double s = q0 < q1 ? v0 * (double)x[i0] : 0.0;
    for (int q = q0 + blockDim.x; q < q1; q += blockDim.x) s += oval[q] * (double)x[oidx[q]];
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        f[k] = r[k] * t;
    }
}

}  // namespace nbp
