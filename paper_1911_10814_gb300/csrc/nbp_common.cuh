// nbp_common.cuh -- shared device helpers and internal data structures of the
// GB300 nested block solver library (libnbp).  Internal header.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cstdint>
#include <cstdio>
#include <functional>
#include <string>
#include <vector>

#include "../../include/nbp.h"

namespace nbp {

constexpr int kMaxLevels = 12;
constexpr int kSMs = 152;                 // GB300: 2 dies x 76 SMs
constexpr int kReduceBlocks = 4 * kSMs;   // fixed grid for deterministic reductions
constexpr int kCoarseDenseMax = 4096;     // largest coarsest level (scalar rows) solved densely

// ------------------------------------------------------------------ errors
struct Error {
    nbp_status st;
    std::string msg;
};

#define NBP_CUDA(call)                                                                        \
    do {                                                                                      \
        cudaError_t _e = (call);                                                              \
        if (_e != cudaSuccess) {                                                              \
            throw ::nbp::Error{_e == cudaErrorMemoryAllocation ? NBP_ERR_OOM : NBP_ERR_CUDA,  \
                               std::string(#call) + ": " + cudaGetErrorString(_e)};           \
        }                                                                                     \
    } while (0)

#define NBP_LAUNCHED()                                                                        \
    do {                                                                                      \
        cudaError_t _e = cudaGetLastError();                                                  \
        if (_e != cudaSuccess)                                                                \
            throw ::nbp::Error{NBP_ERR_CUDA, std::string("kernel launch: ") + cudaGetErrorString(_e)}; \
    } while (0)

inline void require(bool ok, nbp_status st, const std::string &msg) {
    if (!ok) throw Error{st, msg};
}

// ------------------------------------------- programmatic dependent launch
// Inside the device-driven loops a kernel boundary and the first dependent
// loads of the next kernel are a good part of every small kernel's time.
// There consecutive kernels are launched with programmatic stream
// serialization: the next one starts while its predecessor still runs, loads
// what no kernel of a solve writes (matrices, block-diagonal inverses,
// aggregate maps, outlet vectors) and waits (pdl_wait) for the predecessor's
// end before anything else.  Every thread that reads or writes a solve's
// vectors or states waits first; since each kernel waits, the end of one
// implies the end of all before it.  A kernel lets its successor start only
// after its own wait, so that no more than one kernel waits per chain (the
// branches of a batch share the SMs).  Without the attribute both
// instructions are no-ops.
__device__ __forceinline__ void pdl_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// on: this thread is capturing a device-driven solve; prev: the last captured
// node is a kernel (a conditional or copy node cannot be overlapped)
struct PdlState {
    bool on = false, prev = false;
};
inline thread_local PdlState g_pdl;

// kernel<<<grid, block, 0, s>>>(args...), overlapped with its predecessor where
// g_pdl allows; for kernels that call pdl_wait only
template <typename... P, typename... A>
inline void klaunch(void (*kernel)(P...), unsigned grid, unsigned block, cudaStream_t s, A &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = g_pdl.on && g_pdl.prev ? 1 : 0;
    NBP_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
    g_pdl.prev = g_pdl.on;
}

// --------------------------------------------------------------- numerics
template <typename T> struct Acc { using type = T; };
template <> struct Acc<__nv_bfloat16> { using type = float; };

__device__ __forceinline__ double to_d(double v) { return v; }
__device__ __forceinline__ double to_d(float v) { return (double)v; }
__device__ __forceinline__ double to_d(__nv_bfloat16 v) { return (double)__bfloat162float(v); }
__device__ __forceinline__ float to_f(double v) { return (float)v; }
__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename A, typename V> __device__ __forceinline__ A cvt(V v);
template <> __device__ __forceinline__ double cvt<double, double>(double v) { return v; }
template <> __device__ __forceinline__ double cvt<double, float>(float v) { return (double)v; }
template <> __device__ __forceinline__ double cvt<double, __nv_bfloat16>(__nv_bfloat16 v) { return (double)__bfloat162float(v); }
template <> __device__ __forceinline__ float cvt<float, double>(double v) { return (float)v; }
template <> __device__ __forceinline__ float cvt<float, float>(float v) { return v; }
template <> __device__ __forceinline__ float cvt<float, __nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename T> __device__ __forceinline__ T warp_sum(T v, unsigned mask = 0xffffffffu) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
    return v;
}

// Float-float sums (the unevaluated sum hi + lo of two floats, about 44
// significant bits) for the reductions of the FP32 kernels.  GB300's FP64
// pipe retires about two operations per clock and SM (1.25 TFLOP/s for the
// GPU), so a tree of FP64 adds in every block's tail costs microseconds per
// block; these run on the FP32 pipe.  ff_add is Knuth's error-free two-sum of the leading parts, the
// trailing parts added to its error, then Dekker's fast two-sum to
// renormalise; all adds are explicitly rounded (no reassociation).
struct FF {
    float hi, lo;
};
__device__ __forceinline__ FF ff_add(FF a, FF b) {
    const float s = __fadd_rn(a.hi, b.hi);
    const float v = __fsub_rn(s, a.hi);
    float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, v)), __fsub_rn(b.hi, v));
    e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
    const float h = __fadd_rn(s, e);
    return FF{h, __fsub_rn(e, __fsub_rn(h, s))};
}
// the warp's sum in a fixed xor tree; lane 0's value is the one used
__device__ __forceinline__ FF ff_warp_sum(FF a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        FF b;
        b.hi = __shfl_xor_sync(0xffffffffu, a.hi, o);
        b.lo = __shfl_xor_sync(0xffffffffu, a.lo, o);
        a = ff_add(a, b);
    }
    return a;
}
__device__ __forceinline__ double ff_to_double(FF a) { return (double)a.hi + (double)a.lo; }

// ------------------------------------------------------- device structures
// Block CSR matrix with br x bc row-major blocks (nbr block rows).
struct DMat {
    int nbr = 0, nbc = 0, br = 1, bc = 1;
    int64_t nnz = 0;
    int *rp = nullptr, *ci = nullptr;
    double *v = nullptr;             // FP64 values (always present)
    float *v32 = nullptr;            // FP32 copy (mixed precision)
    __nv_bfloat16 *v16 = nullptr;    // BF16 copy (mixed precision)
    // Sliced-ELL copy for square blocks (C-row slices, C = sl_c; slot k of row
    // t of slice s at sl_ptr[s] + C k + t; its bs*bs values component-major:
    // value q of the C slots of one k at (sl_ptr[s] + C k) * bb + C q + t).
    int nslice = 0, sl_c = 32;       // number of slices, rows per slice (8 or 32)
    long long *sl_ptr = nullptr;
    int *sl_ci = nullptr;
    double *sl_v = nullptr;
    float *sl_v32 = nullptr;
    // BF16 values use a paired variant of the same slices (same widths):
    // slots 2p, 2p+1 of a row stored side by side, so that one thread loads
    // both with one 4-byte load (bf16x2) per component and one 8-byte load
    // (int2) of columns: pair slot g = sl2_ptr[s] / 2 + C p, its columns at
    // sl2_ci[2 (g + t) + h], value q at sl_v16[2 ((g bb) + C q + t) + h].  An
    // odd width w's last slot is stored unpaired after the pairs: with
    // g = sl2_ptr[s] + C (w - 1), its columns at sl2_ci[g + t], value q at
    // sl_v16[g bb + C q + t].
    long long *sl2_ptr = nullptr;
    int *sl2_ci = nullptr;
    __nv_bfloat16 *sl_v16 = nullptr;
    int beside = 0;                  // in a batch: threads per row that run, in the sums of the tuned kernel's (fine_threads)
    bool sl_lent = false;            // the sl_* arrays belong to another matrix (lend_sell)
    int tuned = -1;                  // autotuned kernel: -1 untuned, 0 sliced ELL, 1000 + T sliced ELL with T threads per row, other > 0 flat with that many lanes per row
    int bb() const { return br * bc; }
};

// Sparse rank-one data, arranged per velocity block row for the fused epilogue:
// entries lr_rp[i]..lr_rp[i+1]-1 of block row i hold (outlet k, component c, value).
struct LowRank {
    int n_out = 0;
    int no = 0;                              // entries over all outlets
    int *optr = nullptr, *oidx = nullptr;    // per-outlet sparse vectors (device)
    double *oval = nullptr;
    double *r = nullptr;                     // device copy of r_k
    std::vector<double> r_host;
    int *lr_rp = nullptr;                    // N+1
    int *lr_k = nullptr, *lr_c = nullptr;
    double *lr_val = nullptr;
    double *f = nullptr;                     // r_k (a^k . x), device, n_out
    int in_product = -1;                     // the product's blocks take f themselves (SpmvArgs::lr_rev); -1: k_lowrank_dots
};

struct Level {
    DMat M;
    int *agg = nullptr;                      // map to next level (-1 = left out)
    int *mptr = nullptr, *mem = nullptr;     // members of each next-level aggregate
    // A P (rows of this level, columns of the next): the post-smoothing's first
    // residual is r - (A P) e, with r that of before the restriction.  Sliced
    // copies only; empty (no sl_ci) where it was not built
    DMat AP;
    double *dinv = nullptr;                  // bs*bs per row
    float *dinv32 = nullptr;
    double rho = 0.0;
    double cheb_lo = 10.0;                   // Chebyshev interval [rho / cheb_lo, rho]
    // work vectors: [0] b, [1] x, [2] x (ping-pong), [3] r, [4] d, and for the
    // K-cycle [5] r, [6] z1, [7] w1, [8] z2, [9] w2; FP64 and FP32 sets
    static constexpr int kWork = 10;
    double *w64[kWork] = {};
    float *w32[kWork] = {};
    char *work = nullptr;                    // the allocation they lie in
    double *kdots = nullptr;                 // K-cycle inner products (device)
    double *kpart = nullptr;                 // block partials of the K-cycle's product + inner products kernel
    long long kpart_blocks = 0;              // ... for grids up to this many blocks
};

struct Hier {
    int nlev = 0, bs = 1;
    bool kcycle = false;                     // Krylov-accelerated cycle on the coarse levels
    int kdepth = 1;                          // ... 1..kdepth
    int cheb = 2;                            // Chebyshev smoothing degree of this hierarchy
    Level L[kMaxLevels];
    double *cinv = nullptr;                  // coarsest dense inverse (nc x nc, row-major) or null
    float *cinv32 = nullptr;                 // its FP32 copy (FP32 inner solves)
    int nc = 0;
    bool built = false;
};

}  // namespace nbp

namespace nbp {

// ------------------------------------------------------ device memory helpers
// The memory pool of the context this thread works for: set for the extent of
// a call on that context (PoolScope) and null outside, so that no call takes
// memory from another context's pool or through the handle of a destroyed one.
inline thread_local cudaMemPool_t g_pool = nullptr;
struct PoolScope {
    cudaMemPool_t keep;
    explicit PoolScope(cudaMemPool_t pool) : keep(g_pool) { g_pool = pool; }
    ~PoolScope() { g_pool = keep; }
    PoolScope(const PoolScope &) = delete;
    PoolScope &operator=(const PoolScope &) = delete;
};
template <typename T> inline T *dmalloc(size_t n, cudaStream_t s) {
    void *p = nullptr;
    require(g_pool != nullptr, NBP_ERR_STATE, "device memory asked for outside a call on a context");
    NBP_CUDA(cudaMallocFromPoolAsync(&p, (n ? n : 1) * sizeof(T), g_pool, s));
    return (T *)p;
}
inline void dfree(void *p, cudaStream_t s) {
    if (p) cudaFreeAsync(p, s);
}
template <typename T> inline T readback(const T *d, cudaStream_t s) {
    T h;
    NBP_CUDA(cudaMemcpyAsync(&h, d, sizeof(T), cudaMemcpyDeviceToHost, s));
    NBP_CUDA(cudaStreamSynchronize(s));
    return h;
}
inline unsigned grid_for(long long n, int block = 256, long long cap = 16LL * kSMs * 8) {
    long long g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (unsigned)g;
}
inline unsigned grid_exact(long long n, int block = 256) {
    long long g = (n + block - 1) / block;
    return (unsigned)(g < 1 ? 1 : g);
}

void dmat_free(DMat &m, cudaStream_t s);
void drop_sell(DMat &m, cudaStream_t s);
void lend_sell(const DMat &from, DMat &to, cudaStream_t s);
void hier_free(Hier &H, cudaStream_t s);

// Setup entry points (amg_setup.cu)
// Aggregation AMG hierarchy of `fine`; keep_aggregates: rebuild every
// operator of the hierarchy H already holds (same pattern) from the new
// values on its aggregate maps instead of aggregating again.
void amg_build(Hier &H, const DMat &fine, const nbp_options &o, int precision, cudaStream_t s,
               bool keep_aggregates, cudaStream_t side, const std::function<void(int)> &level_ready = nullptr);
void build_shat(const DMat &A, const DMat &B, const DMat &C, const DMat &D, const LowRank &lr, int N, DMat &Shat,
                double *diagA_out, cudaStream_t s);
void make_lowcopies(DMat &m, int precision, cudaStream_t s);
void make_sell(DMat &m, int precision, cudaStream_t s);
void transpose_dmat(const DMat &in, DMat &out, cudaStream_t s);

}  // namespace nbp
