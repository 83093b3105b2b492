// krylov.cu -- non-template kernels of the Krylov layer: the triangular
// solve of the GMRES least-squares problem and the start of a GMRES cycle
// (the Givens update itself is fused into the last Gram-Schmidt kernel of
// each Arnoldi step).
#include "kernels.cuh"

namespace nbp {

// y = H(0:k,0:k)^{-1} g(0:k), upper triangular, by one warp: columns from the
// last, lane i (and i + 32, ...) subtracting column c's term from its rows'
// right-hand sides, so that each step's loads and products run in parallel
// (one thread's row-by-row sums were a chain of dependent loads: 9.3 us per
// inner solve at k = 7).  y holds the running right-hand sides.
__device__ __forceinline__ void trisolve(const double *H, int ldh, const double *g, double *y, int k) {
    const int ln = threadIdx.x & 31;
    if (k <= 32) {   // the right-hand side and the next columns in registers
        double s = ln < k ? g[ln] : 0.0;
        const double d = ln < k ? H[(long long)ln * ldh + ln] : 0.0;
        for (int c1 = k; c1 > 0; c1 -= 8) {   // eight columns' loads in flight
            double h[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int c = c1 - 1 - u;
                h[u] = (c >= 0 && ln < c) ? H[(long long)ln * ldh + c] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int c = c1 - 1 - u;
                if (c < 0) break;
                if (ln == c) s = (d != 0.0) ? s / d : 0.0;
                const double yc = __shfl_sync(0xffffffffu, s, c);
                if (ln < c) s -= h[u] * yc;
            }
        }
        if (ln < k) y[ln] = s;
        return;
    }
    for (int i = ln; i < k; i += 32) y[i] = g[i];
    __syncwarp();
    for (int c = k - 1; c >= 0; --c) {
        const double d = H[(long long)c * ldh + c], yc = (d != 0.0) ? y[c] / d : 0.0;
        __syncwarp();
        if (ln == 0) y[c] = yc;
        for (int i = ln; i < c; i += 32) y[i] -= H[(long long)i * ldh + c] * yc;
        __syncwarp();
    }
}

// launched with one warp
__global__ void k_trisolve(const double *H, int ldh, const double *g, double *y, int k) { trisolve(H, ldh, g, y, k); }

__global__ void k_gm_init(double *g, int m1, const double *beta2, double *beta, GmState *st) {
    const double q = beta2[0];
    const double b = (q >= 0.0) ? sqrt(q) : q;       // NaN passes through (fmax would hide it)
    for (int i = threadIdx.x; i < m1; i += blockDim.x) g[i] = 0.0;
    __syncthreads();
    if (threadIdx.x == 0) {
        g[0] = b;
        *beta = b;
        st->res = b;
        gm_set_beta(st, b);
        st->nan = isfinite(b) ? 0 : 1;
    }
}

__global__ void k_scale_rsqrt(double *v, const double *w, const double *s2, long long n) {
    __shared__ double inv;
    if (threadIdx.x == 0) inv = *s2 > 0.0 ? 1.0 / sqrt(*s2) : 0.0;
    __syncthreads();
    const double f = inv;
    if (f == 0.0) return;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        v[i] = w[i] * f;
}

// ------------------------------------------------ device-driven Krylov loops
// The loop of one GMRES level runs as a graph WHILE node; these one-thread
// (or one-block) kernels keep its state in GmDev and set the node's
// condition at the start and end of a cycle; each iteration ends in the norm
// pass, whose last block applies the Givens update and the stopping rule
// (givens_step).

__global__ void k_dl_init(GmDev *st, double *g, int m1, const double *nrm2, double *beta, GmState *gs,
                          const double *rtol, const double *atol, const int *m, const int *nmax,
                          cudaGraphConditionalHandle h) {
    for (int i = threadIdx.x; i < m1; i += blockDim.x) g[i] = 0.0;
    __syncthreads();
    if (threadIdx.x != 0) return;
    const double q = nrm2[0];
    const double b = (q >= 0.0) ? sqrt(q) : q;   // NaN passes through
    g[0] = b;
    *beta = b;
    gs->res = b;
    gm_set_beta(gs, b);
    gs->nan = isfinite(b) ? 0 : 1;
    st->j = 0;
    st->its = 0;
    st->pad0 = 0;
    st->m = *m;
    st->nmax = *nmax;
    st->bnorm = b;
    st->res = b;
    st->tol = fmax(*rtol * b, *atol);
    st->nan = isfinite(b) ? 0 : 1;
    st->conv = (b <= st->tol) ? 1 : 0;
    st->rel_true = b > 0.0 ? 1.0 : 0.0;
    cudaGraphSetConditional(h, (!st->conv && !st->nan && st->nmax > 0) ? 1u : 0u);
}

__global__ void k_dl_cycle_start(GmDev *st, cudaGraphConditionalHandle h) {
    st->j = 0;
    st->pad0 += 1;   // cycles run (counted for the kernel tally)
    cudaGraphSetConditional(h, 1u);
}

__global__ void k_dl_end(GmDev *st, const double *H, int ldh, const double *g, double *y, long long *its_total,
                         long long *solves) {
    pdl_wait();
    trisolve(H, ldh, g, y, st->j);
    if (threadIdx.x != 0) return;
    st->conv = st->res <= st->tol ? 1 : 0;
    if (its_total) *its_total += st->its;
    if (solves) *solves += 1;
}

__global__ void k_dl_restart(GmDev *st, const double *nrm2, double *g, int m1, double *beta, GmState *gs,
                             cudaGraphConditionalHandle h) {
    const double q = nrm2[0];
    const double r = (q >= 0.0) ? sqrt(q) : q;
    __shared__ int go;
    if (threadIdx.x == 0) {
        st->res = r;
        st->rel_true = st->bnorm > 0.0 ? r / st->bnorm : 0.0;
        if (!isfinite(r)) st->nan = 1;
        st->conv = (r <= st->tol) ? 1 : 0;
        go = (!st->conv && !st->nan && st->its < st->nmax && r != 0.0) ? 1 : 0;
    }
    __syncthreads();
    if (go) {
        for (int i = threadIdx.x; i < m1; i += blockDim.x) g[i] = 0.0;
        __syncthreads();
        if (threadIdx.x == 0) {
            g[0] = r;
            *beta = r;
            gs->res = r;
            gm_set_beta(gs, r);
            gs->nan = 0;
        }
    }
    if (threadIdx.x == 0) cudaGraphSetConditional(h, go ? 1u : 0u);
}

}  // namespace nbp
