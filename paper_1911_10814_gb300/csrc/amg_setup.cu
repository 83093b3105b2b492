// amg_setup.cu -- on-device setup of the nested block solver: aggregation AMG
// hierarchies (strength, handshake matching, aggregate numbering, Galerkin
// product, block-diagonal inverses, Gershgorin bounds, dense coarsest
// inverse), the sparse Schur approximation S_hat = D - C diag(A)^{-1} B
// (paper Sec. 3.1), value copies for mixed precision, and block transposes
// for the adjoint.
//
// Aggregation rule (the paper uses BoomerAMG, Table 1, as prior art; this
// rule is the project's, and the integer aggregate maps are reproducible
// bit for bit because every decision is taken on values computed with the
// same IEEE operations in the same order, with no fused multiply-add):
//   sigma_ij = 0.5 (|A_ij|_F^2 + |A_ji|_F^2) / sqrt(|A_ii|_F^2 |A_jj|_F^2),
//   strong iff sigma_ij >= theta; 3 passes of 64 synchronous handshake rounds
//   (strongest unmatched strong neighbour, ties to the smaller index), pass
//   k+1 on the aggregate graph with max-reduced weights; aggregates numbered
//   by smallest fine index; nodes without any strong connection left out.
#include <cooperative_groups.h>
#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "kernels.cuh"

namespace nbp {

constexpr int kMatchRounds = 64;   // rounds per matching pass (rounds after one that makes no pair change nothing)

// ------------------------------------------------------------- utilities
// the sliced copies of m, freed unless they are another matrix's
void drop_sell(DMat &m, cudaStream_t s) {
    if (!m.sl_lent) {
        dfree(m.sl_ptr, s); dfree(m.sl_ci, s); dfree(m.sl_v, s); dfree(m.sl_v32, s); dfree(m.sl_v16, s);
        dfree(m.sl2_ptr, s); dfree(m.sl2_ci, s);
    }
    m.sl_ptr = nullptr; m.sl_ci = nullptr; m.sl_v = nullptr; m.sl_v32 = nullptr; m.sl_v16 = nullptr;
    m.sl2_ptr = nullptr; m.sl2_ci = nullptr;
    m.sl_lent = false;
}

// `to`, of the same pattern and values, uses the sliced copies of `from`
// until its own are dropped, which has to be before those of `from`
void lend_sell(const DMat &from, DMat &to, cudaStream_t s) {
    drop_sell(to, s);
    to.nslice = from.nslice; to.sl_c = from.sl_c;
    to.sl_ptr = from.sl_ptr; to.sl_ci = from.sl_ci;
    to.sl_v = from.sl_v; to.sl_v32 = from.sl_v32; to.sl_v16 = from.sl_v16;
    to.sl2_ptr = from.sl2_ptr; to.sl2_ci = from.sl2_ci;
    to.sl_lent = true;
}

void dmat_free(DMat &m, cudaStream_t s) {
    dfree(m.rp, s); dfree(m.ci, s); dfree(m.v, s); dfree(m.v32, s); dfree(m.v16, s);
    drop_sell(m, s);
    m = DMat();
}

void hier_free(Hier &H, cudaStream_t s) {
    for (int l = 0; l < H.nlev; ++l) {
        Level &L = H.L[l];
        dmat_free(L.M, s);
        dmat_free(L.AP, s);
        dfree(L.agg, s); dfree(L.mptr, s); dfree(L.mem, s); dfree(L.dinv, s); dfree(L.dinv32, s);
        dfree(L.work, s);
        dfree(L.kdots, s); dfree(L.kpart, s);
        L = Level();
    }
    dfree(H.cinv, s);
    dfree(H.cinv32, s);
    H = Hier();
}

template <typename T> static void exclusive_scan(const T *in, T *out, long long n, cudaStream_t s) {
    size_t bytes = 0;
    NBP_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, bytes, in, out, (int)n, s));
    void *tmp = dmalloc<char>(bytes, s);
    NBP_CUDA(cub::DeviceScan::ExclusiveSum(tmp, bytes, in, out, (int)n, s));
    dfree(tmp, s);
}

template <typename K, typename V>
static void sort_pairs(K *&keys, V *&vals, long long n, int end_bit, cudaStream_t s) {
    require(n < (1LL << 31), NBP_ERR_INVALID, "setup: sort of more than 2^31 items");
    K *k2 = dmalloc<K>(n, s);
    V *v2 = dmalloc<V>(n, s);
    size_t bytes = 0;
    NBP_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, bytes, keys, k2, vals, v2, (int)n, 0, end_bit, s));
    void *tmp = dmalloc<char>(bytes, s);
    NBP_CUDA(cub::DeviceRadixSort::SortPairs(tmp, bytes, keys, k2, vals, v2, (int)n, 0, end_bit, s));
    dfree(tmp, s);
    dfree(keys, s); dfree(vals, s);
    keys = k2; vals = v2;
}

static int bits_for(unsigned long long maxkey) {
    int b = 1;
    while (b < 64 && (maxkey >> b) != 0ULL) ++b;
    return b;
}

__device__ __forceinline__ double fnorm2_rn(const double *blk, int nb) {
    double s = __dmul_rn(blk[0], blk[0]);
    for (int t = 1; t < nb; ++t) s = __dadd_rn(s, __dmul_rn(blk[t], blk[t]));
    return s;
}

__device__ __forceinline__ int find_entry(const int *rp, const int *ci, int i, int j) {
    int lo = rp[i], hi = rp[i + 1] - 1;
    while (lo <= hi) {
        int mid = (lo + hi) >> 1;
        int c = ci[mid];
        if (c == j) return mid;
        if (c < j) lo = mid + 1; else hi = mid - 1;
    }
    return -1;
}

// ------------------------------------------------------ strength graph
__global__ void k_diag_norm(int n, int nb, const int *rp, const int *ci, const double *v, double *dn) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int e = find_entry(rp, ci, i, i);
    dn[i] = (e >= 0) ? fnorm2_rn(v + (long long)e * nb, nb) : 0.0;
}

// w[e] = sigma_ij for off-diagonal entries, -1 on the diagonal.  Eight lanes
// per row: every entry is a chain of its own (the search for (j, i), then two
// blocks), which one thread per row ran one after another (0.56M-unknown
// tangent, all levels: 1.69 -> 1.13 ms).
constexpr int kStrengthLanes = 8;
__global__ void k_strength(int n, int nb, const int *rp, const int *ci, const double *v, const double *dn, double *w) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int i = (int)(t / kStrengthLanes);
    if (i >= n) return;
    for (int e = rp[i] + (int)(t % kStrengthLanes); e < rp[i + 1]; e += kStrengthLanes) {
        const int j = ci[e];
        if (j == i) { w[e] = -1.0; continue; }
        const double fij = fnorm2_rn(v + (long long)e * nb, nb);
        const int et = find_entry(rp, ci, j, i);
        const double fji = (et >= 0) ? fnorm2_rn(v + (long long)et * nb, nb) : 0.0;
        const double d = __dmul_rn(dn[i], dn[j]);
        const double h = __dmul_rn(__dadd_rn(fij, fji), 0.5);
        w[e] = (d > 0.0) ? __ddiv_rn(h, __dsqrt_rn(d)) : 0.0;
    }
}

__global__ void k_isolated(int n, const int *rp, const int *ci, const double *w, double theta, int *iso) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int is = 1;
    for (int e = rp[i]; e < rp[i + 1]; ++e)
        if (ci[e] != i && w[e] >= theta) { is = 0; break; }
    iso[i] = is;
}

// --------------------------------------------------------- matching pass
// A handshake round: every unmatched node picks its strongest unmatched strong
// neighbour (ties to the smaller index), and mutual picks become pairs.  A
// node without a candidate never gets one (the matched set only grows), and a
// round that makes no pair is the last that could.  So the rounds run over a
// list of the nodes still in play, and stop at the first without a pair, with
// the result of kMatchRounds rounds over all nodes.
// 0.56M-unknown tangent, 21 passes: 17.3 ms in 2,688 launches -> 3.1 ms in 117.
//
// The candidates of node u scanned by kPickLanes lanes: the strongest, ties
// to the smaller index, is the same in any order.  mate is read past L1
// (__ldcg): other blocks of the cluster kernel write it.
constexpr int kPickLanes = 4;
__device__ __forceinline__ int pick_of(int u, int l, const int *rp, const int *ci, const double *w, double theta,
                                       const int *mate) {
    int p = -1;
    double best = 0.0;
    if (u >= 0) {
        const int e1 = rp[u + 1];
#pragma unroll 4
        for (int e = rp[u] + l; e < e1; e += kPickLanes) {
            const int v = ci[e];
            const double wv = w[e];
            const bool ok = v != u && wv >= theta && __ldcg(mate + v) < 0;
            if (ok && (p < 0 || wv > best || (wv == best && v < p))) { best = wv; p = v; }
        }
    }
#pragma unroll
    for (int o = 1; o < kPickLanes; o <<= 1) {
        const int q = __shfl_xor_sync(0xffffffffu, p, o);
        const double bq = __shfl_xor_sync(0xffffffffu, best, o);
        if (q >= 0 && (p < 0 || bq > best || (bq == best && q < p))) { best = bq; p = q; }
    }
    return p;
}

// One round over the nodes of list (all n when null; their number at count):
// pick, then (next launch) pair; nodes that stay in play go to next / *ncount.
__global__ void __launch_bounds__(256) k_pick(int n, const int *list, const int *count, const int *rp, const int *ci,
                                              const double *w, double theta, const int *mate, int *pick) {
    const int na = list ? *count : n, l = threadIdx.x % kPickLanes;
    const long long step = (long long)gridDim.x * blockDim.x / kPickLanes;
    // whole warps stay in the loop together (the lanes' shuffles)
    for (long long i0 = ((long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / kPickLanes; i0 < na; i0 += step) {
        const long long i = i0 + (threadIdx.x & 31) / kPickLanes;
        const int u = i < na ? (list ? list[i] : (int)i) : -1;
        const int p = pick_of(u, l, rp, ci, w, theta, mate);
        if (u >= 0 && l == 0) pick[u] = p;
    }
}
__global__ void __launch_bounds__(256) k_pair(int n, const int *list, const int *count, const int *pick, int *mate,
                                              int *next, int *ncount) {
    const int na = list ? *count : n;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < na; i0 += step) {
        const long long i = i0 + (threadIdx.x & 31);
        const int u = i < na ? (list ? list[i] : (int)i) : -1;
        const int v = u >= 0 ? pick[u] : -1;
        bool stay = v >= 0;
        if (stay && pick[v] == u) { mate[u] = v; stay = false; }
        const unsigned m = __ballot_sync(0xffffffffu, stay);   // one atomic per warp; the list's order does not matter
        int base = 0;
        if ((threadIdx.x & 31) == 0 && m) base = atomicAdd(ncount, __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (stay) next[base + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))] = u;
    }
}

// The remaining rounds in one cluster: few nodes are left in play (or the
// graph is small), so a round is a chain of loads, not bandwidth, and two
// cluster barriers (about 1 us each) replace two launches over all nodes.
// made[r] (zeroed): a pair was made in round r.
constexpr int kMatchCluster = 8, kMatchThreads = 1024;
constexpr int kMatchTail = 2 * kMatchCluster * kMatchThreads;   // list length the cluster takes over at
__global__ void __cluster_dims__(kMatchCluster, 1, 1) __launch_bounds__(kMatchThreads)
    k_match_tail(int n, const int *list, const int *count, const int *rp, const int *ci, const double *w, double theta,
                 int round0, int *mate, int *pick, int *made) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int na = list ? *count : n;
    const int T = kMatchCluster * kMatchThreads, me = (int)cl.block_rank() * kMatchThreads + (int)threadIdx.x;
    const int l = me % kPickLanes;
    for (int r = round0; r < kMatchRounds; ++r) {
        for (int i0 = (me & ~31) / kPickLanes; i0 < na; i0 += T / kPickLanes) {
            const int i = i0 + (me & 31) / kPickLanes;
            int u = i < na ? (list ? list[i] : i) : -1;
            // out of play: matched, or without a candidate in an earlier round
            if (u >= 0 && (__ldcg(mate + u) >= 0 || (r > round0 && __ldcg(pick + u) < 0))) u = -1;
            if (__all_sync(0xffffffffu, u < 0)) continue;
            const int p = pick_of(u, l, rp, ci, w, theta, mate);
            if (u >= 0 && l == 0) pick[u] = p;
        }
        cl.sync();
        int mine = 0;
        for (int i = me; i < na; i += T) {
            const int u = list ? list[i] : i;
            if (__ldcg(mate + u) >= 0) continue;
            const int v = __ldcg(pick + u);
            if (v >= 0 && __ldcg(pick + v) == u) { mate[u] = v; mine = 1; }
        }
        if (__syncthreads_or(mine) && threadIdx.x == 0) made[r] = 1;
        cl.sync();
        if (__ldcg(made + r) == 0) break;   // the same for the whole cluster
    }
}

// Numbering of a pass's aggregates by smallest node, and their member lists:
// the root of a pair is its smaller node, so one scan over the nodes of
// (1, members) of every root, packed in 64 bits, gives a root's aggregate and
// where its members start (ascending).  No sort.
__global__ void k_root_size(int n, const int *mate, unsigned long long *v) {
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u > n) return;
    const int m = u < n ? mate[u] : -1;
    const bool root = u < n && (m < 0 || m > u);
    v[u] = root ? (1ULL << 32) | (m >= 0 ? 2ULL : 1ULL) : 0ULL;
}
__global__ void k_pair_members(int n, const int *mate, const unsigned long long *at, int *map, int *mptr, int *mem) {
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u > n) return;
    if (u == n) { mptr[at[n] >> 32] = n; return; }   // the end of the last list
    const int m = mate[u];
    const int root = (m >= 0 && m < u) ? m : u;
    const unsigned long long v = at[root];
    const int I = (int)(v >> 32), p = (int)(v & 0xffffffffULL);
    map[u] = I;
    mem[root == u ? p : p + 1] = u;
    if (root == u) mptr[I] = p;
}

__global__ void k_iota(int n, int *a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = i;
}

// row index of every stored entry
__global__ void k_entry_rows(int n, const int *rp, int *row) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int e = rp[i]; e < rp[i + 1]; ++e) row[e] = i;
}

// keys of an aggregate graph: (map[u], map[v]) for u != v aggregates, sentinel otherwise
__global__ void k_cg_keys(long long nnz, const int *row, const int *ci, const int *map, unsigned long long ncl,
                          int drop_diag, unsigned long long *key, long long *idx) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nnz) return;
    const int I = map[row[e]], J = map[ci[e]];
    const bool drop = I < 0 || J < 0 || (drop_diag && I == J);
    key[e] = drop ? ~0ULL : (unsigned long long)I * ncl + (unsigned long long)J;
    idx[e] = e;
}

// segment heads of sorted keys (sentinel keys are never heads)
__global__ void k_heads(long long n, const unsigned long long *key, int *head) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const unsigned long long k = key[t];
    head[t] = (k != ~0ULL && (t == 0 || key[t - 1] != k)) ? 1 : 0;
}

// start position of each segment; segment s = sid[t] for heads
__global__ void k_seg_starts(long long n, const int *head, const int *sid, long long *start) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    if (head[t]) start[sid[t]] = t;
}

// coarse graph rows: count per row then scan
__global__ void k_seg_rowcount(int nseg, const unsigned long long *key, const long long *start, unsigned long long ncl,
                               int *cnt) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nseg) return;
    const unsigned long long k = key[start[s]];
    atomicAdd(cnt + (int)(k / ncl), 1);
}

// aggregate graph edges: column and max weight over the segment
__global__ void k_cg_fill(int nseg, const unsigned long long *key, const long long *start, long long nvalid,
                          const long long *idx, const double *w, unsigned long long ncl, int *ci_out, double *w_out) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nseg) return;
    const long long a = start[s];
    const long long b = (s + 1 < nseg) ? start[s + 1] : nvalid;
    const unsigned long long k = key[a];
    double m = w[idx[a]];
    for (long long t = a + 1; t < b; ++t) m = fmax(m, w[idx[t]]);
    ci_out[s] = (int)(k % ncl);
    w_out[s] = m;
}

// Galerkin: coarse block = sequential sum of the segment's fine blocks in
// ascending fine entry order (ascending (row, column))
__global__ void k_galerkin_fill(int nseg, int nb, const unsigned long long *key, const long long *start, long long nvalid,
                                const long long *idx, const double *v, unsigned long long ncl, int *ci_out, double *v_out) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nseg) return;
    const long long a = start[s];
    const long long b = (s + 1 < nseg) ? start[s + 1] : nvalid;
    ci_out[s] = (int)(key[a] % ncl);
    double acc[9];
    const double *src = v + idx[a] * nb;
    for (int q = 0; q < nb; ++q) acc[q] = src[q];
    for (long long t = a + 1; t < b; ++t) {
        src = v + idx[t] * nb;
        for (int q = 0; q < nb; ++q) acc[q] = __dadd_rn(acc[q], src[q]);
    }
    for (int q = 0; q < nb; ++q) v_out[(long long)s * nb + q] = acc[q];
}

__global__ void k_count_valid(long long n, const unsigned long long *key, unsigned long long *cnt) {
    // number of non-sentinel keys = position of the first sentinel (keys sorted)
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const bool valid = key[t] != ~0ULL;
    const bool next_invalid = (t + 1 == n) || key[t + 1] == ~0ULL;
    if (valid && next_invalid) *cnt = (unsigned long long)(t + 1);
}

// ---------------------------------------------------- diagonal inverses
__global__ void k_block_dinv(int n, int bs, const int *rp, const int *ci, const double *v, double *dinv, int *singular) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int e = find_entry(rp, ci, i, i);
    double *o = dinv + (long long)i * bs * bs;
    if (bs == 1) {
        const double a = (e >= 0) ? v[e] : 0.0;
        o[0] = (a != 0.0) ? 1.0 / a : 0.0;
        if (a == 0.0) atomicAdd(singular, 1);
        return;
    }
    double a[9];
    for (int q = 0; q < 9; ++q) a[q] = (e >= 0) ? v[(long long)e * 9 + q] : 0.0;
    const double c00 = a[4] * a[8] - a[5] * a[7], c01 = a[5] * a[6] - a[3] * a[8], c02 = a[3] * a[7] - a[4] * a[6];
    const double det = a[0] * c00 + a[1] * c01 + a[2] * c02;
    if (det == 0.0) {
        for (int q = 0; q < 9; ++q) o[q] = 0.0;
        atomicAdd(singular, 1);
        return;
    }
    const double id = 1.0 / det;
    o[0] = c00 * id; o[1] = (a[2] * a[7] - a[1] * a[8]) * id; o[2] = (a[1] * a[5] - a[2] * a[4]) * id;
    o[3] = c01 * id; o[4] = (a[0] * a[8] - a[2] * a[6]) * id; o[5] = (a[2] * a[3] - a[0] * a[5]) * id;
    o[6] = c02 * id; o[7] = (a[1] * a[6] - a[0] * a[7]) * id; o[8] = (a[0] * a[4] - a[1] * a[3]) * id;
}

// Gershgorin bound of D_b^{-1} A: max over scalar rows of sum |(D_b^{-1} A)_rc|
__global__ void k_gershgorin(int n, int bs, const int *rp, const double *v, const double *dinv, unsigned long long *rho_bits) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int nb = bs * bs;
    const double *di = dinv + (long long)i * nb;
    double mx = 0.0;
    for (int a = 0; a < bs; ++a) {
        double s = 0.0;
        for (int e = rp[i]; e < rp[i + 1]; ++e) {
            const double *blk = v + (long long)e * nb;
            for (int c = 0; c < bs; ++c) {
                double t = 0.0;
                for (int k = 0; k < bs; ++k) t += di[a * bs + k] * blk[k * bs + c];
                s += fabs(t);
            }
        }
        mx = fmax(mx, s);
    }
    atomicMax(rho_bits, (unsigned long long)__double_as_longlong(mx));   // order-free for x >= 0
}

// --------------------------------------------------- dense coarsest solve
__global__ void k_dense_from_bsr(int nbr, int bs, const int *rp, const int *ci, const double *v, double *Dm) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nbr) return;
    const int n = nbr * bs, nb = bs * bs;
    for (int e = rp[i]; e < rp[i + 1]; ++e)
        for (int a = 0; a < bs; ++a)
            for (int b = 0; b < bs; ++b)
                Dm[(long long)(i * bs + a) * n + (long long)ci[e] * bs + b] += v[(long long)e * nb + a * bs + b];
}
// Blocked in-place Gauss-Jordan inverse with partial pivoting (rows k.. of
// column k, ties to the smaller row): panels of b columns, each eliminated in
// one block's shared memory, then applied to the whole matrix by k_inv_update.
// In place of [M | I], column k of the panel becomes column k of the
// eliminations' product G, so half of the elements and no identity are
// touched.  A pivot costs two block barriers and its share of a panel's two
// launches instead of three launches over 2 n^2 elements (the coarsest levels of the 0.56M-unknown tangent, 656 pivots:
// 11.0 -> 3.6 us a pivot).  Candidates are compared by their bits (|x| as an
// integer orders as the value does), which keeps them off the narrow FP64 pipe.
constexpr int kInvThreads = 1024;
__global__ void __launch_bounds__(kInvThreads) k_inv_panel(int n, int k0, int b, const double *M, double *G, int *piv,
                                                           int *perm, int *fail) {
    extern __shared__ double S[];              // S[t n + i]: column k0 + t of the panel
    int *sperm = reinterpret_cast<int *>(S + (size_t)b * n);
    __shared__ double row[8];
    __shared__ unsigned long long wv[32];
    __shared__ int wi[32];
    const int tid = threadIdx.x, warp = tid >> 5, ln = tid & 31;
    if (*fail) return;
    for (int q = tid; q < b * n; q += kInvThreads) {
        const int i = q / b, t = q - i * b;
        S[(size_t)t * n + i] = M[(long long)i * n + k0 + t];
    }
    for (int i = tid; i < n; i += kInvThreads) sperm[i] = perm[i];
    __syncthreads();
    unsigned long long best = 0;
    int arg = n;
    auto offer = [&](double x, int i) {   // rows come in ascending order
        const unsigned long long u = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL;
        if (u > best || (u == best && i < arg)) { best = u; arg = i; }
    };
    for (int i = tid; i < n; i += kInvThreads)
        if (i >= k0) offer(S[i], i);
    for (int t = 0; t < b; ++t) {
        const int k = k0 + t;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long u = __shfl_xor_sync(0xffffffffu, best, o);
            const int q = __shfl_xor_sync(0xffffffffu, arg, o);
            if (u > best || (u == best && q < arg)) { best = u; arg = q; }
        }
        if (ln == 0) { wv[warp] = best; wi[warp] = arg; }
        __syncthreads();
        best = wv[ln];
        arg = wi[ln];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long u = __shfl_xor_sync(0xffffffffu, best, o);
            const int q = __shfl_xor_sync(0xffffffffu, arg, o);
            if (u > best || (u == best && q < arg)) { best = u; arg = q; }
        }
        const int p = arg;
        if (best == 0) {   // the same in every thread
            if (tid == 0) *fail = 1;
            return;
        }
        if (tid < b) {
            const double ip = 1.0 / S[(size_t)t * n + p];
            const double a = S[(size_t)tid * n + k], q = S[(size_t)tid * n + p];
            __syncwarp((1u << b) - 1u);   // every lane has read the pivot
            if (p != k) S[(size_t)tid * n + p] = a;
            const double r = tid == t ? ip : q * ip;
            row[tid] = r;
            S[(size_t)tid * n + k] = r;
        } else if (tid == 32) {
            piv[k] = p;
            const int u = sperm[k];
            sperm[k] = sperm[p];
            sperm[p] = u;
        }
        __syncthreads();
        best = 0;
        arg = n;
        const double rt = row[t];
        for (int i = tid; i < n; i += kInvThreads) {
            if (i == k) continue;
            const double f = S[(size_t)t * n + i];
            for (int c = 0; c < b; ++c) {
                if (c == t) continue;
                const double x = S[(size_t)c * n + i] - f * row[c];
                S[(size_t)c * n + i] = x;
                if (c == t + 1 && i > k) offer(x, i);
            }
            S[(size_t)t * n + i] = -f * rt;
        }
    }
    __syncthreads();
    for (int q = tid; q < b * n; q += kInvThreads) {
        const int i = q / b, t = q - i * b;
        G[(long long)i * 8 + t] = S[(size_t)t * n + i];
    }
    for (int i = tid; i < n; i += kInvThreads) perm[i] = sperm[i];
}
// The panel's eliminations applied to every column: out = (rows outside the
// panel's k0 .. k0 + b - 1 of the row-swapped M, zero inside) + G X, X the b
// panel rows of the row-swapped M; the panel's own columns become G.  32 x 32
// tiles: enough blocks for every SM's FP64 pipe from n = 400 on.
__global__ void __launch_bounds__(256) k_inv_update(int n, int k0, int b, const double *M, const double *G, const int *piv,
                                                    double *out, const int *fail) {
    __shared__ double gs[32][9], xs[8][32];
    __shared__ int src[32], xsrc[8];
    if (*fail) return;
    const int c = threadIdx.x & 31, r0 = threadIdx.x >> 5;
    const int j = blockIdx.x * 32 + c, i0 = blockIdx.y * 32;
    auto trace = [&](int i) {   // the row of M that the swaps brought to row i
        for (int t = b - 1; t >= 0; --t) {
            const int p = piv[k0 + t];
            if (i == k0 + t) i = p;
            else if (i == p) i = k0 + t;
        }
        return i;
    };
    if (threadIdx.x < 32) src[threadIdx.x] = i0 + (int)threadIdx.x < n ? trace(i0 + (int)threadIdx.x) : 0;
    else if ((int)threadIdx.x < 32 + b) xsrc[threadIdx.x - 32] = trace(k0 + (int)threadIdx.x - 32);
    {
        const int i = threadIdx.x >> 3, t = threadIdx.x & 7;
        gs[i][t] = (i0 + i < n && t < b) ? G[(long long)(i0 + i) * 8 + t] : 0.0;
    }
    __syncthreads();
    if (r0 < b && j < n) xs[r0][c] = M[(long long)xsrc[r0] * n + j];
    __syncthreads();
    if (j >= n) return;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int r = r0 + 8 * q, i = i0 + r;
        if (i >= n) break;
        double x;
        if (j >= k0 && j < k0 + b) {
            x = gs[r][j - k0];
        } else {
            x = (i >= k0 && i < k0 + b) ? 0.0 : M[(long long)src[r] * n + j];
            for (int t = 0; t < b; ++t) x += gs[r][t] * xs[t][c];
        }
        out[(long long)i * n + j] = x;
    }
}
// column perm[k] of the inverse is column k of the in-place result
__global__ void k_inv_columns(int n, const double *M, const int *perm, double *inv) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)n * n) return;
    const int i = (int)(t / n), k = (int)(t - (long long)i * n);
    inv[(long long)i * n + perm[k]] = M[t];
}

// --------------------------------------------------- value copies
__global__ void k_to_f32(const double *a, float *b, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) b[i] = (float)a[i];
}
__global__ void k_to_bf16(const double *a, __nv_bfloat16 *b, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        b[i] = __float2bfloat16_rn((float)a[i]);
}

// ------------------------------------------------------------ sliced ELL
__global__ void k_sell_width(int nbr, int nslice, int C, const int *rp, long long *slots) {
    const int sl = blockIdx.x * blockDim.x + threadIdx.x;
    if (sl >= nslice) return;
    int w = 0;
    for (int t = 0; t < C; ++t) {
        const int i = sl * C + t;
        if (i < nbr) w = max(w, rp[i + 1] - rp[i]);
    }
    slots[sl] = (long long)C * w;
}
// BF16 values and columns in the paired layout (see DMat::sl2_ptr)
__global__ void k_sell_fill2(int nbr, int nslice, int C, int bb, const int *rp, const int *ci, const double *v,
                             const long long *sp2, int *sci2, __nv_bfloat16 *sv16) {
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    const int sl = row / C, t = row % C;
    if (sl >= nslice) return;
    const long long base = sp2[sl], base2 = base / 2;
    const int w = (int)((sp2[sl + 1] - base) / C);
    const int len = (row < nbr) ? rp[row + 1] - rp[row] : 0;
    const int e0 = (row < nbr) ? rp[row] : 0;
    for (int k = 0; k < w; ++k) {
        const bool real = k < len;
        const int col = real ? ci[e0 + k] : 0;
        if (k < (w & ~1)) {   // slot of pair k / 2
            const long long g = base2 + (long long)C * (k >> 1);
            const int h = k & 1;
            sci2[2 * (g + t) + h] = col;
            for (int q = 0; q < bb; ++q) {
                const double val = real ? v[(long long)(e0 + k) * bb + q] : 0.0;
                sv16[2 * (g * bb + (long long)C * q + t) + h] = __float2bfloat16_rn((float)val);
            }
        } else {              // the unpaired last slot of an odd width
            const long long g = base + (long long)C * k;
            sci2[g + t] = col;
            for (int q = 0; q < bb; ++q) {
                const double val = real ? v[(long long)(e0 + k) * bb + q] : 0.0;
                sv16[g * bb + (long long)C * q + t] = __float2bfloat16_rn((float)val);
            }
        }
    }
}
__global__ void k_sell_fill(int nbr, int nslice, int C, int bb, const int *rp, const int *ci, const double *v,
                            const long long *sp, int *sci, double *sv, float *sv32) {
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    const int sl = row / C, t = row % C;
    if (sl >= nslice) return;
    const long long base = sp[sl];
    const int w = (int)((sp[sl + 1] - base) / C);
    const int len = (row < nbr) ? rp[row + 1] - rp[row] : 0;
    const int e0 = (row < nbr) ? rp[row] : 0;
    for (int k = 0; k < w; ++k) {
        const long long g = base + (long long)C * k;
        const bool real = k < len;
        sci[g + t] = real ? ci[e0 + k] : 0;
        for (int q = 0; q < bb; ++q) {
            const double val = real ? v[(long long)(e0 + k) * bb + q] : 0.0;
            const long long o = g * bb + (long long)C * q + t;
            sv[o] = val;
            if (sv32) sv32[o] = (float)val;
        }
    }
}

// slice pointers for slice height C; returns the padded slot count
static long long sell_layout(const DMat &m, int C, long long *&sp, cudaStream_t s) {
    const int ns = (m.nbr + C - 1) / C;
    long long *slots = dmalloc<long long>(ns + 1, s);
    k_sell_width<<<grid_exact(ns), 256, 0, s>>>(m.nbr, ns, C, m.rp, slots);
    NBP_LAUNCHED();
    NBP_CUDA(cudaMemsetAsync(slots + ns, 0, sizeof(long long), s));
    sp = dmalloc<long long>(ns + 1, s);
    exclusive_scan(slots, sp, ns + 1, s);
    dfree(slots, s);
    return readback(sp + ns, s);
}

// Slice layout: 32-row slices unless their padding exceeds 10 % of the
// stored blocks, else 8-row slices.  The paired BF16 layout uses the same
// slices: every slot is stored, an odd width's last slot unpaired.  (Rows
// sorted by length within windows of 256 rows cut the padding of the coarse
// levels by 15-30 % but made their products slower: the rows that a warp
// takes no longer share their neighbours' x entries.)
void make_sell(DMat &m, int precision, cudaStream_t s) {
    if (m.nbr == 0) return;
    if (m.sl_ci && (precision < 1 || m.sl_v32) && (precision < 2 || m.sl_v16)) return;   // 2, 3: FP32 and BF16
    drop_sell(m, s);
    int C = 32;
    long long total = sell_layout(m, 32, m.sl_ptr, s);
    if (total > m.nnz + m.nnz / 10) {
        dfree(m.sl_ptr, s);
        C = 8;
        total = sell_layout(m, 8, m.sl_ptr, s);
    }
    m.sl_c = C;
    m.nslice = (m.nbr + C - 1) / C;
    const int bb = m.bb();
    m.sl_ci = dmalloc<int>(total, s);
    m.sl_v = dmalloc<double>(total * bb, s);
    if (precision >= 1) m.sl_v32 = dmalloc<float>(total * bb, s);
    k_sell_fill<<<grid_exact((long long)m.nslice * C), 256, 0, s>>>(m.nbr, m.nslice, C, bb, m.rp, m.ci, m.v, m.sl_ptr,
                                                                    m.sl_ci, m.sl_v, m.sl_v32);
    NBP_LAUNCHED();
    if (precision >= 2) {   // BF16: paired layout over the same slices
        m.sl2_ptr = dmalloc<long long>(m.nslice + 1, s);
        NBP_CUDA(cudaMemcpyAsync(m.sl2_ptr, m.sl_ptr, sizeof(long long) * (m.nslice + 1), cudaMemcpyDeviceToDevice, s));
        m.sl2_ci = dmalloc<int>(total, s);
        m.sl_v16 = dmalloc<__nv_bfloat16>(total * bb, s);
        k_sell_fill2<<<grid_exact((long long)m.nslice * C), 256, 0, s>>>(m.nbr, m.nslice, C, bb, m.rp, m.ci, m.v,
                                                                         m.sl2_ptr, m.sl2_ci, m.sl_v16);
        NBP_LAUNCHED();
    }
}

void make_lowcopies(DMat &m, int precision, cudaStream_t s) {
    const long long nv = m.nnz * m.bb();
    if (precision >= 1 && !m.v32) {
        m.v32 = dmalloc<float>(nv, s);
        k_to_f32<<<grid_for(nv), 256, 0, s>>>(m.v, m.v32, nv);
        NBP_LAUNCHED();
    }
    if (precision >= 2 && !m.v16) {
        m.v16 = dmalloc<__nv_bfloat16>(nv, s);
        k_to_bf16<<<grid_for(nv), 256, 0, s>>>(m.v, m.v16, nv);
        NBP_LAUNCHED();
    }
}

// ================================================================ aggregation
struct Graph {
    int n = 0;
    long long nnz = 0;
    int *rp = nullptr, *ci = nullptr;
    double *w = nullptr;
};
static void graph_free(Graph &g, cudaStream_t s) { dfree(g.rp, s); dfree(g.ci, s); dfree(g.w, s); g = Graph(); }

// Sort entries by (map[row], map[col]) and return segments.
struct Segments {
    unsigned long long *key = nullptr;
    long long *idx = nullptr;
    long long *start = nullptr;
    long long nvalid = 0;
    int nseg = 0;
};
static void free_segments(Segments &sg, cudaStream_t s) { dfree(sg.key, s); dfree(sg.idx, s); dfree(sg.start, s); sg = Segments(); }

static Segments group_by_coarse(int n, long long nnz, const int *rp, const int *ci, const int *map, int ncl, int drop_diag,
                                cudaStream_t s) {
    Segments sg;
    if (nnz == 0 || ncl == 0) return sg;
    int *row = dmalloc<int>(nnz, s);
    k_entry_rows<<<grid_exact(n), 256, 0, s>>>(n, rp, row);
    NBP_LAUNCHED();
    sg.key = dmalloc<unsigned long long>(nnz, s);
    sg.idx = dmalloc<long long>(nnz, s);
    k_cg_keys<<<grid_exact(nnz), 256, 0, s>>>(nnz, row, ci, map, (unsigned long long)ncl, drop_diag, sg.key, sg.idx);
    NBP_LAUNCHED();
    dfree(row, s);
    // full 64-bit sort so that the sentinel (all ones) lands last
    sort_pairs(sg.key, sg.idx, nnz, 64, s);
    unsigned long long *cnt = dmalloc<unsigned long long>(1, s);
    NBP_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), s));
    k_count_valid<<<grid_exact(nnz), 256, 0, s>>>(nnz, sg.key, cnt);
    NBP_LAUNCHED();
    sg.nvalid = (long long)readback(cnt, s);
    dfree(cnt, s);
    if (sg.nvalid == 0) return sg;
    int *head = dmalloc<int>(sg.nvalid + 1, s), *sid = dmalloc<int>(sg.nvalid + 1, s);
    k_heads<<<grid_exact(sg.nvalid), 256, 0, s>>>(sg.nvalid, sg.key, head);
    NBP_LAUNCHED();
    NBP_CUDA(cudaMemsetAsync(head + sg.nvalid, 0, sizeof(int), s));
    exclusive_scan(head, sid, sg.nvalid + 1, s);
    sg.nseg = readback(sid + sg.nvalid, s);
    sg.start = dmalloc<long long>(sg.nseg + 1, s);
    k_seg_starts<<<grid_exact(sg.nvalid), 256, 0, s>>>(sg.nvalid, head, sid, sg.start);
    NBP_LAUNCHED();
    dfree(head, s); dfree(sid, s);
    return sg;
}

static int *rowptr_from_segments(const Segments &sg, int ncl, cudaStream_t s) {
    int *cnt = dmalloc<int>(ncl + 1, s);
    NBP_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * (ncl + 1), s));
    if (sg.nseg > 0) {
        k_seg_rowcount<<<grid_exact(sg.nseg), 256, 0, s>>>(sg.nseg, sg.key, sg.start, (unsigned long long)ncl, cnt);
        NBP_LAUNCHED();
    }
    int *rp = dmalloc<int>(ncl + 1, s);
    exclusive_scan(cnt, rp, ncl + 1, s);
    dfree(cnt, s);
    return rp;
}

// Aggregates of one matching pass: their number and member lists
struct Pairs {
    int n = 0;
    int *mptr = nullptr, *mem = nullptr;
};
static void pairs_free(Pairs &P, cudaStream_t s) { dfree(P.mptr, s); dfree(P.mem, s); P = Pairs(); }

// One matching pass on G; map (n) gets aggregate ids.
static Pairs match_pass(const Graph &G, double theta, int *map, cudaStream_t s) {
    const int n = G.n;
    Pairs P;
    int *mate = dmalloc<int>(n, s), *pick = dmalloc<int>(n, s);
    k_fill<int><<<grid_for(n), 256, 0, s>>>(mate, -1, n);
    NBP_LAUNCHED();
    // rounds over the whole GPU while many nodes are in play, the host looking
    // at their number every fourth round; the rest in one cluster
    int *list[2] = {nullptr, nullptr};
    int *cnt = dmalloc<int>(2 * kMatchRounds, s);   // [r]: in play after round r; [kMatchRounds + r]: made
    NBP_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * 2 * kMatchRounds, s));
    int round = 0, left = n;
    if (left > kMatchTail) {
        for (int *&q : list) q = dmalloc<int>(n, s);
        while (round < kMatchRounds && left > kMatchTail) {
            int made = left;
            for (int q = 0; q < 4; ++q, ++round) {
                const int *in = round ? list[round & 1] : nullptr, *nin = round ? cnt + round - 1 : nullptr;
                k_pick<<<grid_for((long long)left * kPickLanes, 256, 8LL * kSMs), 256, 0, s>>>(n, in, nin, G.rp, G.ci, G.w,
                                                                                           theta, mate, pick);
                k_pair<<<grid_for(left, 256, 8LL * kSMs), 256, 0, s>>>(n, in, nin, pick, mate, list[(round + 1) & 1],
                                                                       cnt + round);
                NBP_LAUNCHED();
            }
            left = readback(cnt + round - 1, s);
            if (left == made) break;   // four rounds without a pair
        }
    }
    if (left > 0 && round < kMatchRounds) {
        k_match_tail<<<kMatchCluster, kMatchThreads, 0, s>>>(n, round ? list[round & 1] : nullptr,
                                                             round ? cnt + round - 1 : nullptr, G.rp, G.ci, G.w, theta,
                                                             round, mate, pick, cnt + kMatchRounds);
        NBP_LAUNCHED();
    }
    for (int *q : list) dfree(q, s);
    dfree(cnt, s);
    unsigned long long *size = dmalloc<unsigned long long>(n + 1, s), *at = dmalloc<unsigned long long>(n + 1, s);
    k_root_size<<<grid_exact(n + 1), 256, 0, s>>>(n, mate, size);
    NBP_LAUNCHED();
    exclusive_scan(size, at, n + 1, s);
    const int nc = (int)(readback(at + n, s) >> 32);
    P.n = nc;
    P.mptr = dmalloc<int>(nc + 1, s);
    P.mem = dmalloc<int>(n, s);
    k_pair_members<<<grid_exact(n + 1), 256, 0, s>>>(n, mate, at, map, P.mptr, P.mem);
    NBP_LAUNCHED();
    dfree(mate, s); dfree(pick, s); dfree(size, s); dfree(at, s);
    return P;
}

// ---- coarse rows one per warp: coarse row I gathers its members' entries
// (members ascending, each row's entries in order: ascending fine entry
// index q), maps their columns (dropping map < 0 and, for the graph, I
// itself), sorts them in shared memory by (coarse column, q), and reduces
// each coarse column's entries in order q -- the order of the global sort's
// segments, so the results are the same bit for bit.  For coarse rows of at
// most kGroupCap entries.
constexpr int kGroupCap = 1024;
constexpr int kGroupWarps = 4;   // warps per block (shared: 8 bytes per entry)

// Entries of coarse row I into sk (key = J * kGroupCap + q, padded with ~0u
// to the sort length L, the power of two >= 32 at or above the entry count)
// and their fine entry index into se[q]; returns L, and the number of
// entries kept (dropped ones sort last) in *kept.
__device__ __forceinline__ int group_row_entries(int I, int lane, const int *mptr, const int *mem, const int *rp,
                                                 const int *ci, const int *map, int drop_diag, unsigned *sk, int *se,
                                                 int *kept) {
    const int m0 = mptr[I], nm = mptr[I + 1] - m0;
    int off = 0;
    for (int a0 = 0; a0 < nm; a0 += 32) {   // members, a lane each; their entries at off + prefix
        const int a = a0 + lane;
        const int i = a < nm ? mem[m0 + a] : 0;
        const int len = a < nm ? rp[i + 1] - rp[i] : 0;
        int incl = len;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        // the entries of these members, a lane each: entry q belongs to the last
        // member starting at or before it (its start and first entry by shuffle)
        const int total = __shfl_sync(0xffffffffu, incl, 31), begin = incl - len, e0 = a < nm ? rp[i] : 0;
        for (int p0 = 0; p0 < total; p0 += 32) {
            const int p = p0 + lane;
            int m = 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const int b = __shfl_sync(0xffffffffu, begin, m + o);
                if (b <= p) m += o;
            }
            const int e = __shfl_sync(0xffffffffu, e0, m) + p - __shfl_sync(0xffffffffu, begin, m);
            if (p < total) {
                const int q = off + p;
                const int J = map[ci[e]];
                const bool keep = J >= 0 && !(drop_diag && J == I);
                sk[q] = keep ? (((unsigned)J * (unsigned)kGroupCap) | (unsigned)q) : ~0u;
                se[q] = e;
            }
        }
        off += total;
    }
    int L = 32;
    while (L < off) L <<= 1;
    for (int q = off + lane; q < L; q += 32) sk[q] = ~0u;
    __syncwarp();
    for (int k = 2; k <= L; k <<= 1) {   // bitonic sort, ascending
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int p = lane; p < L; p += 32) {
                const int x = p ^ j;
                if (x > p) {
                    const unsigned u = sk[p], w = sk[x];
                    if ((u > w) == ((p & k) == 0)) { sk[p] = w; sk[x] = u; }
                }
            }
            __syncwarp();
        }
    }
    int c = 0;
    for (int p = lane; p < off; p += 32) c += sk[p] != ~0u ? 1 : 0;
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    *kept = c;
    return L;
}

// entries of each coarse row; a row whose members hold more than kGroupCap
// entries sets *over and is skipped
__global__ void __launch_bounds__(32 * kGroupWarps) k_group_count(int nc, const int *mptr, const int *mem, const int *rp,
                                                                 const int *ci, const int *map, int drop_diag, int *cnt,
                                                                 int *over) {
    __shared__ unsigned keys[kGroupWarps][kGroupCap];
    __shared__ int ents[kGroupWarps][kGroupCap];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int I = blockIdx.x * kGroupWarps + w;
    if (I >= nc) return;
    unsigned *sk = keys[w];
    int all = 0;
    for (int a = mptr[I] + lane; a < mptr[I + 1]; a += 32) all += rp[mem[a] + 1] - rp[mem[a]];
    for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
    if (all > kGroupCap) {
        if (lane == 0) { *over = 1; cnt[I] = 0; }
        return;
    }
    int n;
    group_row_entries(I, lane, mptr, mem, rp, ci, map, drop_diag, sk, ents[w], &n);
    int c = 0;
    for (int p = lane; p < n; p += 32) c += (p == 0 || sk[p] / kGroupCap != sk[p - 1] / kGroupCap) ? 1 : 0;
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) cnt[I] = c;
}

// MAX: the graph's edge weight, fmax over the coarse column's entries (one
// value per entry); otherwise the Galerkin block, the sum of nb (1 or 9) values
// per entry in order q.  3x3 blocks are summed by nine lanes, a component each,
// three coarse columns at a time, so that a block is read as one 72-byte
// segment.
template <bool MAX>
__global__ void __launch_bounds__(32 * kGroupWarps) k_group_fill(int nc, const int *mptr, const int *mem, const int *rp,
                                                                const int *ci, const int *map, int drop_diag, int nb,
                                                                const double *v, const int *rp_out, int *ci_out,
                                                                double *v_out) {
    __shared__ unsigned keys[kGroupWarps][kGroupCap];
    __shared__ int ents[kGroupWarps][kGroupCap];
    __shared__ unsigned short starts[MAX ? 1 : kGroupWarps][MAX ? 1 : kGroupCap];   // first position of each coarse column
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int I = blockIdx.x * kGroupWarps + w;
    if (I >= nc) return;
    unsigned *sk = keys[w];
    const int *se = ents[w];
    unsigned short *first = starts[MAX ? 0 : w];
    int n;
    const int P = group_row_entries(I, lane, mptr, mem, rp, ci, map, drop_diag, sk, ents[w], &n) / 32;
    const int p0 = lane * P;   // P contiguous positions per lane
    int mine = 0;
    for (int u = 0; u < P; ++u) {
        const int p = p0 + u;
        mine += (p < n && (p == 0 || sk[p] / kGroupCap != sk[p - 1] / kGroupCap)) ? 1 : 0;
    }
    int incl = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    long long slot = (long long)rp_out[I] + incl - mine;
    auto in_run = [&](int r, unsigned J) { return r < n && sk[r] / kGroupCap == J; };
    for (int u = 0; u < P; ++u) {
        const int p = p0 + u;
        if (!(p < n && (p == 0 || sk[p] / kGroupCap != sk[p - 1] / kGroupCap))) continue;
        const unsigned J = sk[p] / kGroupCap;
        ci_out[slot] = (int)J;
        if (!MAX && nb == 9) {
            first[slot - rp_out[I]] = (unsigned short)p;
        } else if (MAX) {
            double m = v[se[sk[p] % kGroupCap]];
            for (int r = p + 1; r < n && sk[r] / kGroupCap == J; r += 4) {   // four loads in flight
                double x[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) x[t] = in_run(r + t, J) ? v[se[sk[r + t] % kGroupCap]] : m;
#pragma unroll
                for (int t = 0; t < 4; ++t) m = fmax(m, x[t]);
            }
            v_out[slot] = m;
        } else {
            double acc = v[se[sk[p] % kGroupCap]];
            for (int r = p + 1; r < n && sk[r] / kGroupCap == J; r += 8) {   // eight loads in flight, added in order
                double x[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) x[t] = in_run(r + t, J) ? v[se[sk[r + t] % kGroupCap]] : 0.0;
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if (in_run(r + t, J)) acc = __dadd_rn(acc, x[t]);
            }
            v_out[slot] = acc;
        }
        ++slot;
    }
    if (MAX || nb != 9) return;
    __syncwarp();
    const long long o = rp_out[I];
    const int runs = rp_out[I + 1] - rp_out[I], q = lane % 9;
    if (lane >= 27) return;
    for (int r = lane / 9; r < runs; r += 3) {
        const int a = first[r], b = r + 1 < runs ? first[r + 1] : n;
        auto at = [&](int u) { return v[(long long)se[sk[u] % kGroupCap] * 9 + q]; };
        double acc = at(a);
        for (int u = a + 1; u < b; u += 4) {   // four loads in flight, added in order
            double x[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) x[t] = u + t < b ? at(u + t) : 0.0;
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (u + t < b) acc = __dadd_rn(acc, x[t]);
        }
        v_out[(o + r) * 9 + q] = acc;
    }
}

// Coarse CSR (rp, ci, values) from the per-row grouping; false, with nothing
// made, when a coarse row holds more than kGroupCap entries or the columns
// would not fit the keys
template <bool MAX>
static bool group_rows_local(int nc, const int *mptr, const int *mem, const int *rp, const int *ci, const int *map,
                             int drop_diag, int nb, const double *v, int *&rp_out, int *&ci_out, double *&v_out,
                             long long &nnz_out, cudaStream_t s) {
    if (nc <= 0 || (unsigned long long)nc * kGroupCap >= (1ULL << 32)) return false;
    const unsigned blocks = (unsigned)((nc + kGroupWarps - 1) / kGroupWarps);
    int *cnt = dmalloc<int>(nc + 1, s);
    rp_out = dmalloc<int>(nc + 2, s);   // row pointers, then the overflow flag: read back together
    NBP_CUDA(cudaMemsetAsync(cnt + nc, 0, sizeof(int), s));
    NBP_CUDA(cudaMemsetAsync(rp_out + nc + 1, 0, sizeof(int), s));
    k_group_count<<<blocks, 32 * kGroupWarps, 0, s>>>(nc, mptr, mem, rp, ci, map, drop_diag, cnt, rp_out + nc + 1);
    NBP_LAUNCHED();
    exclusive_scan(cnt, rp_out, nc + 1, s);
    dfree(cnt, s);
    int end[2];
    NBP_CUDA(cudaMemcpyAsync(end, rp_out + nc, sizeof(end), cudaMemcpyDeviceToHost, s));
    NBP_CUDA(cudaStreamSynchronize(s));
    if (end[1]) {
        dfree(rp_out, s);
        rp_out = nullptr;
        return false;
    }
    nnz_out = end[0];
    ci_out = dmalloc<int>(nnz_out > 0 ? nnz_out : 1, s);
    v_out = dmalloc<double>((nnz_out > 0 ? nnz_out : 1) * nb, s);
    k_group_fill<MAX><<<blocks, 32 * kGroupWarps, 0, s>>>(nc, mptr, mem, rp, ci, map, drop_diag, nb, v, rp_out, ci_out,
                                                          v_out);
    NBP_LAUNCHED();
    return true;
}

static Graph coarse_graph(const Graph &G, const int *map, const Pairs &P, cudaStream_t s) {
    const int nc = P.n;
    Graph Gc;
    Gc.n = nc;
    if (group_rows_local<true>(nc, P.mptr, P.mem, G.rp, G.ci, map, 1, 1, G.w, Gc.rp, Gc.ci, Gc.w, Gc.nnz, s)) return Gc;
    Segments sg = group_by_coarse(G.n, G.nnz, G.rp, G.ci, map, nc, 1, s);
    Gc.nnz = sg.nseg;
    Gc.rp = rowptr_from_segments(sg, nc, s);
    Gc.ci = dmalloc<int>(sg.nseg, s);
    Gc.w = dmalloc<double>(sg.nseg, s);
    if (sg.nseg > 0) {
        k_cg_fill<<<grid_exact(sg.nseg), 256, 0, s>>>(sg.nseg, sg.key, sg.start, sg.nvalid, sg.idx, G.w, (unsigned long long)nc,
                                                      Gc.ci, Gc.w);
        NBP_LAUNCHED();
    }
    free_segments(sg, s);
    return Gc;
}

// The members of every final aggregate, from the passes' pair lists: up to two
// nodes a pass, so up to eight, sorted; isolated nodes left out.  cnt: their
// number per kept aggregate (fill: at mptr[newid], and the map of the nodes)
__device__ __forceinline__ int expand_members(int I, const Pairs &a, const Pairs &b, const Pairs &c, const int *iso,
                                              int (&out)[8]) {
    int k = 0;
    for (int p = c.mptr[I]; p < c.mptr[I + 1]; ++p)
        for (int q = b.mptr[c.mem[p]]; q < b.mptr[c.mem[p] + 1]; ++q)
            for (int r = a.mptr[b.mem[q]]; r < a.mptr[b.mem[q] + 1]; ++r)
                if (!iso[a.mem[r]] && k < 8) out[k++] = a.mem[r];
    return k;
}
// v[I] = (1 if the aggregate holds a node, members), packed for one scan
__global__ void k_final_size(int nc, Pairs a, Pairs b, Pairs c, const int *iso, unsigned long long *v) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I > nc) return;
    int m[8];
    const int k = I < nc ? expand_members(I, a, b, c, iso, m) : 0;
    v[I] = k > 0 ? (1ULL << 32) | (unsigned long long)k : 0ULL;
}
__global__ void k_final_members(int nc, Pairs a, Pairs b, Pairs c, const int *iso, const unsigned long long *at, int *agg,
                                int *mptr, int *mem) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I > nc) return;
    const unsigned long long v = at[I];
    const int J = (int)(v >> 32), p = (int)(v & 0xffffffffULL);
    if (I == nc) { mptr[J] = p; return; }
    int m[8];
    const int k = expand_members(I, a, b, c, iso, m);
    if (k == 0) return;
    for (int i = 1; i < k; ++i)   // ascending
        for (int j = i; j > 0 && m[j - 1] > m[j]; --j) {
            const int t = m[j];
            m[j] = m[j - 1];
            m[j - 1] = t;
        }
    mptr[J] = p;
    for (int i = 0; i < k; ++i) {
        mem[p + i] = m[i];
        agg[m[i]] = J;
    }
}

// 3 passes; agg (n) gets the final map (-1 = isolated) and mptr / mem the
// aggregates' member lists (ascending fine index); returns the aggregate count
static int aggregate(const DMat &M, double theta, int *agg, int *&mptr, int *&mem, cudaStream_t s) {
    const int n = M.nbr, nb = M.bb();
    double *dn = dmalloc<double>(n, s);
    k_diag_norm<<<grid_exact(n), 256, 0, s>>>(n, nb, M.rp, M.ci, M.v, dn);
    NBP_LAUNCHED();
    Graph G;
    G.n = n; G.nnz = M.nnz; G.rp = M.rp; G.ci = M.ci;
    G.w = dmalloc<double>(M.nnz, s);
    k_strength<<<grid_exact((long long)n * kStrengthLanes), 256, 0, s>>>(n, nb, M.rp, M.ci, M.v, dn, G.w);
    NBP_LAUNCHED();
    int *iso = dmalloc<int>(n, s);
    k_isolated<<<grid_exact(n), 256, 0, s>>>(n, M.rp, M.ci, G.w, theta, iso);
    NBP_LAUNCHED();
    dfree(dn, s);
    int *map = dmalloc<int>(n, s);
    bool own = false;   // the first graph borrows the matrix pattern
    Pairs P[3];
    for (int pass = 0; pass < 3; ++pass) {
        P[pass] = match_pass(G, theta, map, s);
        if (pass < 2) {   // the last pass needs no graph of its aggregates
            Graph Gc = coarse_graph(G, map, P[pass], s);
            if (own) graph_free(G, s);
            else dfree(G.w, s);
            G = Gc;
            own = true;
        }
    }
    graph_free(G, s);
    dfree(map, s);
    const int nc = P[2].n;
    unsigned long long *size = dmalloc<unsigned long long>(nc + 1, s), *at = dmalloc<unsigned long long>(nc + 1, s);
    k_final_size<<<grid_exact(nc + 1), 256, 0, s>>>(nc, P[0], P[1], P[2], iso, size);
    NBP_LAUNCHED();
    exclusive_scan(size, at, nc + 1, s);
    k_fill<int><<<grid_for(n), 256, 0, s>>>(agg, -1, n);
    mptr = dmalloc<int>(nc + 1, s);   // nc is at least the number of kept aggregates
    mem = dmalloc<int>(n, s);
    k_final_members<<<grid_exact(nc + 1), 256, 0, s>>>(nc, P[0], P[1], P[2], iso, at, agg, mptr, mem);
    NBP_LAUNCHED();
    const int m = (int)(readback(at + nc, s) >> 32);
    for (Pairs &p : P) pairs_free(p, s);
    dfree(size, s); dfree(at, s); dfree(iso, s);
    return m;
}

// mptr/mem: the aggregates' member lists (ascending fine index)
static void galerkin(const DMat &M, const int *agg, const int *mptr, const int *mem, int nc, DMat &Mc, cudaStream_t s) {
    Mc = DMat();
    Mc.nbr = nc; Mc.nbc = nc; Mc.br = M.br; Mc.bc = M.bc;
    long long nnz = 0;
    if (group_rows_local<false>(nc, mptr, mem, M.rp, M.ci, agg, 0, M.bb(), M.v, Mc.rp, Mc.ci, Mc.v, nnz, s)) {
        Mc.nnz = nnz;
        return;
    }
    Segments sg = group_by_coarse(M.nbr, M.nnz, M.rp, M.ci, agg, nc, 0, s);
    Mc.nnz = sg.nseg;
    Mc.rp = rowptr_from_segments(sg, nc, s);
    Mc.ci = dmalloc<int>(sg.nseg, s);
    Mc.v = dmalloc<double>((long long)sg.nseg * M.bb(), s);
    if (sg.nseg > 0) {
        k_galerkin_fill<<<grid_exact(sg.nseg), 256, 0, s>>>(sg.nseg, M.bb(), sg.key, sg.start, sg.nvalid, sg.idx, M.v,
                                                            (unsigned long long)nc, Mc.ci, Mc.v);
        NBP_LAUNCHED();
    }
    free_segments(sg, s);
}

// ---- A P, one row per warp: the row's entries in chunks of 32, each chunk's
// coarse columns looked up in the row's list (first occurrence order), new ones
// appended, and the blocks summed per column in entry order.  Rows with more
// than kApCap coarse columns have no A P (the level keeps the prolongation and
// the full product).
constexpr int kApCap = 64, kApWarps = 8;

// list position of this lane's coarse column J (-1: dropped), the list and its
// length updated; *over is set when the list is full
__device__ __forceinline__ int ap_position(int J, int lane, int *list, int &len, bool *over) {
    int pos = -1;
    for (int t = 0; t < len; ++t)
        if (list[t] == J) pos = t;
    if (J < 0) pos = -1;
    const bool fresh = J >= 0 && pos < 0;
    const unsigned same = __match_any_sync(0xffffffffu, fresh ? J : -1 - lane);
    const bool lead = fresh && (__ffs(same) - 1) == lane;
    const unsigned leads = __ballot_sync(0xffffffffu, lead);
    int at = len + __popc(leads & ((1u << lane) - 1u));
    at = __shfl_sync(0xffffffffu, at, __ffs(same) - 1);
    len += __popc(leads);
    if (len > kApCap) { *over = true; len = kApCap; }
    if (lead && at < kApCap) list[at] = J;
    __syncwarp();
    if (fresh) pos = at < kApCap ? at : -1;
    return pos;
}
__global__ void __launch_bounds__(32 * kApWarps) k_ap_count(int n, const int *rp, const int *ci, const int *agg, int *cnt,
                                                           int *over) {
    __shared__ int lists[kApWarps][kApCap];
    const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kApWarps + wp;
    if (i >= n) return;
    int len = 0;
    bool full = false;
    const int e1 = rp[i + 1];
    for (int e0 = rp[i]; e0 < e1; e0 += 32) {
        const int e = e0 + lane;
        ap_position(e < e1 ? agg[ci[e]] : -1, lane, lists[wp], len, &full);
    }
    if (lane == 0) {
        cnt[i] = len;
        if (full) *over = 1;
    }
}
template <int NB>
__global__ void __launch_bounds__(32 * kApWarps) k_ap_fill(int n, const int *rp, const int *ci, const double *v,
                                                          const int *agg, const int *rp_out, int *ci_out, double *v_out) {
    __shared__ int lists[kApWarps][kApCap];
    __shared__ double sums[kApWarps][kApCap * NB];
    const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kApWarps + wp;
    if (i >= n) return;
    double *acc = sums[wp];
    for (int q = lane; q < kApCap * NB; q += 32) acc[q] = 0.0;
    __syncwarp();
    int len = 0;
    bool full = false;
    const int e1 = rp[i + 1];
    for (int e0 = rp[i]; e0 < e1; e0 += 32) {
        const int e = e0 + lane;
        const int pos = ap_position(e < e1 ? agg[ci[e]] : -1, lane, lists[wp], len, &full);
        unsigned same = __match_any_sync(0xffffffffu, pos >= 0 ? pos : -1 - lane);
        if (pos >= 0 && (__ffs(same) - 1) == lane) {   // the column's first lane adds its blocks in entry order
            double a[NB];
#pragma unroll
            for (int q = 0; q < NB; ++q) a[q] = acc[pos * NB + q];
            while (same) {
                const double *src = v + (long long)(e0 + __ffs(same) - 1) * NB;
                same &= same - 1;
#pragma unroll
                for (int q = 0; q < NB; ++q) a[q] += src[q];
            }
#pragma unroll
            for (int q = 0; q < NB; ++q) acc[pos * NB + q] = a[q];
        }
        __syncwarp();
    }
    const int o = rp_out[i];
    for (int t = lane; t < len; t += 32) ci_out[o + t] = lists[wp][t];
    for (int q = lane; q < len * NB; q += 32) v_out[(long long)o * NB + q] = acc[q];
}

// A P of a level with an aggregate map, in the sliced copies that the solves
// use (the CSR arrays are dropped)
static void make_ap(Level &L, int nc, int precision, cudaStream_t s) {
    const DMat &M = L.M;
    const int n = M.nbr;
    if (n == 0 || nc == 0 || (M.bb() != 9 && M.bb() != 1)) return;
    const unsigned blocks = (unsigned)((n + kApWarps - 1) / kApWarps);
    int *cnt = dmalloc<int>(n + 2, s);   // rows, 0, overflow flag
    NBP_CUDA(cudaMemsetAsync(cnt + n, 0, 2 * sizeof(int), s));
    k_ap_count<<<blocks, 32 * kApWarps, 0, s>>>(n, M.rp, M.ci, L.agg, cnt, cnt + n + 1);
    NBP_LAUNCHED();
    DMat P;
    P.nbr = n; P.nbc = nc; P.br = M.br; P.bc = M.bc;
    P.rp = dmalloc<int>(n + 2, s);
    exclusive_scan(cnt, P.rp, n + 1, s);
    NBP_CUDA(cudaMemcpyAsync(P.rp + n + 1, cnt + n + 1, sizeof(int), cudaMemcpyDeviceToDevice, s));
    int end[2];
    NBP_CUDA(cudaMemcpyAsync(end, P.rp + n, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
    NBP_CUDA(cudaStreamSynchronize(s));
    dfree(cnt, s);
    P.nnz = end[0];
    if (end[1] || P.nnz == 0) { dmat_free(P, s); return; }
    P.ci = dmalloc<int>(P.nnz, s);
    P.v = dmalloc<double>(P.nnz * P.bb(), s);
    if (P.bb() == 9) k_ap_fill<9><<<blocks, 32 * kApWarps, 0, s>>>(n, M.rp, M.ci, M.v, L.agg, P.rp, P.ci, P.v);
    else k_ap_fill<1><<<blocks, 32 * kApWarps, 0, s>>>(n, M.rp, M.ci, M.v, L.agg, P.rp, P.ci, P.v);
    NBP_LAUNCHED();
    make_sell(P, precision, s);
    dfree(P.rp, s); dfree(P.ci, s); dfree(P.v, s);
    P.rp = nullptr; P.ci = nullptr; P.v = nullptr;
    L.AP = P;
}

// The inverse of the coarsest matrix, a chain of small kernels: queued on a
// stream of its own (side), beside the levels' smoothing data and sliced
// copies that s makes, and taken up by finish().  Setups, with the spectral
// estimates queued level by level: cube of 16 7.4 -> 7.0 ms, 0.56M unknowns
// numeric 13.2 -> 12.1, 1.85M 46.0 -> 44.2.
struct DenseInverse {
    cudaStream_t s = nullptr, side = nullptr;
    cudaEvent_t ev = nullptr;
    double *Dm = nullptr, *Dn = nullptr, *G = nullptr;   // Dn: the inverse
    int *piv = nullptr, *perm = nullptr, *fail = nullptr;
    DenseInverse(cudaStream_t s_, cudaStream_t side_) : s(s_), side(side_) {}
    void queue(const DMat &M) {
        NBP_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        NBP_CUDA(cudaEventRecord(ev, s));
        NBP_CUDA(cudaStreamWaitEvent(side, ev, 0));
        const int n = M.nbr * M.br;
        Dm = dmalloc<double>((long long)n * n, side);
        Dn = dmalloc<double>((long long)n * n, side);
        NBP_CUDA(cudaMemsetAsync(Dm, 0, sizeof(double) * (size_t)n * n, side));
        k_dense_from_bsr<<<grid_exact(M.nbr), 256, 0, side>>>(M.nbr, M.br, M.rp, M.ci, M.v, Dm);
        NBP_LAUNCHED();
        G = dmalloc<double>(8LL * n, side);
        piv = dmalloc<int>(n, side);
        perm = dmalloc<int>(n, side);
        fail = dmalloc<int>(1, side);
        NBP_CUDA(cudaMemsetAsync(fail, 0, sizeof(int), side));
        k_iota<<<grid_exact(n), 256, 0, side>>>(n, perm);
        NBP_LAUNCHED();
        // panel width: b columns and the permutation in one block's shared memory
        const int B = n <= 3300 ? 8 : 4;
        static_assert((4 * sizeof(double) + sizeof(int)) * (size_t)kCoarseDenseMax <= 227u * 1024u, "panel fits");
        const size_t smem = ((size_t)B * sizeof(double) + sizeof(int)) * (size_t)n;
        NBP_CUDA(cudaFuncSetAttribute(k_inv_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024));
        const dim3 tiles((n + 31) / 32, (n + 31) / 32);
        for (int k0 = 0; k0 < n; k0 += B) {   // Dm and Dn in turn
            const int b = std::min(B, n - k0);
            k_inv_panel<<<1, kInvThreads, smem, side>>>(n, k0, b, Dm, G, piv, perm, fail);
            k_inv_update<<<tiles, 256, 0, side>>>(n, k0, b, Dm, G, piv, Dn, fail);
            std::swap(Dm, Dn);
        }
        k_inv_columns<<<grid_exact((long long)n * n), 256, 0, side>>>(n, Dm, perm, Dn);
        NBP_LAUNCHED();
    }
    bool join() {   // s goes on after side
        return cudaEventRecord(ev, side) == cudaSuccess && cudaStreamWaitEvent(s, ev, 0) == cudaSuccess;
    }
    double *finish() {
        require(join(), NBP_ERR_CUDA, "setup: the coarsest inverse's stream could not be joined");
        require(readback(fail, s) == 0, NBP_ERR_INVALID, "setup: coarsest AMG matrix is singular");
        double *inv = Dn;
        Dn = nullptr;
        return inv;
    }
    ~DenseInverse() {   // also where a setup ends with an error: side reads the hierarchy
        if (!ev) return;
        if (!join()) cudaStreamSynchronize(side);
        cudaEventDestroy(ev);
        dfree(fail, s); dfree(Dm, s); dfree(Dn, s); dfree(G, s); dfree(piv, s); dfree(perm, s);
    }
};

void amg_build(Hier &H, const DMat &fine, const nbp_options &o, int precision, cudaStream_t s, bool keep_aggregates,
               cudaStream_t side, const std::function<void(int)> &level_ready) {
    // numeric re-setup: the aggregate maps and member lists of the hierarchy
    // H holds are taken over (same pattern); every operator is rebuilt
    int knlev = 0, knc[kMaxLevels] = {};
    int *kagg[kMaxLevels] = {}, *kmptr[kMaxLevels] = {}, *kmem[kMaxLevels] = {};
    if (keep_aggregates) {
        require(H.built && H.nlev >= 1 && H.L[0].M.nbr == fine.nbr && H.L[0].M.nnz == fine.nnz && H.bs == fine.br,
                NBP_ERR_STATE, "setup: no earlier hierarchy of this pattern to build on");
        knlev = H.nlev;
        for (int l = 0; l + 1 < knlev; ++l) {
            kagg[l] = H.L[l].agg; kmptr[l] = H.L[l].mptr; kmem[l] = H.L[l].mem;
            knc[l] = H.L[l + 1].M.nbr;
            H.L[l].agg = nullptr; H.L[l].mptr = nullptr; H.L[l].mem = nullptr;
        }
    }
    auto drop_kept = [&](int from) {
        for (int l = from; l + 1 < knlev; ++l) { dfree(kagg[l], s); dfree(kmptr[l], s); dfree(kmem[l], s); }
    };
    int l = 0;
    try {
        hier_free(H, s);
        H.bs = fine.br;
        // level 0 is a private copy of the fine matrix pattern and values
        DMat &F = H.L[0].M;
        F.nbr = fine.nbr; F.nbc = fine.nbc; F.br = fine.br; F.bc = fine.bc; F.nnz = fine.nnz;
        F.rp = dmalloc<int>(F.nbr + 1, s);
        F.ci = dmalloc<int>(F.nnz, s);
        F.v = dmalloc<double>(F.nnz * F.bb(), s);
        NBP_CUDA(cudaMemcpyAsync(F.rp, fine.rp, sizeof(int) * (F.nbr + 1), cudaMemcpyDeviceToDevice, s));
        NBP_CUDA(cudaMemcpyAsync(F.ci, fine.ci, sizeof(int) * F.nnz, cudaMemcpyDeviceToDevice, s));
        NBP_CUDA(cudaMemcpyAsync(F.v, fine.v, sizeof(double) * F.nnz * F.bb(), cudaMemcpyDeviceToDevice, s));
        const int maxlev = std::max(1, std::min((int)o.amg_max_levels, kMaxLevels));
        while (keep_aggregates ? l + 1 < knlev : (H.L[l].M.nbr > o.amg_coarse_max && l + 1 < maxlev)) {
            Level &L = H.L[l];
            const int n = L.M.nbr;
            int nc;
            if (keep_aggregates) {   // the kept map, now owned by this level
                L.agg = kagg[l]; L.mptr = kmptr[l]; L.mem = kmem[l];
                kagg[l] = kmptr[l] = kmem[l] = nullptr;
                nc = knc[l];
            } else {
                L.agg = dmalloc<int>(n, s);
                nc = aggregate(L.M, o.theta, L.agg, L.mptr, L.mem, s);
                if (nc >= n || nc == 0) {
                    dfree(L.agg, s); dfree(L.mptr, s); dfree(L.mem, s);
                    L.agg = nullptr; L.mptr = nullptr; L.mem = nullptr;
                    break;
                }
            }
            galerkin(L.M, L.agg, L.mptr, L.mem, nc, H.L[l + 1].M, s);
            ++l;
        }
    } catch (...) {
        drop_kept(0);
        throw;
    }
    H.nlev = l + 1;
    const Level &C = H.L[H.nlev - 1];
    const bool dense = (long long)C.M.nbr * H.bs <= kCoarseDenseMax;
    DenseInverse inverse(s, side);
    if (dense) inverse.queue(C.M);
    int *singular = dmalloc<int>(1, s);
    NBP_CUDA(cudaMemsetAsync(singular, 0, sizeof(int), s));
    unsigned long long *rb = dmalloc<unsigned long long>(1, s);
    for (int k = 0; k < H.nlev; ++k) {
        Level &L = H.L[k];
        const int n = L.M.nbr, bs = H.bs;
        const long long nv = (long long)n * bs;
        const size_t v64 = ((size_t)nv * 8 + 255) / 256 * 256, v32 = ((size_t)nv * 4 + 255) / 256 * 256;
        L.work = dmalloc<char>(Level::kWork * (v64 + v32), s);
        for (int q = 0; q < Level::kWork; ++q) {
            L.w64[q] = reinterpret_cast<double *>(L.work + q * v64);
            L.w32[q] = reinterpret_cast<float *>(L.work + Level::kWork * v64 + q * v32);
        }
        L.kdots = dmalloc<double>(8 + 4 * kKdotBlocks, s);
        NBP_CUDA(cudaMemsetAsync(L.kdots, 0, sizeof(double) * (8 + 4 * kKdotBlocks), s));
        {   // every level, the coarsest included (it is smoothed when too large for a dense solve)
            L.dinv = dmalloc<double>(nv * bs, s);
            k_block_dinv<<<grid_exact(n), 256, 0, s>>>(n, bs, L.M.rp, L.M.ci, L.M.v, L.dinv, singular);
            NBP_CUDA(cudaMemsetAsync(rb, 0, sizeof(unsigned long long), s));
            k_gershgorin<<<grid_exact(n), 256, 0, s>>>(n, bs, L.M.rp, L.M.v, L.dinv, rb);
            NBP_LAUNCHED();
            const unsigned long long bits = readback(rb, s);
            std::memcpy(&L.rho, &bits, sizeof(double));
            if (precision >= 1) {
                L.dinv32 = dmalloc<float>(nv * bs, s);
                k_to_f32<<<grid_for(nv * bs), 256, 0, s>>>(L.dinv, L.dinv32, nv * bs);
                NBP_LAUNCHED();
            }
            make_lowcopies(L.M, precision, s);
            make_sell(L.M, precision, s);
            if (k + 1 < H.nlev) make_ap(L, H.L[k + 1].M.nbr, precision, s);
            if (L.M.sl_ci) {   // grids of the sliced kernels, up to 8 threads per row
                L.kpart_blocks = ((long long)L.M.nslice * L.M.sl_c * 8 + 255) / 256;
                L.kpart = dmalloc<double>(4 * L.kpart_blocks, s);
            }
            if (level_ready) level_ready(k);
        }
    }
    dfree(rb, s);
    const int sing = readback(singular, s);
    dfree(singular, s);
    require(sing == 0, NBP_ERR_INVALID, "setup: singular diagonal block in an AMG level");
    if (dense) {
        H.cinv = inverse.finish();
        H.nc = C.M.nbr * H.bs;
        const long long nn = (long long)H.nc * H.nc;
        H.cinv32 = dmalloc<float>(nn, s);
        k_to_f32<<<grid_for(nn), 256, 0, s>>>(H.cinv, H.cinv32, nn);
        NBP_LAUNCHED();
    } else { H.cinv = nullptr; H.nc = 0; }
    H.built = true;
}

// ================================================================== S_hat
__global__ void k_diagA(int N, const int *rp, const int *ci, const double *v, double *diag) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int e = find_entry(rp, ci, i, i);
    for (int a = 0; a < 3; ++a) diag[3 * i + a] = (e >= 0) ? v[(long long)e * 9 + 4 * a] : 0.0;
}
// diag[idx] += r_k (a*a) for outlet k (one launch per outlet: k ascending)
__global__ void k_diagA_lowrank(int beg, int end, const int *oidx, const double *oval, const double *r, int k, double *diag) {
    const int q = beg + blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= end) return;
    const double a = oval[q];
    diag[oidx[q]] = __dadd_rn(diag[oidx[q]], __dmul_rn(r[k], __dmul_rn(a, a)));
}
__global__ void k_recip(long long n, const double *a, double *b) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = 1.0 / a[i];
}
// tuples per row of S_hat: D entries, then C_ik B_kj terms (k ascending, j ascending)
__global__ void k_shat_count(int N, const int *drp, const int *crp, const int *cci, const int *brp, long long *cnt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    long long c = drp[i + 1] - drp[i];
    for (int e = crp[i]; e < crp[i + 1]; ++e) {
        const int k = cci[e];
        c += brp[k + 1] - brp[k];
    }
    cnt[i] = c;
}
__global__ void k_shat_fill(int N, const int *drp, const int *dci, const int *crp, const int *cci, const double *cv,
                            const int *brp, const int *bci, const double *bv, const double *dinv, const long long *off,
                            unsigned long long *key, double *t) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    long long p = off[i];
    for (int e = drp[i]; e < drp[i + 1]; ++e) {
        key[p] = (unsigned long long)i * (unsigned long long)N + (unsigned long long)dci[e];
        t[p++] = 0.0;
    }
    for (int e = crp[i]; e < crp[i + 1]; ++e) {
        const int k = cci[e];
        const double w0 = __dmul_rn(cv[3LL * e], dinv[3LL * k]);
        const double w1 = __dmul_rn(cv[3LL * e + 1], dinv[3LL * k + 1]);
        const double w2 = __dmul_rn(cv[3LL * e + 2], dinv[3LL * k + 2]);
        for (int f = brp[k]; f < brp[k + 1]; ++f) {
            double tt = __dmul_rn(w0, bv[3LL * f]);
            tt = __dadd_rn(tt, __dmul_rn(w1, bv[3LL * f + 1]));
            tt = __dadd_rn(tt, __dmul_rn(w2, bv[3LL * f + 2]));
            key[p] = (unsigned long long)i * (unsigned long long)N + (unsigned long long)bci[f];
            t[p++] = tt;
        }
    }
}
__global__ void k_heads_all(long long n, const unsigned long long *key, int *head) {
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    head[q] = (q == 0 || key[q - 1] != key[q]) ? 1 : 0;
}
// entry (i, j): s = D_ij (or 0), then s = s - t for each tuple in order
__global__ void k_shat_reduce(int nseg, long long ntup, const unsigned long long *key, const long long *start, const double *t,
                              int N, const int *drp, const int *dci, const double *dv, int *ci_out, double *v_out,
                              int *rowcnt) {
    const int sg = blockIdx.x * blockDim.x + threadIdx.x;
    if (sg >= nseg) return;
    const long long a = start[sg];
    const long long b = (sg + 1 < nseg) ? start[sg + 1] : ntup;
    const unsigned long long k = key[a];
    const int i = (int)(k / (unsigned long long)N), j = (int)(k % (unsigned long long)N);
    const int e = find_entry(drp, dci, i, j);
    double s = (e >= 0) ? dv[e] : 0.0;
    for (long long q = a; q < b; ++q) s = __dsub_rn(s, t[q]);
    ci_out[sg] = j;
    v_out[sg] = s;
    atomicAdd(rowcnt + i, 1);
}

// ---- S_hat one row per warp, for rows of at most kShatRowTuples tuples: the
// row's distinct columns (D's and those of the B rows that C's row meets) are
// collected in a hash table in shared memory and sorted; then the terms
// C_ik B_kj are subtracted from D_ij entry by entry of C's row (k ascending),
// a lane per entry of B's row k, which are distinct columns: every entry of
// S_hat takes its terms in the order that k_shat_fill numbers them and
// k_shat_reduce sums them, without sorting the terms themselves (0.56M
// unknowns, count + fill: 1.93 -> 1.00 ms).
constexpr int kShatRowTuples = 256;
constexpr int kShatTable = 512;   // hash slots: at most half full
constexpr int kShatWarps = 8;     // warps per block

// this lane's column j (< 0: none) into the table; true where it is new
__device__ __forceinline__ bool shat_insert(int *table, int j) {
    if (j < 0) return false;
    unsigned h = ((unsigned)j * 2654435761u) >> 23;   // 9 bits
    for (int t = 0; t < kShatTable; ++t, h = (h + 1) & (kShatTable - 1)) {
        const int old = atomicCAS(table + h, -1, j);
        if (old == -1) return true;
        if (old == j) return false;
    }
    return false;
}
// the distinct columns of row i into the table (cleared first); their number
__device__ __forceinline__ int shat_columns(int i, int lane, const int *drp, const int *dci, const int *crp, const int *cci,
                                            const int *brp, const int *bci, int *table) {
    for (int q = lane; q < kShatTable; q += 32) table[q] = -1;
    __syncwarp();
    int c = 0;
    for (int q = drp[i] + lane; q < drp[i + 1]; q += 32) c += shat_insert(table, dci[q]) ? 1 : 0;
    for (int e = crp[i]; e < crp[i + 1]; ++e) {
        const int k = cci[e], b1 = brp[k + 1];
        for (int f = brp[k] + lane; f < b1; f += 32) c += shat_insert(table, bci[f]) ? 1 : 0;
    }
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    __syncwarp();
    return c;
}

// entries per row (distinct columns)
__global__ void __launch_bounds__(32 * kShatWarps) k_shat_row_count(int N, const int *drp, const int *dci, const int *crp,
                                                                   const int *cci, const int *brp, const int *bci, int *cnt) {
    __shared__ int tables[kShatWarps][kShatTable];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kShatWarps + w;
    if (i >= N) return;
    const int n = shat_columns(i, lane, drp, dci, crp, cci, brp, bci, tables[w]);
    if (lane == 0) cnt[i] = n;
}

// the row's entries at rp_out[i]..: columns ascending, each D_ij (or 0)
// minus its terms in order
__global__ void __launch_bounds__(32 * kShatWarps) k_shat_row_fill(int N, const int *drp, const int *dci, const double *dv,
                                                                  const int *crp, const int *cci, const double *cv,
                                                                  const int *brp, const int *bci, const double *bv,
                                                                  const double *dinv, const int *rp_out, int *ci_out,
                                                                  double *v_out) {
    __shared__ int tables[kShatWarps][kShatTable];
    __shared__ int cols[kShatWarps][kShatRowTuples];
    __shared__ double sums[kShatWarps][kShatRowTuples];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kShatWarps + w;
    if (i >= N) return;
    int *table = tables[w], *col = cols[w];
    double *sum = sums[w];
    const int n = shat_columns(i, lane, drp, dci, crp, cci, brp, bci, table);
    int at = 0;   // the table's columns packed, then sorted (bitonic, padded to a power of two)
    for (int q = lane; q < kShatTable; q += 32) {
        const int j = table[q];
        const unsigned m = __ballot_sync(0xffffffffu, j >= 0);
        if (j >= 0) col[at + __popc(m & ((1u << lane) - 1u))] = j;
        at += __popc(m);
    }
    int L = 32;
    while (L < n) L <<= 1;
    for (int q = n + lane; q < L; q += 32) col[q] = 0x7fffffff;
    __syncwarp();
    for (int k = 2; k <= L; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int p = lane; p < L; p += 32) {
                const int x = p ^ j;
                if (x > p) {
                    const int a = col[p], b = col[x];
                    if ((a > b) == ((p & k) == 0)) { col[p] = b; col[x] = a; }
                }
            }
            __syncwarp();
        }
    auto find = [&](int j) {   // j is in the list
        int lo = 0, hi = n - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (col[mid] < j) lo = mid + 1; else hi = mid;
        }
        return lo;
    };
    for (int q = lane; q < n; q += 32) sum[q] = 0.0;
    __syncwarp();
    for (int q = drp[i] + lane; q < drp[i + 1]; q += 32) {
        const int u = find(dci[q]);
        sum[u] = __dsub_rn(dv[q], 0.0);   // D_ij minus its placeholder term
    }
    __syncwarp();
    // two entries of C's row at a time, half a warp each, where B's rows fit (an
    // FP64 operation holds the pipe for a warp whatever lanes it has): the
    // terms together, then the first entry's subtracted before the second's
    const int c1 = crp[i + 1], half = lane >> 4;
    auto term = [&](int e, int k, int f) {
        const double w0 = __dmul_rn(cv[3LL * e], dinv[3LL * k]);
        const double w1 = __dmul_rn(cv[3LL * e + 1], dinv[3LL * k + 1]);
        const double w2 = __dmul_rn(cv[3LL * e + 2], dinv[3LL * k + 2]);
        double tt = __dmul_rn(w0, bv[3LL * f]);
        tt = __dadd_rn(tt, __dmul_rn(w1, bv[3LL * f + 1]));
        return __dadd_rn(tt, __dmul_rn(w2, bv[3LL * f + 2]));
    };
    for (int e0 = crp[i]; e0 < c1; e0 += 2) {
        const int e = e0 + half;
        const int k = e < c1 ? cci[e] : 0;
        const int b0 = e < c1 ? brp[k] : 0, len = e < c1 ? brp[k + 1] - b0 : 0;
        if (__all_sync(0xffffffffu, len <= 16)) {
            const bool on = (lane & 15) < len;
            const int f = b0 + (lane & 15);
            int u = 0;
            double tt = 0.0;
            if (on) {
                tt = term(e, k, f);
                u = find(bci[f]);
            }
            if (on && half == 0) sum[u] = __dsub_rn(sum[u], tt);
            __syncwarp();
            if (on && half == 1) sum[u] = __dsub_rn(sum[u], tt);
            __syncwarp();
            continue;
        }
        for (int e2 = e0; e2 < min(c1, e0 + 2); ++e2) {
            const int k2 = cci[e2], b1 = brp[k2 + 1];
            for (int f = brp[k2] + lane; f < b1; f += 32) {
                const double tt = term(e2, k2, f);
                const int u = find(bci[f]);
                sum[u] = __dsub_rn(sum[u], tt);
            }
            __syncwarp();
        }
    }
    const int o = rp_out[i];
    for (int q = lane; q < n; q += 32) {
        ci_out[o + q] = col[q];
        v_out[o + q] = sum[q];
    }
}

__global__ void k_max_ll(long long n, const long long *a, unsigned long long *out) {
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q < n) atomicMax(out, (unsigned long long)a[q]);
}

void build_shat(const DMat &A, const DMat &B, const DMat &C, const DMat &D, const LowRank &lr, int N, DMat &S,
                double *diagA_out, cudaStream_t s) {
    double *diag = diagA_out;
    k_diagA<<<grid_exact(N), 256, 0, s>>>(N, A.rp, A.ci, A.v, diag);
    NBP_LAUNCHED();
    for (int k = 0; k < lr.n_out; ++k) {
        int se[2];
        NBP_CUDA(cudaMemcpyAsync(se, lr.optr + k, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
        NBP_CUDA(cudaStreamSynchronize(s));
        if (se[1] > se[0]) {
            k_diagA_lowrank<<<grid_exact(se[1] - se[0]), 256, 0, s>>>(se[0], se[1], lr.oidx, lr.oval, lr.r, k, diag);
            NBP_LAUNCHED();
        }
    }
    double *dinv = dmalloc<double>(3LL * N, s);
    k_recip<<<grid_exact(3LL * N), 256, 0, s>>>(3LL * N, diag, dinv);
    long long *cnt = dmalloc<long long>(N + 1, s), *off = dmalloc<long long>(N + 1, s);
    k_shat_count<<<grid_exact(N), 256, 0, s>>>(N, D.rp, C.rp, C.ci, B.rp, cnt);
    NBP_LAUNCHED();
    {   // every row within one warp's sort: the per-row build, no global sort
        unsigned long long *mx = dmalloc<unsigned long long>(1, s);
        NBP_CUDA(cudaMemsetAsync(mx, 0, sizeof(unsigned long long), s));
        k_max_ll<<<grid_exact(N), 256, 0, s>>>(N, cnt, mx);
        NBP_LAUNCHED();
        const unsigned long long maxtup = readback(mx, s);
        dfree(mx, s);
        if (maxtup <= (unsigned long long)kShatRowTuples && N < (1 << 24)) {
            dfree(cnt, s); dfree(off, s);
            int *rowcnt = dmalloc<int>(N + 1, s);
            const unsigned blocks = (unsigned)((N + kShatWarps - 1) / kShatWarps);
            k_shat_row_count<<<blocks, 32 * kShatWarps, 0, s>>>(N, D.rp, D.ci, C.rp, C.ci, B.rp, B.ci, rowcnt);
            NBP_LAUNCHED();
            NBP_CUDA(cudaMemsetAsync(rowcnt + N, 0, sizeof(int), s));
            dmat_free(S, s);
            S.nbr = N; S.nbc = N; S.br = 1; S.bc = 1;
            S.rp = dmalloc<int>(N + 1, s);
            exclusive_scan(rowcnt, S.rp, N + 1, s);
            dfree(rowcnt, s);
            S.nnz = readback(S.rp + N, s);
            S.ci = dmalloc<int>(S.nnz, s);
            S.v = dmalloc<double>(S.nnz, s);
            k_shat_row_fill<<<blocks, 32 * kShatWarps, 0, s>>>(N, D.rp, D.ci, D.v, C.rp, C.ci, C.v, B.rp, B.ci, B.v, dinv,
                                                               S.rp, S.ci, S.v);
            NBP_LAUNCHED();
            dfree(dinv, s);
            return;
        }
    }
    NBP_CUDA(cudaMemsetAsync(cnt + N, 0, sizeof(long long), s));
    exclusive_scan(cnt, off, N + 1, s);
    const long long ntup = readback(off + N, s);
    unsigned long long *key = dmalloc<unsigned long long>(ntup, s);
    double *t = dmalloc<double>(ntup, s);
    k_shat_fill<<<grid_exact(N), 256, 0, s>>>(N, D.rp, D.ci, C.rp, C.ci, C.v, B.rp, B.ci, B.v, dinv, off, key, t);
    NBP_LAUNCHED();
    dfree(cnt, s); dfree(off, s); dfree(dinv, s);
    sort_pairs(key, t, ntup, bits_for((unsigned long long)N * (unsigned long long)N), s);
    int *head = dmalloc<int>(ntup + 1, s), *sid = dmalloc<int>(ntup + 1, s);
    k_heads_all<<<grid_exact(ntup), 256, 0, s>>>(ntup, key, head);
    NBP_LAUNCHED();
    NBP_CUDA(cudaMemsetAsync(head + ntup, 0, sizeof(int), s));
    exclusive_scan(head, sid, ntup + 1, s);
    const int nseg = readback(sid + ntup, s);
    long long *start = dmalloc<long long>(nseg + 1, s);
    k_seg_starts<<<grid_exact(ntup), 256, 0, s>>>(ntup, head, sid, start);
    NBP_LAUNCHED();
    dfree(head, s); dfree(sid, s);
    dmat_free(S, s);
    S.nbr = N; S.nbc = N; S.br = 1; S.bc = 1; S.nnz = nseg;
    S.ci = dmalloc<int>(nseg, s);
    S.v = dmalloc<double>(nseg, s);
    int *rowcnt = dmalloc<int>(N + 1, s);
    NBP_CUDA(cudaMemsetAsync(rowcnt, 0, sizeof(int) * (N + 1), s));
    k_shat_reduce<<<grid_exact(nseg), 256, 0, s>>>(nseg, ntup, key, start, t, N, D.rp, D.ci, D.v, S.ci, S.v, rowcnt);
    NBP_LAUNCHED();
    S.rp = dmalloc<int>(N + 1, s);
    exclusive_scan(rowcnt, S.rp, N + 1, s);
    dfree(rowcnt, s); dfree(key, s); dfree(t, s); dfree(start, s);
}

// ============================================================== transpose
__global__ void k_tr_keys(int n, const int *rp, const int *ci, unsigned int *key, int *val) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int e = rp[i]; e < rp[i + 1]; ++e) { key[e] = (unsigned)ci[e]; val[e] = e; }
}
__global__ void k_tr_count(long long nnz, const int *ci, int *cnt) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < nnz) atomicAdd(cnt + ci[e], 1);
}
__global__ void k_tr_fill(long long nnz, int br, int bc, const int *row, const int *perm, const double *v, int *ci_out,
                          double *v_out) {
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nnz) return;
    const int e = perm[p];
    ci_out[p] = row[e];
    const double *src = v + (long long)e * br * bc;
    double *dst = v_out + p * br * bc;
    for (int a = 0; a < br; ++a)
        for (int b = 0; b < bc; ++b) dst[b * br + a] = src[a * bc + b];
}

// out = in^T (blocks transposed); rows of out sorted by column (stable sort)
void transpose_dmat(const DMat &in, DMat &out, cudaStream_t s) {
    dmat_free(out, s);
    out.nbr = in.nbc; out.nbc = in.nbr; out.br = in.bc; out.bc = in.br; out.nnz = in.nnz;
    unsigned int *key = dmalloc<unsigned int>(in.nnz, s);
    int *perm = dmalloc<int>(in.nnz, s);
    k_tr_keys<<<grid_exact(in.nbr), 256, 0, s>>>(in.nbr, in.rp, in.ci, key, perm);
    NBP_LAUNCHED();
    sort_pairs(key, perm, in.nnz, bits_for((unsigned long long)in.nbc), s);
    int *row = dmalloc<int>(in.nnz, s);
    k_entry_rows<<<grid_exact(in.nbr), 256, 0, s>>>(in.nbr, in.rp, row);
    int *cnt = dmalloc<int>(out.nbr + 1, s);
    NBP_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * (out.nbr + 1), s));
    k_tr_count<<<grid_exact(in.nnz), 256, 0, s>>>(in.nnz, in.ci, cnt);
    NBP_LAUNCHED();
    out.rp = dmalloc<int>(out.nbr + 1, s);
    exclusive_scan(cnt, out.rp, out.nbr + 1, s);
    out.ci = dmalloc<int>(out.nnz, s);
    out.v = dmalloc<double>(out.nnz * out.bb(), s);
    k_tr_fill<<<grid_exact(in.nnz), 256, 0, s>>>(in.nnz, in.br, in.bc, row, perm, in.v, out.ci, out.v);
    NBP_LAUNCHED();
    dfree(key, s); dfree(perm, s); dfree(row, s); dfree(cnt, s);
}

}  // namespace nbp
