// spmv.cu -- instantiation and dispatch of the block-sparse product kernels
// (A: 3x3, B: 3x1, C: 1x3, D / S_hat: 1x1 blocks) for FP64, FP32 and BF16
// values, FP64 or FP32 vectors, and the fused epilogues.
#include "kernels.cuh"
#include "spmv.cuh"

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

namespace nbp {

template <int BR, int BC, int G, typename VT, typename XT>
static void launch_epi(const SpmvArgs &a, int epi, bool lr, cudaStream_t s) {
    const long long threads = (long long)a.nbr * G;
    const unsigned grid = grid_exact(threads);
    switch (epi) {
    case EPI_SET:
        if constexpr (BR == 3 && BC == 3) {
            if (lr) { klaunch(k_bspmv<BR, BC, G, VT, XT, EPI_SET, true>, grid, 256u, s, a); break; }
        }
        klaunch(k_bspmv<BR, BC, G, VT, XT, EPI_SET, false>, grid, 256u, s, a);
        break;
    case EPI_ADD: klaunch(k_bspmv<BR, BC, G, VT, XT, EPI_ADD, false>, grid, 256u, s, a); break;
    case EPI_SUB: klaunch(k_bspmv<BR, BC, G, VT, XT, EPI_SUB, false>, grid, 256u, s, a); break;
    case EPI_RES:
        if constexpr (BR == BC) { klaunch(k_bspmv<BR, BC, G, VT, XT, EPI_RES, false>, grid, 256u, s, a); break; }
        throw Error{NBP_ERR_INVALID, "spmv: residual epilogue needs square blocks"};
    case EPI_CHEB:
        if constexpr (BR == BC) { klaunch(k_bspmv<BR, BC, G, VT, XT, EPI_CHEB, false>, grid, 256u, s, a); break; }
        throw Error{NBP_ERR_INVALID, "spmv: Chebyshev epilogue needs square blocks"};
    default: throw Error{NBP_ERR_INVALID, "spmv: unknown epilogue"};
    }
    NBP_LAUNCHED();
}

template <int BR, int BC, typename VT, typename XT>
static void launch_g(const SpmvArgs &a, int G, int epi, bool lr, cudaStream_t s) {
    if constexpr (BR == BC) {
        switch (G) {
        case 4: launch_epi<BR, BC, 4, VT, XT>(a, epi, lr, s); return;
        case 8: launch_epi<BR, BC, 8, VT, XT>(a, epi, lr, s); return;
        case 16: launch_epi<BR, BC, 16, VT, XT>(a, epi, lr, s); return;
        default: launch_epi<BR, BC, 32, VT, XT>(a, epi, lr, s); return;
        }
    } else {
        launch_epi<BR, BC, 8, VT, XT>(a, epi, lr, s);
    }
}

template <int BR, int BC, typename XT>
static void launch_vt(const DMat &M, int vsel, SpmvArgs a, int G, int epi, bool lr, cudaStream_t s) {
    if constexpr (sizeof(XT) == 8) {
        require(vsel == 0, NBP_ERR_INVALID, "spmv: FP64 vectors need FP64 values");
        a.val = M.v;
        launch_g<BR, BC, double, double>(a, G, epi, lr, s);
    } else {
        if (vsel == 2) {
            require(M.v16 != nullptr, NBP_ERR_STATE, "spmv: BF16 values not built (run setup with precision 2)");
            a.val = M.v16;
            launch_g<BR, BC, __nv_bfloat16, float>(a, G, epi, lr, s);
        } else {
            require(M.v32 != nullptr, NBP_ERR_STATE, "spmv: FP32 values not built (run setup with precision >= 1)");
            a.val = M.v32;
            launch_g<BR, BC, float, float>(a, G, epi, lr, s);
        }
    }
}

int fine_threads(int rows) { return rows < 12000 ? 8 : rows < 45000 ? 4 : rows < 200000 ? 2 : 1; }

int choose_group(const DMat &M) {
    const double per_row = M.nbr ? (double)M.nnz * M.bb() / M.nbr : 0.0;
    if (per_row <= 10) return 4;
    if (per_row <= 40) return 8;
    if (per_row <= 160) return 16;
    return 32;
}

// threads per row of the sliced kernel that M is tuned to (0: a flat kernel)
static int sell_threads(const DMat &M) {
    const int G = M.tuned >= 0 ? M.tuned : 0;
    return G == 0 ? 1 : (is_sellm(G) ? G - kSellMT : 0);
}

template <int BS, typename VT, typename XT, int C>
static void launch_sell_epi(const SpmvArgs &a, int epi, bool lr, cudaStream_t s) {
    const unsigned grid = grid_exact((long long)a.nslice * C);
    switch (epi) {
    case EPI_SET:
        if constexpr (BS == 3) {
            if (lr) { klaunch(k_sell<BS, VT, XT, EPI_SET, true, C>, grid, 256u, s, a); break; }
        }
        klaunch(k_sell<BS, VT, XT, EPI_SET, false, C>, grid, 256u, s, a);
        break;
    case EPI_ADD: klaunch(k_sell<BS, VT, XT, EPI_ADD, false, C>, grid, 256u, s, a); break;
    case EPI_SUB: klaunch(k_sell<BS, VT, XT, EPI_SUB, false, C>, grid, 256u, s, a); break;
    case EPI_RES: klaunch(k_sell<BS, VT, XT, EPI_RES, false, C>, grid, 256u, s, a); break;
    case EPI_CHEB: klaunch(k_sell<BS, VT, XT, EPI_CHEB, false, C>, grid, 256u, s, a); break;
    default: throw Error{NBP_ERR_INVALID, "spmv: unknown epilogue"};
    }
    NBP_LAUNCHED();
}

template <int BS, typename VT, typename XT, int C, int T>
static void launch_sellm_epi(const SpmvArgs &a, int epi, bool lr, cudaStream_t s) {
    const unsigned grid = grid_exact((long long)a.nslice * C * T);
    switch (epi) {
    case EPI_SET:
        if constexpr (BS == 3) {
            if (lr) { klaunch(k_sellm<BS, VT, XT, EPI_SET, C, T, true>, grid, 256u, s, a); break; }
        }
        klaunch(k_sellm<BS, VT, XT, EPI_SET, C, T>, grid, 256u, s, a);
        break;
    case EPI_ADD: klaunch(k_sellm<BS, VT, XT, EPI_ADD, C, T>, grid, 256u, s, a); break;
    case EPI_SUB: klaunch(k_sellm<BS, VT, XT, EPI_SUB, C, T>, grid, 256u, s, a); break;
    case EPI_RES: klaunch(k_sellm<BS, VT, XT, EPI_RES, C, T>, grid, 256u, s, a); break;
    case EPI_CHEB: klaunch(k_sellm<BS, VT, XT, EPI_CHEB, C, T>, grid, 256u, s, a); break;
    default: throw Error{NBP_ERR_INVALID, "spmv: unknown epilogue"};
    }
    NBP_LAUNCHED();
}

template <int BS, typename VT, typename XT, int C>
static void launch_sellm_t(const SpmvArgs &a, int epi, bool lr, cudaStream_t s, int T) {
    if (T == 8) launch_sellm_epi<BS, VT, XT, C, 8>(a, epi, lr, s);
    else if (T == 4) launch_sellm_epi<BS, VT, XT, C, 4>(a, epi, lr, s);
    else launch_sellm_epi<BS, VT, XT, C, 2>(a, epi, lr, s);
}

// one thread per row in the sums of V (BF16 values); false: no such form
template <int BS, int C, int V> static bool launch_chains_v(const SpmvArgs &a, int epi, bool lr, cudaStream_t s) {
    using B = __nv_bfloat16;
    constexpr int K = C == 32 ? 2 : 1;
    const unsigned grid = grid_exact((long long)a.nslice * C);
    if (epi == EPI_RES) klaunch(k_sell<BS, B, float, EPI_RES, false, C, K, V>, grid, 256u, s, a);
    else if (epi == EPI_CHEB) klaunch(k_sell<BS, B, float, EPI_CHEB, false, C, K, V>, grid, 256u, s, a);
    else if (epi != EPI_SET || BS != 3) return false;
    else if (lr) klaunch(k_sell<3, B, float, EPI_SET, true, C, K, V>, grid, 256u, s, a);
    else klaunch(k_sell<3, B, float, EPI_SET, false, C, K, V>, grid, 256u, s, a);
    NBP_LAUNCHED();
    return true;
}
template <int BS, int C> static bool launch_chains(const SpmvArgs &a, int epi, bool lr, cudaStream_t s, int V) {
    if (V == 8) return launch_chains_v<BS, C, 8>(a, epi, lr, s);
    if (V == 4) return launch_chains_v<BS, C, 4>(a, epi, lr, s);
    return V == 2 && launch_chains_v<BS, C, 2>(a, epi, lr, s);
}

// P threads per row in the sums of V; false: no such form
template <int BS, typename VT, int C, int P, int V>
static bool launch_few_v(const SpmvArgs &a, int epi, bool lr, cudaStream_t s) {
    constexpr int K = C == 32 && std::is_same<VT, __nv_bfloat16>::value ? 2 : 1;
    const unsigned grid = grid_exact((long long)a.nslice * C * P);
    if (epi == EPI_RES) klaunch(k_sellm<BS, VT, float, EPI_RES, C, P, false, K, V>, grid, 256u, s, a);
    else if (epi == EPI_CHEB) klaunch(k_sellm<BS, VT, float, EPI_CHEB, C, P, false, K, V>, grid, 256u, s, a);
    else if (epi != EPI_SET || BS != 3) return false;
    else if (lr) klaunch(k_sellm<3, VT, float, EPI_SET, C, P, true, K, V>, grid, 256u, s, a);
    else klaunch(k_sellm<3, VT, float, EPI_SET, C, P, false, K, V>, grid, 256u, s, a);
    NBP_LAUNCHED();
    return true;
}
// as few threads per row as a batch's rows leave room for, in the sums of V
template <int BS, typename VT, int C>
static bool launch_beside(const SpmvArgs &a, int epi, bool lr, cudaStream_t s, int P, int V) {
    if (P == 2 && V == 8) return launch_few_v<BS, VT, C, 2, 8>(a, epi, lr, s);
    if (P == 2 && V == 4) return launch_few_v<BS, VT, C, 2, 4>(a, epi, lr, s);
    if (P == 4 && V == 8) return launch_few_v<BS, VT, C, 4, 8>(a, epi, lr, s);
    if (P != 1) return false;
    if constexpr (std::is_same<VT, __nv_bfloat16>::value) return launch_chains<BS, C>(a, epi, lr, s, V);
    else if (V == 8) return launch_few_v<BS, VT, C, 1, 8>(a, epi, lr, s);
    else if (V == 4) return launch_few_v<BS, VT, C, 1, 4>(a, epi, lr, s);
    else return V == 2 && launch_few_v<BS, VT, C, 1, 2>(a, epi, lr, s);
}

// T threads per row (T = 1: the one-thread kernel)
template <int BS, typename VT, typename XT>
static void launch_sell_c(const DMat &M, const SpmvArgs &a, int epi, bool lr, cudaStream_t s, int T) {
    if constexpr (std::is_same<VT, __nv_bfloat16>::value || (std::is_same<VT, float>::value && BS == 3))
        if (M.beside && M.beside < T &&
            (M.sl_c == 8 ? launch_beside<BS, VT, 8>(a, epi, lr, s, M.beside, T)
                         : launch_beside<BS, VT, 32>(a, epi, lr, s, M.beside, T)))
            return;
    if (T > 1) {
        if (M.sl_c == 8) launch_sellm_t<BS, VT, XT, 8>(a, epi, lr, s, T);
        else launch_sellm_t<BS, VT, XT, 32>(a, epi, lr, s, T);
        return;
    }
    if (M.sl_c == 8) launch_sell_epi<BS, VT, XT, 8>(a, epi, lr, s);
    else launch_sell_epi<BS, VT, XT, 32>(a, epi, lr, s);
}

template <int BS, typename XT>
static void launch_sell(const DMat &M, int vsel, SpmvArgs a, int epi, bool lr, cudaStream_t s, int T) {
    a.nslice = M.nslice;
    a.sl_ptr = M.sl_ptr;
    a.sl_ci = M.sl_ci;
    if constexpr (sizeof(XT) == 8) {
        a.val = M.sl_v;
        launch_sell_c<BS, double, double>(M, a, epi, lr, s, T);
    } else if (vsel == 2) {
        require(M.sl_v16 != nullptr, NBP_ERR_STATE, "spmv: BF16 sliced values not built");
        a.sl_ptr = M.sl2_ptr;   // paired layout
        a.sl_ci = M.sl2_ci;
        a.val = M.sl_v16;
        launch_sell_c<BS, __nv_bfloat16, float>(M, a, epi, lr, s, T);
    } else {
        require(M.sl_v32 != nullptr, NBP_ERR_STATE, "spmv: FP32 sliced values not built");
        a.val = M.sl_v32;
        launch_sell_c<BS, float, float>(M, a, epi, lr, s, T);
    }
}

template <int BR, int BC, typename VT, typename XT, int C, int T>
static void launch_sellr_t(const SpmvArgs &a, int epi, cudaStream_t s) {
    const unsigned grid = grid_exact((long long)a.nslice * C * T);
    switch (epi) {
    case EPI_SET: klaunch(k_sellr<BR, BC, VT, XT, EPI_SET, C, T>, grid, 256u, s, a); break;
    case EPI_ADD: klaunch(k_sellr<BR, BC, VT, XT, EPI_ADD, C, T>, grid, 256u, s, a); break;
    case EPI_SUB: klaunch(k_sellr<BR, BC, VT, XT, EPI_SUB, C, T>, grid, 256u, s, a); break;
    default: throw Error{NBP_ERR_INVALID, "spmv: rectangular blocks take SET, ADD or SUB"};
    }
    NBP_LAUNCHED();
}
template <int BR, int BC, typename VT, typename XT, int C>
static void launch_sellr_epi(const SpmvArgs &a, int T, int epi, cudaStream_t s) {
    switch (T) {
    case 8: launch_sellr_t<BR, BC, VT, XT, C, 8>(a, epi, s); break;
    case 4: launch_sellr_t<BR, BC, VT, XT, C, 4>(a, epi, s); break;
    case 2: launch_sellr_t<BR, BC, VT, XT, C, 2>(a, epi, s); break;
    default: launch_sellr_t<BR, BC, VT, XT, C, 1>(a, epi, s);
    }
}

// rectangular blocks (3x1, 1x3) on their sliced-ELL copy, FP64 or FP32 values
template <int BR, int BC, typename XT>
static void launch_sellr(const DMat &M, int vsel, SpmvArgs a, int epi, cudaStream_t s) {
    a.nslice = M.nslice;
    a.sl_ptr = M.sl_ptr;
    a.sl_ci = M.sl_ci;
    const int T = std::max(1, sell_threads(M));
    if constexpr (sizeof(XT) == 8) {
        a.val = M.sl_v;
        if (M.sl_c == 8) launch_sellr_epi<BR, BC, double, double, 8>(a, T, epi, s);
        else launch_sellr_epi<BR, BC, double, double, 32>(a, T, epi, s);
    } else {
        a.val = M.sl_v32;
        if (M.sl_c == 8) launch_sellr_epi<BR, BC, float, float, 8>(a, T, epi, s);
        else launch_sellr_epi<BR, BC, float, float, 32>(a, T, epi, s);
    }
}

// Algorithmic bytes of one product y = epilogue(M x): every stored block's
// values and column index once, the row pointers (flat kernel) or the slice
// pointers (sliced layouts; their padding is not counted), x once, and the
// epilogue's vectors: SET writes y; ADD and SUB read and write y; RES reads
// b and writes y; CHEB reads b, d and the block-diagonal inverse and writes
// d and xout (x_i itself is the product's input, counted once).
static double product_bytes(const DMat &M, int vsel, int xs, int epi, bool sliced) {
    const double vb = xs == 8 ? 8.0 : (vsel == 2 ? 2.0 : 4.0);
    double b = (double)M.nnz * (M.bb() * vb + 4.0);
    b += sliced ? (double)(M.nslice + 1) * 8.0 : (double)(M.nbr + 1) * 4.0;
    const double nx = (double)M.nbc * M.bc * xs, ny = (double)M.nbr * M.br * xs;
    b += nx;
    if (epi == EPI_SET) b += ny;
    else if (epi == EPI_CHEB) b += 4.0 * ny + (double)M.nbr * M.br * M.br * xs;
    else b += 2.0 * ny;
    return b;
}

bool spmv_dot_ok(const DMat &M, int vsel, int xbytes, long long max_blocks) {
    if (M.br != 1 || M.bc != 1 || !M.sl_ci || M.nbr == 0) return false;
    const int T = sell_threads(M);
    if (T == 0) return false;
    if (((long long)M.nslice * M.sl_c * T + 255) / 256 > max_blocks) return false;
    if (xbytes == 8) return M.sl_v != nullptr;
    return vsel == 2 ? M.sl_v16 != nullptr : M.sl_v32 != nullptr;
}

template <typename VT, typename XT, int C>
static void launch_sell_dot(const SpmvArgs &a, const DotArgs &q, int T, cudaStream_t s) {
    const unsigned grid = grid_exact((long long)a.nslice * C * T);
    if (T == 8) klaunch(k_sell_dot<VT, XT, C, 8>, grid, 256u, s, a, q);
    else if (T == 4) klaunch(k_sell_dot<VT, XT, C, 4>, grid, 256u, s, a, q);
    else if (T == 2) klaunch(k_sell_dot<VT, XT, C, 2>, grid, 256u, s, a, q);
    else klaunch(k_sell_dot<VT, XT, C, 1>, grid, 256u, s, a, q);
    NBP_LAUNCHED();
}
template <typename VT, typename XT>
static void launch_sell_dot_c(const DMat &M, const SpmvArgs &a, const DotArgs &q, int T, cudaStream_t s) {
    if (M.sl_c == 8) launch_sell_dot<VT, XT, 8>(a, q, T, s);
    else launch_sell_dot<VT, XT, 32>(a, q, T, s);
}

template <typename XT>
double spmv_dot(const DMat &M, int vsel, SpmvArgs a, const DotArgs &q, cudaStream_t s) {
    const int T = sell_threads(M);
    a.nbr = M.nbr;
    a.nslice = M.nslice;
    a.sl_ptr = M.sl_ptr;
    a.sl_ci = M.sl_ci;
    if constexpr (sizeof(XT) == 8) {
        a.val = M.sl_v;
        launch_sell_dot_c<double, double>(M, a, q, T, s);
    } else if (vsel == 2) {
        a.sl_ptr = M.sl2_ptr;   // paired layout
        a.sl_ci = M.sl2_ci;
        a.val = M.sl_v16;
        launch_sell_dot_c<__nv_bfloat16, float>(M, a, q, T, s);
    } else {
        a.val = M.sl_v32;
        launch_sell_dot_c<float, float>(M, a, q, T, s);
    }
    const double ny = (double)M.nbr * sizeof(XT);
    return product_bytes(M, vsel, (int)sizeof(XT), EPI_SET, true) + ny + (q.db ? ny : 0.0);
}

template <typename XT>
double spmv(const DMat &M, int vsel, SpmvArgs a, int epi, bool lr, cudaStream_t s, int G) {
    a.nbr = M.nbr;
    a.rp = M.rp;
    a.ci = M.ci;
    if (a.nbr == 0) return 0.0;
    constexpr int xs = (int)sizeof(XT);
    // rectangular coupling blocks: sliced ELL for FP64 / FP32 values (BF16: flat kernel)
    if (M.br != M.bc && M.sl_ci && G <= 0 && epi <= EPI_SUB && vsel != 2 &&
        (sizeof(XT) == 8 ? M.sl_v != nullptr : M.sl_v32 != nullptr)) {
        if (M.br == 3 && M.bc == 1) { launch_sellr<3, 1, XT>(M, vsel, a, epi, s); return product_bytes(M, vsel, xs, epi, true); }
        if (M.br == 1 && M.bc == 3) { launch_sellr<1, 3, XT>(M, vsel, a, epi, s); return product_bytes(M, vsel, xs, epi, true); }
    }
    const bool sell_ok = M.sl_ci && M.br == M.bc && (sizeof(XT) == 8 ? M.sl_v != nullptr : true);
    if (G < 0) G = (M.tuned >= 0) ? M.tuned : (sell_ok ? 0 : choose_group(M));
    if ((G == 0 || is_sellm(G)) && !sell_ok) G = choose_group(M);
    if (sell_ok && (G == 0 || is_sellm(G))) {
        const int T = G == 0 ? 1 : G - kSellMT;
        if (M.br == 3) launch_sell<3, XT>(M, vsel, a, epi, lr, s, T);
        else launch_sell<1, XT>(M, vsel, a, epi, lr, s, T);
        return product_bytes(M, vsel, xs, epi, true);
    }
    if (M.br == 3 && M.bc == 3) launch_vt<3, 3, XT>(M, vsel, a, G, epi, lr, s);
    else if (M.br == 3 && M.bc == 1) launch_vt<3, 1, XT>(M, vsel, a, G, epi, lr, s);
    else if (M.br == 1 && M.bc == 3) launch_vt<1, 3, XT>(M, vsel, a, G, epi, lr, s);
    else if (M.br == 1 && M.bc == 1) launch_vt<1, 1, XT>(M, vsel, a, G, epi, lr, s);
    else throw Error{NBP_ERR_INVALID, "spmv: unsupported block shape"};
    return product_bytes(M, vsel, xs, epi, false);
}

// Threads per row of the post-smoothing product (rows of A P hold 6-8 blocks,
// those of S_hat P 10-20 scalars): one streams long levels, its epilogue's
// operands loaded after the products; two with two pairs at once fill the GPU on
// shorter ones; four where a row's chain of loads is all there is.  Solves with
// one / two / four threads on the levels of each range, ms: from 400,000 rows on
// 4.34M unknowns 648 / 675; between 654 / 648 / 653, 0.56M 156.5 / 155.6 / 159.1,
// 24x24x96 FP64 77.4 / 74.2 / 76.3; below (two / four) cube of 16 17.3 / 17.0,
// 19x23x61 FP32 43.3 / 42.1, 24x24x96 FP64 76.1 / 74.2.
static int post_threads(const DMat &AP, bool paired) {
    if (AP.nbr < (paired ? 8000 : 40000)) return 4;
    return AP.nbr < 400000 ? 2 : 1;
}

template <int BS, typename VT, typename XT>
static void launch_post(const DMat &AP, const SpmvArgs &a, cudaStream_t s) {
    const int T = post_threads(AP, std::is_same<VT, __nv_bfloat16>::value);
    const unsigned grid = grid_exact((long long)AP.nslice * AP.sl_c * T);
    auto with_t = [&](auto c) {
        constexpr int C = decltype(c)::value;
        if (T == 4) klaunch(k_sellm<BS, VT, XT, EPI_POST, C, 4, false, 1>, grid, 256u, s, a);
        else if (T == 2) klaunch(k_sellm<BS, VT, XT, EPI_POST, C, 2, false, 2>, grid, 256u, s, a);
        else klaunch(k_sell<BS, VT, XT, EPI_POST, false, C, 2>, grid, 256u, s, a);
    };
    if (AP.sl_c == 8) with_t(std::integral_constant<int, 8>());
    else with_t(std::integral_constant<int, 32>());
    NBP_LAUNCHED();
}
template <int BS, typename XT> static void launch_post_v(const DMat &AP, int vsel, SpmvArgs a, cudaStream_t s) {
    if constexpr (sizeof(XT) == 8) {
        a.val = AP.sl_v;
        launch_post<BS, double, double>(AP, a, s);
    } else if (vsel == 2) {
        require(AP.sl_v16 != nullptr, NBP_ERR_STATE, "spmv: BF16 sliced values not built");
        a.sl_ptr = AP.sl2_ptr;   // paired layout
        a.sl_ci = AP.sl2_ci;
        a.val = AP.sl_v16;
        launch_post<BS, __nv_bfloat16, float>(AP, a, s);
    } else {
        require(AP.sl_v32 != nullptr, NBP_ERR_STATE, "spmv: FP32 sliced values not built");
        a.val = AP.sl_v32;
        launch_post<BS, float, float>(AP, a, s);
    }
}
template <typename XT> double spmv_post(const DMat &AP, int vsel, SpmvArgs a, cudaStream_t s) {
    a.nbr = AP.nbr;
    a.nslice = AP.nslice;
    a.sl_ptr = AP.sl_ptr;
    a.sl_ci = AP.sl_ci;
    if (AP.br == 3) launch_post_v<3, XT>(AP, vsel, a, s);
    else launch_post_v<1, XT>(AP, vsel, a, s);
    constexpr int xs = (int)sizeof(XT);
    const double ny = (double)AP.nbr * AP.br * xs;
    // the product's bytes (with b read and xout written), xin and the
    // aggregates read, the block-diagonal inverse, d where it is written
    return product_bytes(AP, vsel, xs, EPI_RES, true) + ny + (double)AP.nbr * 4.0 + ny * AP.br + (a.d_write ? ny : 0.0);
}
template double spmv_post<double>(const DMat &, int, SpmvArgs, cudaStream_t);
template double spmv_post<float>(const DMat &, int, SpmvArgs, cudaStream_t);
template double spmv<double>(const DMat &, int, SpmvArgs, int, bool, cudaStream_t, int);
template double spmv<float>(const DMat &, int, SpmvArgs, int, bool, cudaStream_t, int);
template double spmv_dot<double>(const DMat &, int, SpmvArgs, const DotArgs &, cudaStream_t);
template double spmv_dot<float>(const DMat &, int, SpmvArgs, const DotArgs &, cudaStream_t);

}  // namespace nbp
