// vms.cu -- on-device assembly of the residual and of the consistent tangent
// of the P1-P1 residual-based VMS / generalized-alpha discretisation.
//
// Residual (Sec. 2.3, B_m^vol + B_m^bc + B_m^bf and B_p, evaluated at
// vdot_{n+alpha_m}, v_{n+alpha_f}, p_{n+alpha_f} as Sec. 2.4 prescribes):
// per quadrature point of a tet, with u = v_h, the fine scales
// v' = -tau_M (rho udot + rho (u.grad) u + grad p) (P1: the viscous second
// derivatives vanish inside an element; no body force) and p' = -tau_C div u,
// the momentum row of node a, component i, gains
//   rho N_a (udot_i + (u.grad u)_i) - dN_a/dx_i p + mu dN_a/dx_j (du_i/dx_j + du_j/dx_i)
//   - rho v'_i (u.grad N_a) + rho N_a (v'.grad) u_i - rho v'_i (v'.grad N_a) - dN_a/dx_i p'
// and the continuity row N_a div u - grad N_a . v'.  tau_M, tau_C follow
// Sec. 2.3 (C_T, C_I, the metric G with the simplex matrix M), evaluated at a
// given velocity (the state itself, or a frozen one).  The outlet traction
// adds sum_k P_k a^k; backflow (B_m^bf) adds -rho beta (u.n)_- N_a u_i on the
// outlet triangles.
//
// Tangent (Sec. 2.5, F + the blocks B, C, D; K stays the solvers' matrix-free
// rank-one term): the derivative of the residual with respect to
// (vdot_{n+1}, pdot_{n+1}), i.e. alpha_m d/dvdot_{n+alpha_m} + alpha_f gamma
// dt d/d(v, p)_{n+alpha_f}, with tau_M and tau_C held fixed.  The FP64 tangent
// of a tet is the rows' derivative written out (k_tan_tet64); the FP32 one and
// the outlet triangles' are taken by forward-mode dual numbers with four
// partials, one thread per (element, column node b) seeding the unknowns of b
// and evaluating the element's rows.
//
// Determinism: every tet (triangle) writes its own scratch slots; gather
// kernels then sum, per residual row and per pattern slot, the slots of the
// incident elements in ascending element order.  No atomics.
#include "nbp_common.cuh"
#include "vms.cuh"

namespace nbp {

// ---------------------------------------------------------------- dual numbers
template <typename T> struct D4 {
    T v, d[4];
};
template <typename T> __device__ __forceinline__ D4<T> operator+(D4<T> a, const D4<T> &b) {
    a.v += b.v;
#pragma unroll
    for (int q = 0; q < 4; ++q) a.d[q] += b.d[q];
    return a;
}
template <typename T> __device__ __forceinline__ D4<T> operator-(D4<T> a, const D4<T> &b) {
    a.v -= b.v;
#pragma unroll
    for (int q = 0; q < 4; ++q) a.d[q] -= b.d[q];
    return a;
}
template <typename T> __device__ __forceinline__ D4<T> operator*(const D4<T> &a, const D4<T> &b) {
    D4<T> r;
    r.v = a.v * b.v;
#pragma unroll
    for (int q = 0; q < 4; ++q) r.d[q] = a.d[q] * b.v + a.v * b.d[q];
    return r;
}
template <typename T> __device__ __forceinline__ D4<T> operator*(D4<T> a, T s) {
    a.v *= s;
#pragma unroll
    for (int q = 0; q < 4; ++q) a.d[q] *= s;
    return a;
}

// uniform access for plain and dual values
template <typename V> struct Num;
template <> struct Num<double> {
    using T = double;
    __device__ static double cst(double c) { return c; }
    __device__ static double val(double x) { return x; }
};
template <typename T_> struct Num<D4<T_>> {
    using T = T_;
    __device__ static D4<T_> cst(T_ c) {
        D4<T_> r;
        r.v = c;
#pragma unroll
        for (int q = 0; q < 4; ++q) r.d[q] = T_(0);
        return r;
    }
    __device__ static T_ val(const D4<T_> &x) { return x.v; }
};

// ---------------------------------------------------------------- geometry
template <typename T> __device__ __forceinline__ void cross3(const T a[3], const T b[3], T c[3]) {
    c[0] = a[1] * b[2] - a[2] * b[1];
    c[1] = a[2] * b[0] - a[0] * b[2];
    c[2] = a[0] * b[1] - a[1] * b[0];
}
template <typename T> __device__ __forceinline__ T dot3(const T a[3], const T b[3]) {
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}
// Barycentric gradients by cross products: grad l_1 = (e2 x e3) / det, etc.,
// e_k = x_k - x_0, det = e1 . (e2 x e3), grad l_0 = -(sum of the others).
// Returns the volume.
template <typename T> __device__ __forceinline__ T tet_gradients(const T e[3][3], T dN[4][3]) {
    T c23[3], c31[3], c12[3];
    cross3(e[1], e[2], c23);
    cross3(e[2], e[0], c31);
    cross3(e[0], e[1], c12);
    const T det = dot3(e[0], c23);
    const T inv = T(1) / det;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        dN[1][r] = c23[r] * inv;
        dN[2][r] = c31[r] * inv;
        dN[3][r] = c12[r] * inv;
        dN[0][r] = -(dN[1][r] + dN[2][r] + dN[3][r]);
    }
    return fabs(det) / T(6);
}

// The degree-2 rule on a tet: N_a is kQHi at point a and kQLo at the other
// three ((5 + 3 sqrt 5) / 20, (5 - sqrt 5) / 20), each point of weight vol / 4.
constexpr double kQHi = 0.58541019662496845446, kQLo = 0.13819660112501051518;
// The metric of Sec. 2.3 is G = m0 sum_a grad l_a (x) grad l_a (with xi_k =
// l_k and M = m0 (1 + delta_kl), sum_kl dxi_k M_kl dxi_l expands to that), so
// u.G u = m0 sum_a (u . grad l_a)^2, G:G = m0^2 sum_ab (grad l_a . grad l_b)^2
// and tr G = m0 sum_a |grad l_a|^2.
constexpr double kM0 = 0.62996052494743658238;   // 2^(1/3) / 2

// The same geometry as the dual-number rows of the FP32 tangent take it:
// G = m0 sum_{a=0..3} grad l_a (x) grad l_a: with xi_k = l_k (k = 1..3) and
// M = m0 (1 + delta_kl), sum_kl dxi_k M_kl dxi_l expands to exactly this.
template <typename T> struct Geo {
    T dN[4][3];
    T vol, G[3][3], GG, trG;
};
template <typename T> __device__ void tet_geo(const double *X, const int *nd, Geo<T> &g) {
    T x0[3], e[3][3];
    for (int r = 0; r < 3; ++r) x0[r] = (T)X[3LL * nd[0] + r];
    for (int k = 0; k < 3; ++k)
        for (int r = 0; r < 3; ++r) e[k][r] = (T)X[3LL * nd[k + 1] + r] - x0[r];
    T c23[3], c31[3], c12[3];
    cross3(e[1], e[2], c23);
    cross3(e[2], e[0], c31);
    cross3(e[0], e[1], c12);
    const T det = e[0][0] * c23[0] + e[0][1] * c23[1] + e[0][2] * c23[2];
    const T inv = T(1) / det;
    for (int r = 0; r < 3; ++r) {
        g.dN[1][r] = c23[r] * inv;
        g.dN[2][r] = c31[r] * inv;
        g.dN[3][r] = c12[r] * inv;
        g.dN[0][r] = -(g.dN[1][r] + g.dN[2][r] + g.dN[3][r]);
    }
    g.vol = fabs(det) / T(6);
    const T m0 = T(0.62996052494743658238);   // 2^(1/3) / 2
    g.GG = T(0);
    g.trG = T(0);
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) {
            T s = T(0);
            for (int a = 0; a < 4; ++a) s += g.dN[a][i] * g.dN[a][j];
            g.G[i][j] = m0 * s;
            g.GG += g.G[i][j] * g.G[i][j];
        }
    g.trG = g.G[0][0] + g.G[1][1] + g.G[2][2];
}

// ------------------------------------------------------------ element rows
// Rows of all four nodes of one tet: Rm[a][i] (momentum), Rp[a] (continuity).
// UD, U, P: nodal vdot, v, p (plain or seeded duals); UT: the velocity tau is
// evaluated at.
template <typename V>
__device__ void tet_rows(const VmsConst &k, const Geo<typename Num<V>::T> &g, const V UD[4][3], const V U[4][3],
                         const V P[4], const typename Num<V>::T UT[4][3], V Rm[4][3], V Rp[4]) {
    using T = typename Num<V>::T;
    using Nm = Num<V>;
    const T rho = (T)k.rho, mu = (T)k.mu;
    V Gv[3][3], gp[3];
    for (int i = 0; i < 3; ++i) {
        gp[i] = P[0] * g.dN[0][i] + P[1] * g.dN[1][i] + P[2] * g.dN[2][i] + P[3] * g.dN[3][i];
        for (int j = 0; j < 3; ++j)
            Gv[i][j] = U[0][i] * g.dN[0][j] + U[1][i] * g.dN[1][j] + U[2][i] * g.dN[2][j] + U[3][i] * g.dN[3][j];
    }
    const V dv = Gv[0][0] + Gv[1][1] + Gv[2][2];
    for (int a = 0; a < 4; ++a) {
        Rp[a] = Nm::cst(T(0));
        for (int i = 0; i < 3; ++i) Rm[a][i] = Nm::cst(T(0));
    }
    const T q_hi = T(0.58541019662496845446), q_lo = T(0.13819660112501051518);   // (5 + 3 sqrt5)/20, (5 - sqrt5)/20
    const T w = g.vol * T(0.25);
    const T visc2 = T(k.CI) * (mu / rho) * (mu / rho) * g.GG + T(k.CT / (k.dt * k.dt));
    for (int q = 0; q < 4; ++q) {
        T Nq[4];
        for (int b = 0; b < 4; ++b) Nq[b] = (b == q) ? q_hi : q_lo;
        V u[3], ud[3];
        T ut[3];
        for (int i = 0; i < 3; ++i) {
            u[i] = U[0][i] * Nq[0] + U[1][i] * Nq[1] + U[2][i] * Nq[2] + U[3][i] * Nq[3];
            ud[i] = UD[0][i] * Nq[0] + UD[1][i] * Nq[1] + UD[2][i] * Nq[2] + UD[3][i] * Nq[3];
            ut[i] = UT[0][i] * Nq[0] + UT[1][i] * Nq[1] + UT[2][i] * Nq[2] + UT[3][i] * Nq[3];
        }
        const V pq = P[0] * Nq[0] + P[1] * Nq[1] + P[2] * Nq[2] + P[3] * Nq[3];
        T uGu = T(0);
        for (int i = 0; i < 3; ++i) uGu += ut[i] * (g.G[i][0] * ut[0] + g.G[i][1] * ut[1] + g.G[i][2] * ut[2]);
        const T tauM = T(1) / (rho * sqrt(visc2 + uGu));
        const T tauC = T(1) / (tauM * g.trG);
        V cv[3], vp[3];
        for (int i = 0; i < 3; ++i) {
            cv[i] = Gv[i][0] * u[0] + Gv[i][1] * u[1] + Gv[i][2] * u[2];
            vp[i] = (ud[i] * rho + cv[i] * rho + gp[i]) * (-tauM);
        }
        const V pf = dv * (-tauC);
        V gvp[3];
        for (int i = 0; i < 3; ++i) gvp[i] = Gv[i][0] * vp[0] + Gv[i][1] * vp[1] + Gv[i][2] * vp[2];
        for (int a = 0; a < 4; ++a) {
            const T *d = g.dN[a];
            const V udN = u[0] * d[0] + u[1] * d[1] + u[2] * d[2];
            const V vdN = vp[0] * d[0] + vp[1] * d[1] + vp[2] * d[2];
            const V adv = (udN + vdN) * rho;   // rho (u + v') . grad N_a
            for (int i = 0; i < 3; ++i) {
                V t = (ud[i] + cv[i] + gvp[i]) * (rho * Nq[a]);
                t = t - (pq + pf) * d[i];
                t = t + ((Gv[i][0] + Gv[0][i]) * d[0] + (Gv[i][1] + Gv[1][i]) * d[1] + (Gv[i][2] + Gv[2][i]) * d[2]) * mu;
                t = t - vp[i] * adv;
                Rm[a][i] = Rm[a][i] + t * w;
            }
            Rp[a] = Rp[a] + (dv * Nq[a] - vdN) * w;
        }
    }
}

// Backflow rows of one outlet triangle: -rho beta (u.n)_- N_a u_i with the
// 3-point rule at barycentric (2/3, 1/6, 1/6) and its permutations.
template <typename V>
__device__ void tri_rows(const VmsConst &k, const double *X, const int *nd, const V U[3][3], V Rm[3][3]) {
    using T = typename Num<V>::T;
    using Nm = Num<V>;
    T e1[3], e2[3], n[3];
    for (int r = 0; r < 3; ++r) {
        e1[r] = (T)(X[3LL * nd[1] + r] - X[3LL * nd[0] + r]);
        e2[r] = (T)(X[3LL * nd[2] + r] - X[3LL * nd[0] + r]);
    }
    cross3(e1, e2, n);
    const T len = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
    for (int r = 0; r < 3; ++r) n[r] /= len;
    const T w = len / T(6);   // area / 3
    const T c = -(T)(k.rho * k.beta);
    for (int a = 0; a < 3; ++a)
        for (int i = 0; i < 3; ++i) Rm[a][i] = Nm::cst(T(0));
    for (int q = 0; q < 3; ++q) {
        T Nq[3];
        for (int b = 0; b < 3; ++b) Nq[b] = (b == q) ? T(2) / T(3) : T(1) / T(6);
        V u[3];
        for (int i = 0; i < 3; ++i) u[i] = U[0][i] * Nq[0] + U[1][i] * Nq[1] + U[2][i] * Nq[2];
        const V un = u[0] * n[0] + u[1] * n[1] + u[2] * n[2];
        if (!(Nm::val(un) < T(0))) continue;
        for (int a = 0; a < 3; ++a)
            for (int i = 0; i < 3; ++i) Rm[a][i] = Rm[a][i] + (un * u[i]) * (c * Nq[a] * w);
    }
}

// ------------------------------------------------------------------ residual
// Rows of one tet per thread, bound by the FP64 pipe (2 operations a clock
// and SM), so the quadrature sum is regrouped into what each point must
// contribute: with M = sum_q [2 mu sym(grad u) - rho v' (x) (u + v') - (p + p') I]
// and F_q = udot + u.grad u + v'.grad u the momentum row of node a is
// w (rho sum_q N_a F_q + M grad N_a), and N_a takes two values only.
// 786,432 tets: 1.50 ms with every point's rows formed one by one, 1.06 ms so.
__global__ void __launch_bounds__(128) k_res_tet(int E, const double *X, const int *tets, const double *vd,
                                                 const double *v, const double *p, const double *vt, VmsConst k,
                                                 double *Re) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= E) return;
    const int4 n4 = reinterpret_cast<const int4 *>(tets)[e];
    const int nd[4] = {n4.x, n4.y, n4.z, n4.w};
    double x[3][3], UD[4][3], U[4][3], UT[4][3], dN[4][3], SP = 0.0, gp[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            if (a > 0) x[a - 1][i] = X[3LL * nd[a] + i] - X[3LL * nd[0] + i];
            UD[a][i] = vd[3LL * nd[a] + i];
            U[a][i] = v[3LL * nd[a] + i];
            UT[a][i] = vt[3LL * nd[a] + i];
        }
    const double vol = tet_gradients<double>(x, dN);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const double pa = p[nd[a]];
        SP += pa;
#pragma unroll
        for (int i = 0; i < 3; ++i) gp[i] += pa * dN[a][i];
    }
    double GG = 0.0, tr = 0.0;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const double d = dot3(dN[a], dN[a]);
        tr += d;
        GG += d * d;
#pragma unroll
        for (int b = a + 1; b < 4; ++b) {
            const double o = dot3(dN[a], dN[b]);
            GG += 2.0 * o * o;
        }
    }
    const double visc2 = k.CI * (k.mu / k.rho) * (k.mu / k.rho) * (kM0 * kM0 * GG) + k.CT / (k.dt * k.dt);
    const double rtr = 1.0 / (kM0 * tr);
    double Gv[3][3], SU[3], SUD[3], SUT[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        SU[i] = kQLo * (U[0][i] + U[1][i] + U[2][i] + U[3][i]);
        SUD[i] = kQLo * (UD[0][i] + UD[1][i] + UD[2][i] + UD[3][i]);
        SUT[i] = kQLo * (UT[0][i] + UT[1][i] + UT[2][i] + UT[3][i]);
#pragma unroll
        for (int j = 0; j < 3; ++j)
            Gv[i][j] = U[0][i] * dN[0][j] + U[1][i] * dN[1][j] + U[2][i] * dN[2][j] + U[3][i] * dN[3][j];
    }
    const double dv = Gv[0][0] + Gv[1][1] + Gv[2][2];
    constexpr double dq = kQHi - kQLo;
    double M[3][3] = {}, Rm[4][3], SF[3] = {}, Svp[3] = {}, Srs = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        double u[3], ud[3], ut[3], cv[3], vp[3], uv[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            u[i] = SU[i] + dq * U[q][i];
            ud[i] = SUD[i] + dq * UD[q][i];
            ut[i] = SUT[i] + dq * UT[q][i];
        }
        const double s1 = dot3(ut, dN[1]), s2 = dot3(ut, dN[2]), s3 = dot3(ut, dN[3]), s0 = s1 + s2 + s3;
        const double rs = k.rho * sqrt(visc2 + kM0 * (s0 * s0 + s1 * s1 + s2 * s2 + s3 * s3));   // 1 / tau_M
        const double mt = -1.0 / rs;
        Srs += rs;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            cv[i] = ud[i] + dot3(Gv[i], u);
            vp[i] = mt * (k.rho * cv[i] + gp[i]);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            uv[i] = u[i] + vp[i];
            Svp[i] += vp[i];
            const double F = cv[i] + dot3(Gv[i], vp);
            SF[i] += F;
            Rm[q][i] = dq * F;
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) M[i][j] += vp[i] * uv[j];
    }
    const double ps = SP - dv * (Srs * rtr);   // sum_q (p + p'), p' = -div u / (tau_M tr G)
    const double w = 0.25 * vol, m4 = 4.0 * k.mu;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) M[i][j] = m4 * (Gv[i][j] + Gv[j][i]) - k.rho * M[i][j] - (i == j ? ps : 0.0);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        double2 *o = reinterpret_cast<double2 *>(Re + 16LL * e + 4 * a);
        double r[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) r[i] = w * (k.rho * (kQLo * SF[i] + Rm[a][i]) + dot3(M[i], dN[a]));
        o[0] = make_double2(r[0], r[1]);
        o[1] = make_double2(r[2], w * (dv - dot3(Svp, dN[a])));
    }
}

__global__ void k_res_tri(int T, const double *X, const int *tris, const double *v, VmsConst k, double *Rf) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    int nd[3];
    for (int a = 0; a < 3; ++a) nd[a] = tris[3LL * t + a];
    double U[3][3], Rm[3][3];
    for (int b = 0; b < 3; ++b)
        for (int i = 0; i < 3; ++i) U[b][i] = v[3LL * nd[b] + i];
    tri_rows<double>(k, X, nd, U, Rm);
    for (int a = 0; a < 3; ++a)
        for (int i = 0; i < 3; ++i) Rf[9LL * t + 3 * a + i] = Rm[a][i];
}

// R rows of node A: its tets' rows (ascending e), its triangles' rows
// (ascending t), the outlet traction sum_k P_k a^k; Dirichlet momentum rows 0.
__global__ void k_res_gather(int N, const int *n2t_ptr, const int *n2t, const int *n2f_ptr, const int *n2f,
                             const double *Re, const double *Rf, const int *lr_rp, const int *lr_k, const int *lr_c,
                             const double *lr_v, const double *P, const uint8_t *dir, double *R) {
    const int A = blockIdx.x * blockDim.x + threadIdx.x;
    if (A >= N) return;
    double r0 = 0.0, r1 = 0.0, r2 = 0.0, r3 = 0.0;
    for (int q = n2t_ptr[A]; q < n2t_ptr[A + 1]; ++q) {
        const double *s = Re + 4LL * n2t[q];   // 16 e + 4 la
        r0 += s[0];
        r1 += s[1];
        r2 += s[2];
        r3 += s[3];
    }
    for (int q = n2f_ptr[A]; q < n2f_ptr[A + 1]; ++q) {
        const double *s = Rf + 3LL * n2f[q];   // 9 t + 3 la
        r0 += s[0];
        r1 += s[1];
        r2 += s[2];
    }
    if (P && lr_rp)
        for (int j = lr_rp[A]; j < lr_rp[A + 1]; ++j) {
            const double f = P[lr_k[j]] * lr_v[j];
            const int c = lr_c[j];
            if (c == 0) r0 += f;
            else if (c == 1) r1 += f;
            else r2 += f;
        }
    if (dir[A]) r0 = r1 = r2 = 0.0;
    R[3LL * A] = r0;
    R[3LL * A + 1] = r1;
    R[3LL * A + 2] = r2;
    R[3LL * N + A] = r3;
}

// ------------------------------------------------------------------- tangent
// 32 bytes (8 floats, 4 doubles) in one store: a whole sector per thread
__device__ __forceinline__ void st32(float *p, const float *v) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}
__device__ __forceinline__ void st32(double *p, const double *v) {
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3])
                 : "memory");
}

// Thread (e, b): seeds the unknowns of local node b -- vdot with alpha_m and
// v with alpha_f gamma dt (partials 0..2), p with alpha_f gamma dt (partial 3)
// -- and writes the blocks (a, b) of all four rows a.
template <typename T>
__global__ void k_tan_tet(int E, const double *X, const int *tets, const double *vd, const double *v, const double *p,
                          const double *vt, VmsConst k, T *Ke) {
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= 4LL * E) return;
    const int e = (int)(tid >> 2), b = (int)(tid & 3);
    int nd[4];
    for (int a = 0; a < 4; ++a) nd[a] = tets[4LL * e + a];
    Geo<T> g;
    tet_geo<T>(X, nd, g);
    D4<T> UD[4][3], U[4][3], P[4];
    T UT[4][3];
    for (int c = 0; c < 4; ++c) {
        for (int i = 0; i < 3; ++i) {
            UD[c][i] = Num<D4<T>>::cst((T)vd[3LL * nd[c] + i]);
            U[c][i] = Num<D4<T>>::cst((T)v[3LL * nd[c] + i]);
            UT[c][i] = (T)vt[3LL * nd[c] + i];
        }
        P[c] = Num<D4<T>>::cst((T)p[nd[c]]);
    }
    for (int i = 0; i < 3; ++i) {
        UD[b][i].d[i] = (T)k.am;
        U[b][i].d[i] = (T)k.c;
    }
    P[b].d[3] = (T)k.c;
    D4<T> Rm[4][3], Rp[4];
    tet_rows<D4<T>>(k, g, UD, U, P, UT, Rm, Rp);
    for (int a = 0; a < 4; ++a) {
        T o[16];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int i = 0; i < 3; ++i) o[4 * i + j] = Rm[a][i].d[j];
            o[12 + j] = Rp[a].d[j];
        }
        T *out = Ke + 16LL * (16LL * e + 4 * a + b);
        st32(out, o);
        st32(out + 8, o + 8);
    }
}

// Four lanes per tet; lane b makes the blocks (a, b) of column node b for all
// four rows a.  The partials are those of vdot with alpha_m and of v and p
// with alpha_f gamma dt (am, c).  With s = u . grad N, t = v' . grad N,
//   dv' / d(b, j) = alpha_b e_j + beta_b Gv e_j,  alpha_b = -tau_M rho (am N_b + c s_b),
//   beta_b = -tau_M rho c N_b,  dv' / dp_b = gamma grad N_b,  gamma = -tau_M c,
// the derivative of the rows (the formulas at the top of the file) is a sum
// of a few matrices that are constant on the tet (I, Gv = grad u, Gv Gv, outer
// products of gradients) with scalar or vector coefficients summed over the
// quadrature points: about 5 kflop per tet in all, where seeding the rows with
// four-partial dual numbers took about 47.  What the lanes share is made once
// and passed by shuffles (an FP64 operation holds the pipe for 16 clocks a
// warp, a shuffle for two): lane b loads node b, lanes 1-3 a gradient each,
// lane i row i of grad u and of its square (lane 3 grad p), lane b quadrature
// point b.  Bound by the FP64 pipe.  786,432 tets: 29.8 -> 4.6 ms.
// FP64 tangents only: in FP32 the regrouped sums round differently from the
// dual numbers, and since the corrector stops after a few inexact steps that
// moved the accepted ydot by up to 3e-8 (k_tan_tet keeps FP32 as it was).
__global__ void __launch_bounds__(128) k_tan_tet64(int E, const double *X, const int *tets, const double *vd,
                                                   const double *v, const double *p, const double *vt, VmsConst k,
                                                   double *Ke) {
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = tid < 4LL * E;
    const int e = live ? (int)(tid >> 2) : E - 1, b = (int)(tid & 3);
    const long long nb = tets[4LL * e + b];
    const int l0 = threadIdx.x & 28;
    auto from = [&](double val, int a) { return __shfl_sync(0xffffffffu, val, l0 + a); };
    auto sum4 = [&](double val) {
        val += __shfl_xor_sync(0xffffffffu, val, 1);
        return val + __shfl_xor_sync(0xffffffffu, val, 2);
    };
    auto pick = [&](double v0, double v1, double v2, double v3) { return b == 0 ? v0 : b == 1 ? v1 : b == 2 ? v2 : v3; };
    const double rho = k.rho, mu = k.mu, c = k.c, am = k.am;
    const double lo = kQLo, dq = kQHi - kQLo;
    double Ub[3], Db[3], eb[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double xb = X[3 * nb + i];
        eb[i] = xb - from(xb, 0);
        Ub[i] = v[3 * nb + i];
        Db[i] = vd[3 * nb + i];
    }
    const double Pb = p[nb];
    double dN[4][3], dNb[3], vol;
    {   // lane 1: e2 x e3, lane 2: e3 x e1, lane 3: e1 x e2, over det = e1 . (e2 x e3)
        double e1[3], pa[3], pb[3], cb[3], c23[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            e1[i] = from(eb[i], 1);
            pa[i] = from(eb[i], b == 2 ? 3 : b == 3 ? 1 : 2);
            pb[i] = from(eb[i], b == 2 ? 1 : b == 3 ? 2 : 3);
        }
        cross3(pa, pb, cb);
#pragma unroll
        for (int i = 0; i < 3; ++i) c23[i] = from(cb[i], 1);
        const double det = dot3(e1, c23);
        const double inv = 1.0 / det;
        vol = fabs(det) / 6.0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            cb[i] *= inv;
            dN[1][i] = from(cb[i], 1);
            dN[2][i] = from(cb[i], 2);
            dN[3][i] = from(cb[i], 3);
            dN[0][i] = -(dN[1][i] + dN[2][i] + dN[3][i]);
            dNb[i] = b == 0 ? dN[0][i] : cb[i];
        }
    }
    double D[4], GG = 0.0;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        D[a] = dot3(dN[a], dNb);
        GG += D[a] * D[a];
    }
    GG = sum4(GG);
    const double tr = sum4(pick(D[0], D[1], D[2], D[3]));
    double Gv[3][3], G2[3][3], H[4][3], kb[3], gp[3];
    {
        double row[3] = {0.0, 0.0, 0.0}, sq[3], hb[3];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const double f = pick(from(Ub[0], a), from(Ub[1], a), from(Ub[2], a), from(Pb, a));
#pragma unroll
            for (int j = 0; j < 3; ++j) row[j] += f * dN[a][j];
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
#pragma unroll
            for (int i = 0; i < 3; ++i) Gv[i][j] = from(row[j], i);
            gp[j] = from(row[j], 3);
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            sq[j] = row[0] * Gv[0][j] + row[1] * Gv[1][j] + row[2] * Gv[2][j];
            hb[j] = dNb[0] * Gv[0][j] + dNb[1] * Gv[1][j] + dNb[2] * Gv[2][j];
            kb[j] = dot3(Gv[j], dNb);
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
#pragma unroll
            for (int i = 0; i < 3; ++i) G2[i][j] = from(sq[j], i);
#pragma unroll
            for (int a = 0; a < 4; ++a) H[a][j] = from(hb[j], a);   // grad N_a . grad u
        }
    }
    // quadrature point b: s = u . grad N_a, st = (u + v') . grad N_a, 1 / (tau_M rho)
    double vp[3], s[4], st[4], tmr, SrC;
    {
        double u[3], uv[3], ss = 0.0;
#pragma unroll
        for (int i = 0; i < 3; ++i) u[i] = lo * sum4(Ub[i]) + dq * Ub[i];
#pragma unroll
        for (int a = 0; a < 4; ++a) s[a] = dot3(u, dN[a]);
        if (vt == v) {
#pragma unroll
            for (int a = 0; a < 4; ++a) ss += s[a] * s[a];
        } else {
            double ut[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const double Tb = vt[3 * nb + i];
                ut[i] = lo * sum4(Tb) + dq * Tb;
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const double x = dot3(ut, dN[a]);
                ss += x * x;
            }
        }
        const double visc2 = k.CI * (k.mu / k.rho) * (k.mu / k.rho) * (kM0 * kM0) * GG + k.CT / (k.dt * k.dt);
        const double rt = sqrt(visc2 + kM0 * ss);
        tmr = 1.0 / rt;
        SrC = sum4(rt) * (rho / (kM0 * tr));   // sum over the points of tau_C
        const double tm = tmr / rho;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double ud = lo * sum4(Db[i]) + dq * Db[i];
            vp[i] = -(tmr * (ud + dot3(Gv[i], u)) + tm * gp[i]);
            uv[i] = u[i] + vp[i];
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) st[a] = dot3(uv, dN[a]);
    }
    // sums over the points; N_a is lo + dq at point a and lo elsewhere
    double E4[4], F4[4], H4[4], K4[4], L4[4] = {}, V1[3] = {}, V2[3] = {}, Vg[3] = {};
    double Es[4] = {}, Fs[4] = {}, Sa = 0.0, Sb = 0.0, Sg = 0.0, Scn = 0.0, Sed = 0.0;
    const double w = vol * 0.25;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        double sq[4], tq[4], vq[3];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            sq[a] = from(s[a], q);
            tq[a] = from(st[a], q);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) vq[i] = from(vp[i], q);
        const double tm = from(tmr, q);
        const double Nb = b == q ? kQHi : kQLo;
        const double sb = pick(sq[0], sq[1], sq[2], sq[3]), stb = pick(tq[0], tq[1], tq[2], tq[3]);
        const double amN = am * Nb, cN = c * Nb;
        const double al = -tm * (amN + c * sb), be = -tm * cN, ga = -tm;   // gamma without its factor c / rho
        const double cn = cN + al, ed = amN + c * stb;
        Sa += al;
        Sb += be;
        Sg += ga;
        Scn += cn;
        Sed += ed;
        E4[q] = ed;
        F4[q] = cn;
        H4[q] = be;
        K4[q] = ga;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            V1[i] += cn * vq[i];
            V2[i] += be * vq[i];
            Vg[i] += ga * vq[i];
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            Es[a] += al * tq[a];
            Fs[a] += be * tq[a];
            L4[a] += ga * tq[a];
        }
    }
    double dm[3], bm[3];
    const double rw = rho * w, tc = w * c * SrC, mc = mu * c * vol, cw = c * w, gw = c / rho * w;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        dm[i] = mc * dNb[i] - rw * V1[i];
        bm[i] = -rw * V2[i];
        Vg[i] *= cw;
    }
    Sa *= w;
    Sb *= w;
    Sg *= gw;
    Scn *= lo;
    Sed *= lo;
    if (!live) return;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        double o[16];
        const double f = rw * (Scn + dq * F4[a] - Fs[a]), diag = rw * (Sed + dq * E4[a] - Es[a]) + mc * D[a];
        const double g = rho * (lo * Sb + w * (dq * H4[a])), kk = rho * (lo * Sg + gw * (dq * K4[a])), ll = cw * L4[a];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double ti = tc * dN[a][i];
#pragma unroll
            for (int j = 0; j < 3; ++j)
                o[4 * i + j] = f * Gv[i][j] + g * G2[i][j] + ti * dNb[j] + dm[i] * dN[a][j] + bm[i] * H[a][j] +
                               (i == j ? diag : 0.0);
            o[4 * i + 3] = kk * kb[i] - cw * dN[a][i] - ll * dNb[i] - D[a] * Vg[i];
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) o[12 + j] = cw * dNb[j] - (Sa * dN[a][j] + Sb * H[a][j]);
        o[15] = -Sg * D[a];
        double *out = Ke + 16LL * (16LL * e + 4 * a + b);
#pragma unroll
        for (int q = 0; q < 16; q += 4) st32(out + q, o + q);
    }
}

template <typename T>
__global__ void k_tan_tri(int Tn, const double *X, const int *tris, const double *v, VmsConst k, T *Kf) {
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= 3LL * Tn) return;
    const int t = (int)(tid / 3), b = (int)(tid % 3);
    int nd[3];
    for (int a = 0; a < 3; ++a) nd[a] = tris[3LL * t + a];
    D4<T> U[3][3], Rm[3][3];
    for (int c = 0; c < 3; ++c)
        for (int i = 0; i < 3; ++i) U[c][i] = Num<D4<T>>::cst((T)v[3LL * nd[c] + i]);
    for (int i = 0; i < 3; ++i) U[b][i].d[i] = (T)k.c;
    tri_rows<D4<T>>(k, X, nd, U, Rm);
    for (int a = 0; a < 3; ++a) {
        T *o = Kf + 9LL * (9LL * t + 3 * a + b);
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) o[3 * i + j] = Rm[a][i].d[j];
    }
}

// Pattern slot s (row A, column B): sum of its tet blocks (ascending e) and
// triangle blocks (ascending t), then the Dirichlet rules: A keeps only the
// diagonal entries of Dirichlet rows/columns, B rows and C columns of
// Dirichlet nodes are zero.
// Four lanes per slot, lane i the i-th row of the 4x4 block: the quad reads a
// source block as one contiguous segment (one thread per slot read 16 values
// one by one, 64 or 128 bytes apart between neighbours) and each value is
// still summed by one thread in the same order.  2,063,265 slots, before ->
// now: FP32 2.80 -> 1.95 ms (its conversions to FP64 hold the narrow pipe),
// FP64 1.60 -> 1.02 ms.
__device__ __forceinline__ void add4(const float *p, double acc[4]) {
    const float4 u = __ldg(reinterpret_cast<const float4 *>(p));
    acc[0] += (double)u.x;
    acc[1] += (double)u.y;
    acc[2] += (double)u.z;
    acc[3] += (double)u.w;
}
__device__ __forceinline__ void add4(const double *p, double acc[4]) {
    const double2 u = __ldg(reinterpret_cast<const double2 *>(p)), t = __ldg(reinterpret_cast<const double2 *>(p) + 1);
    acc[0] += u.x;
    acc[1] += u.y;
    acc[2] += t.x;
    acc[3] += t.y;
}
template <typename T>
__global__ void __launch_bounds__(256) k_tan_gather(long long nnz, const int *slot_row, const int *col,
                                                    const int *sl_ptr, const int *sl_src, const int *fl_ptr,
                                                    const int *fl_src, const T *Ke, const T *Kf, const uint8_t *dir,
                                                    double *Av, double *Bv, double *Cv, double *Dv) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x, s = t >> 2;
    if (s >= nnz) return;
    const int i = (int)(t & 3);
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const int j1 = sl_ptr[s + 1];
#pragma unroll 4
    for (int j = sl_ptr[s]; j < j1; ++j) add4(Ke + 16LL * sl_src[j] + 4 * i, acc);
    if (i < 3)
        for (int j = fl_ptr[s]; j < fl_ptr[s + 1]; ++j) {
            const T *o = Kf + 9LL * fl_src[j] + 3 * i;
            for (int jj = 0; jj < 3; ++jj) acc[jj] += (double)o[jj];
        }
    const int A = slot_row[s], Bn = col[s];
    const bool dA = dir[A] != 0, dB = dir[Bn] != 0;
    if (i < 3) {
        for (int j = 0; j < 3; ++j) {
            const bool keep = (A == Bn && i == j) || (!dA && !dB);
            Av[9 * s + 3 * i + j] = keep ? acc[j] : 0.0;
        }
        Bv[3 * s + i] = dA ? 0.0 : acc[3];
    } else {
        for (int j = 0; j < 3; ++j) Cv[3 * s + j] = dB ? 0.0 : acc[j];
        Dv[s] = acc[3];
    }
}

// ------------------------------------------------------------------ launchers
void vms_residual(const VmsDev &m, const VmsConst &k, const double *vd, const double *v, const double *p,
                  const double *vtau, int n_out, const int *lr_rp, const int *lr_k, const int *lr_c,
                  const double *lr_v, const double *P, double *R, cudaStream_t s) {
    const double *vt = vtau ? vtau : v;
    if (m.E > 0) {
        k_res_tet<<<(m.E + 127) / 128, 128, 0, s>>>(m.E, m.X, m.tets, vd, v, p, vt, k, m.Re);
        NBP_LAUNCHED();
    }
    if (m.T > 0) {
        k_res_tri<<<(m.T + 127) / 128, 128, 0, s>>>(m.T, m.X, m.tris, v, k, m.Rf);
        NBP_LAUNCHED();
    }
    k_res_gather<<<(m.N + 255) / 256, 256, 0, s>>>(m.N, m.n2t_ptr, m.n2t, m.n2f_ptr, m.n2f, m.Re, m.Rf,
                                                    n_out > 0 ? lr_rp : nullptr, lr_k, lr_c, lr_v,
                                                    n_out > 0 ? P : nullptr, m.dir, R);
    NBP_LAUNCHED();
}

template <typename T>
static void tangent_t(const VmsDev &m, const VmsConst &k, const double *vd, const double *v, const double *p,
                      const double *vt, double *A, double *B, double *C, double *D, cudaStream_t s) {
    T *Ke = (T *)m.Ke, *Kf = (T *)m.Kf;
    if (m.E > 0) {
        const unsigned grid = (unsigned)((4LL * m.E + 127) / 128);
        if constexpr (sizeof(T) == 8) k_tan_tet64<<<grid, 128, 0, s>>>(m.E, m.X, m.tets, vd, v, p, vt, k, Ke);
        else k_tan_tet<T><<<grid, 128, 0, s>>>(m.E, m.X, m.tets, vd, v, p, vt, k, Ke);
        NBP_LAUNCHED();
    }
    if (m.T > 0) {
        k_tan_tri<T><<<(unsigned)((3LL * m.T + 127) / 128), 128, 0, s>>>(m.T, m.X, m.tris, v, k, Kf);
        NBP_LAUNCHED();
    }
    if (m.nnz > 0) {
        k_tan_gather<T><<<(unsigned)((4LL * m.nnz + 255) / 256), 256, 0, s>>>(m.nnz, m.slot_row, m.col, m.sl_ptr, m.sl_src,
                                                                        m.fl_ptr, m.fl_src, Ke, Kf, m.dir, A, B, C, D);
        NBP_LAUNCHED();
    }
}

void vms_tangent(const VmsDev &m, const VmsConst &k, const double *vd, const double *v, const double *p,
                 const double *vtau, double *A, double *B, double *C, double *D, cudaStream_t s) {
    const double *vt = vtau ? vtau : v;
    if (m.tangent_fp32) tangent_t<float>(m, k, vd, v, p, vt, A, B, C, D, s);
    else tangent_t<double>(m, k, vd, v, p, vt, A, B, C, D, s);
}

}  // namespace nbp
