// solid.cu -- the immersed hyperelastic solid of Sec. 2.2 on a Q1 hexahedral
// solid mesh (Eq. solid_weak_form):
//
//   R^s_a = sum_g N_a (rho_s - rho_f)(uddot(g) - f) detJ0            (inertia)
//         + sum_g P(F) grad_X N_a detJ0                              (int grad w : sigma)
//         - sum_g 2 mu_f D grad_x N_a J detJ0                        (artificial fluid)
//
// with the compressible neo-Hookean P = mu (F - F^-T) + lam ln J F^-T, 2x2x2
// Gauss points in the reference configuration, D the symmetric velocity
// gradient of the solid's own velocity field on the configuration at the
// start of the step (frozen like C), and generalized-alpha / Newmark
// kinematics: the residual is taken at uddot_{n+alpha_m}, v_{n+alpha_f},
// u_{n+alpha_f}, all functions of uddot_{n+1} = C^T Vdot_{n+1} (the solid
// nodes are the Lagrange multiplier points, Sec. 2.3).  The linearisation
// w.r.t. uddot_{n+1} carries the chain factors alpha_m (inertia),
// alpha_f beta dt^2 (stress), alpha_f gamma dt (viscous).
//
// GPU layout: eight lanes per element; lane a is first "node a" (it loads the
// node's record) and then "Gauss point a".  On the trilinear map values and
// parent gradients follow from the nodal values by three butterfly stages over
// the lane bits, and the projection onto the test functions is the transposed
// butterfly.  All stresses are taken in the Kirchhoff form tau = P F^T, so that
// one inverse per configuration, K = (dx/dxi)^-1 at the alpha level and Kn at the
// start of the step, serves every gradient and every test function: the
// reference configuration enters through det J0 and F = dx/dxi J0^-1 only.  With
// H = grad_x(w) = (dw/dxi) K of the direction w,
//
//   tau       = mu (b - I) + lam ln J I,                    b = F F^T,
//   dP F^T    = c_u (mu H b + (mu - lam ln J) H^T + lam tr H I).
//
// What the tangent needs of the state (K, Kn, mu b, mu - lam ln J, the viscous
// scale, det J0: 27 values per Gauss point) is formed once per linearisation into
// a table; a tangent apply reads it.  Contributions go to an element scratch
// [es][8][3]; each node then sums its element slots through a node -> (element,
// corner) table in a fixed order.  No atomics; deterministic.
//
// Bound: the FP64 pipe (2 operations per SM and clock).  One thread per element,
// which formed dN/dX, F, F^-1 and both configurations' gradients of all 8 nodes at
// every point of every apply, took 584 us per FP64 tangent apply of 20,736
// hexahedra; an FP64 implicit step with that body on a 24^3 grid went from 76 to
// 38 ms with this form.
#include <cmath>
#include <vector>

#include "fsi_internal.cuh"

struct fsi_solid {
    fsi_mesh *mesh;
    int64_t ns, es;
    double *X;           // [ns][3] reference coordinates
    int32_t *conn;       // [es][8]
    int32_t *node_start; // [ns+1] CSR of element slots e*8+a per node
    int32_t *node_slot;  // [es*8]
    void *elem_f;        // [es][8][3] scratch, 8 bytes per value
    void *state;         // [es][27][8] state of the tangent, 8 bytes per value
    double rho_s, mu_s, lam_s;
};

namespace fsi {
namespace {

template <typename T> struct M3 {
    T a[3][3];
};

template <typename T> __device__ __forceinline__ T det3(const M3<T> &m)
{
    return m.a[0][0] * (m.a[1][1] * m.a[2][2] - m.a[1][2] * m.a[2][1]) -
           m.a[0][1] * (m.a[1][0] * m.a[2][2] - m.a[1][2] * m.a[2][0]) +
           m.a[0][2] * (m.a[1][0] * m.a[2][1] - m.a[1][1] * m.a[2][0]);
}

// inverse by cofactors; returns the determinant
template <typename T> __device__ __forceinline__ T inv3(const M3<T> &m, M3<T> &r)
{
    const T d = det3(m);
    const T id = T(1) / d;
    r.a[0][0] = (m.a[1][1] * m.a[2][2] - m.a[1][2] * m.a[2][1]) * id;
    r.a[0][1] = (m.a[0][2] * m.a[2][1] - m.a[0][1] * m.a[2][2]) * id;
    r.a[0][2] = (m.a[0][1] * m.a[1][2] - m.a[0][2] * m.a[1][1]) * id;
    r.a[1][0] = (m.a[1][2] * m.a[2][0] - m.a[1][0] * m.a[2][2]) * id;
    r.a[1][1] = (m.a[0][0] * m.a[2][2] - m.a[0][2] * m.a[2][0]) * id;
    r.a[1][2] = (m.a[0][2] * m.a[1][0] - m.a[0][0] * m.a[1][2]) * id;
    r.a[2][0] = (m.a[1][0] * m.a[2][1] - m.a[1][1] * m.a[2][0]) * id;
    r.a[2][1] = (m.a[0][1] * m.a[2][0] - m.a[0][0] * m.a[2][1]) * id;
    r.a[2][2] = (m.a[0][0] * m.a[1][1] - m.a[0][1] * m.a[1][0]) * id;
    return d;
}

template <typename T> __device__ __forceinline__ T log_t(T v);
template <> __device__ __forceinline__ double log_t(double v) { return log(v); }
template <> __device__ __forceinline__ float log_t(float v) { return logf(v); }

struct SolidArgs {
    int64_t es;
    const double *X;
    const int32_t *conn;
    double drho, mu, lam, mu_f;
    double g[3];
    double c_a, c_u, c_v;  // tangent chain factors
};

constexpr double kGq = 0.57735026918962576451;  // 1/sqrt(3)

template <typename T> __device__ __forceinline__ T shx(T v, int m)
{
    return __shfl_xor_sync(0xffffffffu, v, m);
}

// value and parent gradient at this lane's Gauss point of the trilinear field
// whose value at this lane's node is u; s[k] = +-1/2 (the node's side along xi_k)
template <typename T, bool VALUE>
__device__ __forceinline__ T eval_parent(T u, const T (&s)[3], T (&g)[3])
{
    const T b1 = T(0.5 * (1.0 + kGq));
    const T uo = shx(u, 1), tD = u - uo, tB = fma(b1, tD, uo);
    const T tBo = shx(tB, 2), tDo = shx(tD, 2), tBD = tB - tBo;
    const T tBB = fma(b1, tBD, tBo), tDB = fma(b1, tD - tDo, tDo);
    const T tBBo = shx(tBB, 4), tBDo = shx(tBD, 4), tDBo = shx(tDB, 4), d = tBB - tBBo;
    g[0] = s[0] * fma(b1, tDB - tDBo, tDBo);
    g[1] = s[1] * fma(b1, tBD - tBDo, tBDo);
    g[2] = s[2] * d;
    return VALUE ? fma(b1, d, tBBo) : T(0);
}

// transposed: sum over the Gauss points of N_a X + dN_a/dxi . Y for this lane's node
template <typename T>
__device__ __forceinline__ T project_parent(T X, T Y0, T Y1, T Y2, const T (&s)[3])
{
    const T b1 = T(0.5 * (1.0 + kGq)), b2 = T(0.5 * (1.0 - kGq));
    const T Xo = shx(X, 4), Y2o = shx(Y2, 4), Y0o = shx(Y0, 4), Y1o = shx(Y1, 4);
    const T P1 = fma(s[2], Y2 + Y2o, fma(b1, X, b2 * Xo));
    const T P2 = fma(b1, Y0, b2 * Y0o), P3 = fma(b1, Y1, b2 * Y1o);
    const T P1o = shx(P1, 2), P2o = shx(P2, 2), P3o = shx(P3, 2);
    const T Q1 = fma(s[1], P3 + P3o, fma(b1, P1, b2 * P1o));
    const T Q2 = fma(b1, P2, b2 * P2o);
    const T Q1o = shx(Q1, 1), Q2o = shx(Q2, 1);
    return fma(s[0], Q2 + Q2o, fma(b1, Q1, b2 * Q1o));
}

// the lane's place: element, corner / Gauss point, node, gradient signs
template <typename T> struct Lane {
    int64_t e;
    int node;
    bool valid;
    T s[3];
    __device__ __forceinline__ Lane(const SolidArgs &a, int64_t t)
    {
        const int g = (int)(t & 7);
        valid = (t >> 3) < a.es;
        e = valid ? t >> 3 : 0;  // idle lanes repeat element 0, unused
        node = a.conn[8 * e + g];
        for (int k = 0; k < 3; ++k) s[k] = ((g >> k) & 1) ? T(0.5) : T(-0.5);
    }
};

// Kinematics of the configuration X + u at one Gauss point from the parent
// gradient du of u: G = du/dX, K = (dx/dxi)^-1 = J0^-1 F^-1 with F = I + G;
// returns det F
template <typename T>
__device__ __forceinline__ T kinematics(const M3<T> &du, const M3<T> &J0i, M3<T> &G, M3<T> &K)
{
    M3<T> F, Fi;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            G.a[i][j] = du.a[i][0] * J0i.a[0][j] + du.a[i][1] * J0i.a[1][j] + du.a[i][2] * J0i.a[2][j];
            F.a[i][j] = (i == j ? T(1) : T(0)) + G.a[i][j];
        }
    const T J = inv3(F, Fi);
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            K.a[k][j] = J0i.a[k][0] * Fi.a[0][j] + J0i.a[k][1] * Fi.a[1][j] + J0i.a[k][2] * Fi.a[2][j];
    return J;
}

// State of one Gauss point: the two inverses, b - I (00 01 02 11 12 22), ln J,
// J_n and det J0
template <typename T> struct State {
    M3<T> K, Kn;
    T e[6], lnJ, Jn, det0;
};
template <typename T>
__device__ __forceinline__ void solid_state(const SolidArgs &a, const Lane<T> &L,
                                            const T *__restrict__ u_af,
                                            const double *__restrict__ u_n, State<T> &q)
{
    M3<T> J0, J0i, d, G;
    const int64_t n3 = 3 * (int64_t)L.node;
#pragma unroll
    for (int i = 0; i < 3; ++i) eval_parent<T, false>((T)a.X[n3 + i], L.s, J0.a[i]);
    q.det0 = inv3(J0, J0i);
#pragma unroll
    for (int i = 0; i < 3; ++i) eval_parent<T, false>((T)u_n[n3 + i], L.s, d.a[i]);
    q.Jn = kinematics(d, J0i, G, q.Kn);
#pragma unroll
    for (int i = 0; i < 3; ++i) eval_parent<T, false>(u_af[n3 + i], L.s, d.a[i]);
    q.lnJ = log_t(kinematics(d, J0i, G, q.K));
    // b - I = G + G^T + G G^T: small strains keep their digits
    int n = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j)
            q.e[n++] = (G.a[i][j] + G.a[j][i]) +
                       (G.a[i][0] * G.a[j][0] + G.a[i][1] * G.a[j][1] + G.a[i][2] * G.a[j][2]);
}

// Y = S K^T (ACC: -=), S symmetric given as 00 01 02 11 12 22
template <typename T, bool SUB>
__device__ __forceinline__ void sym_times_kt(const T (&S)[6], const M3<T> &K, M3<T> &Y)
{
    const int id[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const T s0 = S[id[i][0]], s1 = S[id[i][1]], s2 = S[id[i][2]];
            if (SUB)
                Y.a[i][k] = fma(-s2, K.a[k][2], fma(-s1, K.a[k][1], fma(-s0, K.a[k][0], Y.a[i][k])));
            else
                Y.a[i][k] = fma(s2, K.a[k][2], fma(s1, K.a[k][1], s0 * K.a[k][0]));
        }
}
// D = vs (L + L^T), L = W Kn (00 01 02 11 12 22)
template <typename T>
__device__ __forceinline__ void viscous(const M3<T> &W, const M3<T> &Kn, T vs, T (&D)[6])
{
    M3<T> L;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            L.a[i][j] = W.a[i][0] * Kn.a[0][j] + W.a[i][1] * Kn.a[1][j] + W.a[i][2] * Kn.a[2][j];
    int n = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) D[n++] = i == j ? (vs + vs) * L.a[i][i] : vs * (L.a[i][j] + L.a[j][i]);
}
template <typename T>
__device__ __forceinline__ void project_store(const Lane<T> &L, const T (&X)[3], const M3<T> &Y,
                                              T *__restrict__ ef, int64_t t)
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const T r = project_parent(X[i], Y.a[i][0], Y.a[i][1], Y.a[i][2], L.s);
        if (L.valid) ef[3 * t + i] = r;
    }
}

// residual from (u_af, v_af, a_am, u_n), FP64
__global__ void __launch_bounds__(128)
    solid_residual_kernel(SolidArgs s, const double *__restrict__ u_af, const double *__restrict__ v_af,
                          const double *__restrict__ a_am, const double *__restrict__ u_n,
                          double *__restrict__ ef)
{
    using T = double;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const Lane<T> L(s, t);
    State<T> q;
    solid_state<T>(s, L, u_af, u_n, q);
    T S[6];
    const T m0 = q.det0 * s.mu, l0 = q.det0 * s.lam * q.lnJ;
#pragma unroll
    for (int n = 0; n < 6; ++n) S[n] = m0 * q.e[n] + (n == 0 || n == 3 || n == 5 ? l0 : T(0));
    M3<T> Y, W;
    sym_times_kt<T, false>(S, q.K, Y);
    const int64_t n3 = 3 * (int64_t)L.node;
#pragma unroll
    for (int i = 0; i < 3; ++i) eval_parent<T, false>(v_af[n3 + i], L.s, W.a[i]);
    viscous(W, q.Kn, q.det0 * s.mu_f * q.Jn, S);
    sym_times_kt<T, true>(S, q.Kn, Y);
    T X[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        T g[3];
        X[i] = q.det0 * s.drho * (eval_parent<T, true>(a_am[n3 + i], L.s, g) - s.g[i]);
    }
    project_store(L, X, Y, ef, t);
}

// The tangent's state table, [element][value][Gauss point]: K, Kn, c_u mu b,
// c_u (mu - lam ln J), c_v mu_f J_n and det J0, the stress terms times det J0
constexpr int kState = 27;
template <typename T>
__global__ void __launch_bounds__(128)
    solid_state_kernel(SolidArgs s, const T *__restrict__ u_af, const double *__restrict__ u_n,
                       T *__restrict__ tab)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const Lane<T> L(s, t);
    State<T> q;
    solid_state<T>(s, L, u_af, u_n, q);
    if (!L.valid) return;  // after the last shuffle
    T *o = tab + L.e * (8 * kState) + (t & 7);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        o[8 * k] = q.K.a[k / 3][k % 3];
        o[8 * (9 + k)] = q.Kn.a[k / 3][k % 3];
    }
    const T cu = (T)s.c_u * q.det0, m0 = cu * (T)s.mu;
#pragma unroll
    for (int n = 0; n < 6; ++n)
        o[8 * (18 + n)] = m0 * (q.e[n] + (n == 0 || n == 3 || n == 5 ? T(1) : T(0)));
    o[8 * 24] = m0 - cu * (T)s.lam * q.lnJ;
    o[8 * 25] = q.det0 * (T)(s.c_v * s.mu_f) * q.Jn;
    o[8 * 26] = q.det0;
}

// tangent apply along x from the state table
template <typename T>
__global__ void __launch_bounds__(128)
    solid_tangent_kernel(SolidArgs s, const T *__restrict__ tab, const T *__restrict__ x,
                         T *__restrict__ ef)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const Lane<T> L(s, t);
    const T *o = tab + L.e * (8 * kState) + (t & 7);
    M3<T> W, K, H, Y;
    T X[3];
    const T det0 = __ldg(o + 8 * 26);
    const int64_t n3 = 3 * (int64_t)L.node;
#pragma unroll
    for (int i = 0; i < 3; ++i)
        X[i] = (T)(s.c_a * s.drho) * det0 * eval_parent<T, true>(x[n3 + i], L.s, W.a[i]);
    // stress: S = mu H b + (mu - lam ln J) H^T + lam tr H I, H = W K
#pragma unroll
    for (int k = 0; k < 9; ++k) K.a[k / 3][k % 3] = __ldg(o + 8 * k);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            H.a[i][j] = W.a[i][0] * K.a[0][j] + W.a[i][1] * K.a[1][j] + W.a[i][2] * K.a[2][j];
    T b[6];
#pragma unroll
    for (int n = 0; n < 6; ++n) b[n] = __ldg(o + 8 * (18 + n));
    const T c1 = __ldg(o + 8 * 24);
    const T tr = (T)(s.c_u * s.lam) * det0 * (H.a[0][0] + H.a[1][1] + H.a[2][2]);
    M3<T> S;
    const int id[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            T v = c1 * H.a[j][i];
            if (i == j) v += tr;
#pragma unroll
            for (int k = 0; k < 3; ++k) v = fma(H.a[i][k], b[id[k][j]], v);
            S.a[i][j] = v;
        }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k)
            Y.a[i][k] = S.a[i][0] * K.a[k][0] + S.a[i][1] * K.a[k][1] + S.a[i][2] * K.a[k][2];
    // artificial fluid, on the configuration at the start of the step
#pragma unroll
    for (int k = 0; k < 9; ++k) K.a[k / 3][k % 3] = __ldg(o + 8 * (9 + k));
    T D[6];
    viscous(W, K, __ldg(o + 8 * 25), D);
    sym_times_kt<T, true>(D, K, Y);
    project_store(L, X, Y, ef, t);
}

// R_b = sum of the element slots of node b (fixed order), overwrite
template <typename T>
__global__ void solid_gather_kernel(int64_t ns, const int32_t *__restrict__ start,
                                    const int32_t *__restrict__ slot, const T *__restrict__ ef,
                                    T *__restrict__ R)
{
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < ns;
         b += (int64_t)gridDim.x * blockDim.x) {
        T r0 = T(0), r1 = T(0), r2 = T(0);
        for (int q = start[b]; q < start[b + 1]; ++q) {
            const T *p = ef + 3 * (int64_t)slot[q];
            r0 += p[0];
            r1 += p[1];
            r2 += p[2];
        }
        R[3 * b] = r0;
        R[3 * b + 1] = r1;
        R[3 * b + 2] = r2;
    }
}

// generalized-alpha / Newmark stage values from uddot_{n+1}
__global__ void solid_stage_kernel(int64_t n3, double dt, double am, double af, double gm,
                                   double beta, const double *u, const double *v, const double *a,
                                   const double *a1, double *u_af, double *v_af, double *a_am)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n3;
         q += (int64_t)gridDim.x * blockDim.x) {
        const double v1 = v[q] + dt * ((1.0 - gm) * a[q] + gm * a1[q]);
        const double u1 = u[q] + dt * v[q] + dt * dt * ((0.5 - beta) * a[q] + beta * a1[q]);
        u_af[q] = u[q] + af * (u1 - u[q]);
        v_af[q] = v[q] + af * (v1 - v[q]);
        a_am[q] = a[q] + am * (a1[q] - a[q]);
    }
}

// history advance: (u, v, a) <- (u_{n+1}, v_{n+1}, uddot_{n+1})
__global__ void solid_advance_kernel(int64_t n3, double dt, double gm, double beta, double *u,
                                     double *v, double *a, const double *a1)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n3;
         q += (int64_t)gridDim.x * blockDim.x) {
        const double v1 = v[q] + dt * ((1.0 - gm) * a[q] + gm * a1[q]);
        const double u1 = u[q] + dt * v[q] + dt * dt * ((0.5 - beta) * a[q] + beta * a1[q]);
        u[q] = u1;
        v[q] = v1;
        a[q] = a1[q];
    }
}

__global__ void positions_kernel(int64_t n3, const double *X, const double *u, double *x)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n3;
         q += (int64_t)gridDim.x * blockDim.x)
        x[q] = X[q] + u[q];
}

int grid_of(int64_t n, int threads = 128)
{
    const int64_t b = (n + threads - 1) / threads;
    return (int)(b < 1 ? 1 : (b > sm_count() * 32 ? sm_count() * 32 : b));
}

// eight lanes per element, 16 elements per CTA
int lanes_grid(const fsi_solid *b) { return (int)((b->es + 15) / 16); }

SolidArgs args_of(const fsi_solid *b, const double g[3])
{
    const fsi_mesh *m = b->mesh;
    SolidArgs s;
    s.es = b->es;
    s.X = b->X;
    s.conn = b->conn;
    s.drho = b->rho_s - m->phys.rho;
    s.mu = b->mu_s;
    s.lam = b->lam_s;
    s.mu_f = m->phys.mu;
    for (int i = 0; i < 3; ++i) s.g[i] = g ? g[i] : 0.0;
    const double beta = 0.25 * (1.0 + m->alpha_m - m->alpha_f) * (1.0 + m->alpha_m - m->alpha_f);
    const double dt = m->phys.dt;
    s.c_a = m->alpha_m;
    s.c_u = m->alpha_f * beta * dt * dt;
    s.c_v = m->alpha_f * m->gamma * dt;
    return s;
}

}  // namespace

// ---------------------------------------------------------------- internal API
fsi_status solid_residual_impl(fsi_solid *b, const double *u_af, const double *v_af,
                               const double *a_am, const double *u_n, const double g[3], double *R)
{
    cudaStream_t s = b->mesh->stream;
    solid_residual_kernel<<<lanes_grid(b), 128, 0, s>>>(args_of(b, g), u_af, v_af, a_am, u_n,
                                                       (double *)b->elem_f);
    FSI_TRY(check_launch("solid element kernel"));
    solid_gather_kernel<double><<<grid_of(b->ns, 256), 256, 0, s>>>(
        b->ns, b->node_start, b->node_slot, (const double *)b->elem_f, R);
    return check_launch("solid gather kernel");
}

// the tangent's state at (u_af, u_n) into the body's table
template <typename T> fsi_status solid_linearise(fsi_solid *b, const T *u_af, const double *u_n)
{
    solid_state_kernel<T><<<lanes_grid(b), 128, 0, b->mesh->stream>>>(args_of(b, nullptr), u_af, u_n,
                                                                     (T *)b->state);
    return check_launch("solid state kernel");
}
// Jx = tangent x at the state of the last solid_linearise (same T)
template <typename T> fsi_status solid_tangent_impl(fsi_solid *b, const T *x, T *Jx)
{
    cudaStream_t s = b->mesh->stream;
    solid_tangent_kernel<T><<<lanes_grid(b), 128, 0, s>>>(args_of(b, nullptr), (const T *)b->state, x,
                                                         (T *)b->elem_f);
    FSI_TRY(check_launch("solid element kernel"));
    solid_gather_kernel<T><<<grid_of(b->ns, 256), 256, 0, s>>>(
        b->ns, b->node_start, b->node_slot, (const T *)b->elem_f, Jx);
    return check_launch("solid gather kernel");
}
template fsi_status solid_linearise<double>(fsi_solid *, const double *, const double *);
template fsi_status solid_linearise<float>(fsi_solid *, const float *, const double *);
template fsi_status solid_tangent_impl<double>(fsi_solid *, const double *, double *);
template fsi_status solid_tangent_impl<float>(fsi_solid *, const float *, float *);

fsi_status solid_stage_impl(fsi_solid *b, const double *u, const double *v, const double *a,
                            const double *a1, double *u_af, double *v_af, double *a_am)
{
    const fsi_mesh *m = b->mesh;
    const double beta = 0.25 * (1.0 + m->alpha_m - m->alpha_f) * (1.0 + m->alpha_m - m->alpha_f);
    solid_stage_kernel<<<grid_of(3 * b->ns, 256), 256, 0, m->stream>>>(
        3 * b->ns, m->phys.dt, m->alpha_m, m->alpha_f, m->gamma, beta, u, v, a, a1, u_af, v_af,
        a_am);
    return check_launch("solid stage kernel");
}

int64_t solid_nodes(const fsi_solid *b) { return b->ns; }

}  // namespace fsi

// ---------------------------------------------------------------- C ABI
using namespace fsi;

extern "C" {

fsi_status fsi_solid_create(fsi_mesh *mesh, int64_t n_nodes, int64_t n_elems, const double *X,
                            const int32_t *conn, double rho_s, double mu_s, double lambda_s,
                            fsi_solid **out)
{
    FSI_TRY(validate_mesh(mesh));
    if (!out) return set_error(FSI_ERR_ARG, "fsi_solid_create: out is NULL");
    *out = nullptr;
    if (n_nodes < 1 || n_elems < 1 || n_nodes > INT32_MAX / 3 || n_elems > INT32_MAX / 8)
        return set_error(FSI_ERR_ARG, "fsi_solid_create: sizes out of range");
    if (!X || !conn) return set_error(FSI_ERR_ARG, "fsi_solid_create: NULL array");
    if (!(rho_s > 0.0) || !(mu_s > 0.0) || !(lambda_s >= 0.0))
        return set_error(FSI_ERR_ARG, "fsi_solid_create: rho_s, mu_s > 0 and lambda_s >= 0");
    FSI_DEVICE(mesh->device);
    // node -> element-slot table, built on the host from the connectivity
    std::vector<int32_t> hconn((size_t)n_elems * 8);
    FSI_CUDA(cudaMemcpy(hconn.data(), conn, hconn.size() * sizeof(int32_t), cudaMemcpyDeviceToHost),
             "memcpy");
    std::vector<int32_t> start((size_t)n_nodes + 1, 0), slot(hconn.size());
    for (int32_t v : hconn) {
        if (v < 0 || v >= n_nodes)
            return set_error(FSI_ERR_ARG, "fsi_solid_create: connectivity entry %d out of range", v);
        start[(size_t)v + 1]++;
    }
    for (int64_t b = 0; b < n_nodes; ++b) start[b + 1] += start[b];
    {
        std::vector<int32_t> fill(start.begin(), start.end() - 1);
        for (size_t q = 0; q < hconn.size(); ++q) slot[fill[hconn[q]]++] = (int32_t)q;
    }
    fsi_solid *b = new (std::nothrow) fsi_solid();
    if (!b) return set_error(FSI_ERR_OOM, "host allocation failed");
    b->mesh = mesh;
    b->ns = n_nodes;
    b->es = n_elems;
    b->rho_s = rho_s;
    b->mu_s = mu_s;
    b->lam_s = lambda_s;
    struct {
        void **p;
        size_t bytes;
    } req[] = {{(void **)&b->X, (size_t)n_nodes * 3 * sizeof(double)},
               {(void **)&b->conn, hconn.size() * sizeof(int32_t)},
               {(void **)&b->node_start, start.size() * sizeof(int32_t)},
               {(void **)&b->node_slot, slot.size() * sizeof(int32_t)},
               {&b->elem_f, (size_t)n_elems * 24 * sizeof(double)},
               {&b->state, (size_t)n_elems * 8 * kState * sizeof(double)}};
    for (auto &r : req) {
        if (cudaMalloc(r.p, r.bytes) != cudaSuccess) {
            cudaGetLastError();
            fsi_solid_destroy(b);
            return set_error(FSI_ERR_OOM, "fsi_solid_create: cudaMalloc failed");
        }
    }
    cudaError_t e = cudaMemcpy(b->X, X, (size_t)n_nodes * 3 * sizeof(double), cudaMemcpyDeviceToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b->conn, conn, hconn.size() * sizeof(int32_t), cudaMemcpyDeviceToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b->node_start, start.data(), start.size() * sizeof(int32_t),
                       cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b->node_slot, slot.data(), slot.size() * sizeof(int32_t),
                       cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        fsi_solid_destroy(b);
        return check_cuda(e, "fsi_solid_create: copy");
    }
    *out = b;
    return FSI_OK;
}

void fsi_solid_destroy(fsi_solid *b)
{
    if (!b) return;
    fsi::DeviceGuard _fsi_device_guard(b->mesh->device);
    cudaStreamSynchronize(b->mesh->stream);
    cudaFree(b->X);
    cudaFree(b->conn);
    cudaFree(b->node_start);
    cudaFree(b->node_slot);
    cudaFree(b->elem_f);
    cudaFree(b->state);
    delete b;
}

fsi_status fsi_solid_residual(fsi_solid *b, const double *u_af, const double *v_af,
                              const double *a_am, const double *u_n, const double *g, double *R)
{
    if (!b) return set_error(FSI_ERR_ARG, "fsi_solid_residual: solid is NULL");
    if (!u_af || !v_af || !a_am || !u_n || !R)
        return set_error(FSI_ERR_ARG, "fsi_solid_residual: NULL argument");
    FSI_DEVICE(b->mesh->device);
    return solid_residual_impl(b, u_af, v_af, a_am, u_n, g, R);
}

fsi_status fsi_solid_tangent_apply(fsi_solid *b, fsi_prec prec, const void *u_af, const double *u_n,
                                   const void *x, void *Jx)
{
    if (!b) return set_error(FSI_ERR_ARG, "fsi_solid_tangent_apply: solid is NULL");
    if (!u_af || !u_n || !x || !Jx)
        return set_error(FSI_ERR_ARG, "fsi_solid_tangent_apply: NULL argument");
    if (prec != FSI_F64 && prec != FSI_F32) return set_error(FSI_ERR_ARG, "bad precision");
    FSI_DEVICE(b->mesh->device);
    if (prec == FSI_F64) {
        FSI_TRY(solid_linearise<double>(b, (const double *)u_af, u_n));
        return solid_tangent_impl<double>(b, (const double *)x, (double *)Jx);
    }
    FSI_TRY(solid_linearise<float>(b, (const float *)u_af, u_n));
    return solid_tangent_impl<float>(b, (const float *)x, (float *)Jx);
}

fsi_status fsi_solid_stage(fsi_solid *b, const double *u, const double *v, const double *a,
                           const double *a_next, double *u_af, double *v_af, double *a_am)
{
    if (!b || !u || !v || !a || !a_next || !u_af || !v_af || !a_am)
        return set_error(FSI_ERR_ARG, "fsi_solid_stage: NULL argument");
    FSI_DEVICE(b->mesh->device);
    return solid_stage_impl(b, u, v, a, a_next, u_af, v_af, a_am);
}

fsi_status fsi_solid_advance(fsi_solid *b, double *u, double *v, double *a, const double *a_next)
{
    if (!b || !u || !v || !a || !a_next)
        return set_error(FSI_ERR_ARG, "fsi_solid_advance: NULL argument");
    FSI_DEVICE(b->mesh->device);
    const fsi_mesh *m = b->mesh;
    const double beta = 0.25 * (1.0 + m->alpha_m - m->alpha_f) * (1.0 + m->alpha_m - m->alpha_f);
    solid_advance_kernel<<<grid_of(3 * b->ns, 256), 256, 0, m->stream>>>(
        3 * b->ns, m->phys.dt, m->gamma, beta, u, v, a, a_next);
    return check_launch("solid advance kernel");
}

fsi_status fsi_solid_positions(fsi_solid *b, const double *u, double *x)
{
    if (!b || !u || !x) return set_error(FSI_ERR_ARG, "fsi_solid_positions: NULL argument");
    FSI_DEVICE(b->mesh->device);
    positions_kernel<<<grid_of(3 * b->ns, 256), 256, 0, b->mesh->stream>>>(3 * b->ns, b->X, u, x);
    return check_launch("solid positions kernel");
}

}  // extern "C"
