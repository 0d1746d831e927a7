// vms_device.cuh -- per-work-item device code of the VMS operators, shared by
// the single-mesh kernels (vms.cu) and the batched persistent kernels
// (batch.cu).  See vms.cu for the design.
#pragma once

#include <type_traits>

#include "df64.cuh"
#include "fsi_internal.cuh"
#include "pairs.cuh"

namespace fsi {
namespace vmsd {

constexpr double kQ = 0.57735026918962576451;  // 1/sqrt(3): Gauss abscissa
constexpr double kB1 = 0.5 * (1.0 + kQ);      // 1D linear basis at the near point
constexpr double kB2 = 0.5 * (1.0 - kQ);      // ... at the far point
// the same constants as exact float pairs (split at compile time)
constexpr float kB1h = static_cast<float>(kB1);
constexpr float kB1l = static_cast<float>(kB1 - static_cast<double>(kB1h));
constexpr float kB2h = static_cast<float>(kB2);
constexpr float kB2l = static_cast<float>(kB2 - static_cast<double>(kB2h));

template <typename T> __device__ __forceinline__ T cB1() { return T(kB1); }
template <typename T> __device__ __forceinline__ T cB2() { return T(kB2); }
template <> __device__ __forceinline__ df64 cB1<df64>() { return df64(kB1h, kB1l); }
template <> __device__ __forceinline__ df64 cB2<df64>() { return df64(kB2h, kB2l); }

// record that the kernel before in the chain wrote, in compute type (double-float:
// two float4 loads)
template <typename T> __device__ __forceinline__ vec4<T> ld4_blk(const vec4<T> *p)
{
    return ld4_chain(p);
}
template <> __device__ __forceinline__ vec4<df64> ld4_blk<df64>(const vec4<df64> *p)
{
    const float4 *q = reinterpret_cast<const float4 *>(p);
    const float4 a = ldg_chain(q), b = ldg_chain(q + 1);
    return {df64(a.x, a.y), df64(a.z, a.w), df64(b.x, b.y), df64(b.z, b.w)};
}

// Per-Gauss-point geometry of a mapped grid, built once per coordinate set and
// compute type and read by the VMS kernels: Ji[9] (row-major), G00 G01 G02 G11
// G12 G22, G:G, 1/tr G, det J.  Layout [element][value][Gauss point], so the 8
// lanes of an element read 8 consecutive entries per value.  Double-float
// entries are stored as (hi, lo) float pairs.
constexpr int kMapGeo = 18;
template <typename T> struct GeoStore {
    using type = T;
};
template <> struct GeoStore<df64> {
    using type = float2;
};
template <typename T> __device__ __forceinline__ T geo_ld(const typename GeoStore<T>::type *p)
{
    return __ldg(p);
}
template <> __device__ __forceinline__ df64 geo_ld<df64>(const float2 *p)
{
    const float2 v = __ldg(p);
    return df64(v.x, v.y);
}
template <typename T> __device__ __forceinline__ typename GeoStore<T>::type geo_st(T v) { return v; }
template <> __device__ __forceinline__ float2 geo_st<df64>(df64 v) { return make_float2(v.hi, v.lo); }

template <typename T> struct VmsArgs {
    using S = typename StorageOf<T>::type;
    int Nx, Ny, Nz;
    int bx, by, bz;
    int nbx, nby, nbz;
    T rho, mu, inv_rho;
    T G0, G1, G2, inv_trG, q0;  // q0 = C_T/dt^2 + C_I (mu/rho)^2 G:G
    T ih0, ih1, ih2;            // 1/h_k
    T detJ, rdetJ;              // det J and rho det J of the uniform grid
    T nu, nu2;                  // mu / rho and twice that
    T c_a, c_v;                 // d A / d y_v, d U / d y_v
    T c_av;                     // c_a / c_v
    T ct_dt2, CInu2;            // C_T/dt^2 and C_I (mu/rho)^2 (mapped grids: G per Gauss point)
    int has_s;
    const vec4<S> *Xc;          // mapped grids: node coordinates [n][4] (x, y, z, 0), else null
    const typename GeoStore<T>::type *geo;  // mapped grids: [E][kMapGeo][8] Gauss-point geometry
    const vec4<S> *U, *A, *f, *x;
    vec4<T> *blocks;  // [n_bricks][(bx+1)(by+1)(bz+1)], in the compute type
    vec4<S> *out;     // [n]
    // fused residual + Jacobian apply: the residual's node blocks and output
    vec4<T> *blocks2;
    vec4<S> *out2;
};

// a b + c and a b + c d: plain expressions (contracted to FMAs) for float and
// double, one renormalisation for double-float.
template <typename T> __device__ __forceinline__ T fma_t(T a, T b, T c) { return a * b + c; }
template <> __device__ __forceinline__ df64 fma_t<df64>(df64 a, df64 b, df64 c)
{
    return df_fma(a, b, c);
}
template <typename T> __device__ __forceinline__ T dot2_t(T a, T b, T c, T d)
{
    return a * b + c * d;
}
template <> __device__ __forceinline__ df64 dot2_t<df64>(df64 a, df64 b, df64 c, df64 d)
{
    return df_dot2(a, b, c, d);
}
// a . b over three components
template <typename T> __device__ __forceinline__ T dot3_t(T a0, T b0, T a1, T b1, T a2, T b2)
{
    return fma_t(a2, b2, dot2_t(a0, b0, a1, b1));
}

template <typename T> __device__ __forceinline__ T shx(T v, int m)
{
    return __shfl_xor_sync(0xffffffffu, v, m);
}
template <> __device__ __forceinline__ df64 shx<df64>(df64 v, int m) { return df_shfl_xor(v, m); }

// the same operations on pairs of values (pairs.cuh): two fields per call
using pd = pair2<double>;
template <> __device__ __forceinline__ f32x2 fma_t<f32x2>(f32x2 a, f32x2 b, f32x2 c)
{
    return pair_fma(a, b, c);
}
template <> __device__ __forceinline__ df64x2 fma_t<df64x2>(df64x2 a, df64x2 b, df64x2 c)
{
    return pair_fma(a, b, c);
}
template <> __device__ __forceinline__ pd fma_t<pd>(pd a, pd b, pd c) { return pair_fma(a, b, c); }
template <> __device__ __forceinline__ f32x2 dot2_t<f32x2>(f32x2 a, f32x2 b, f32x2 c, f32x2 d)
{
    return pair_dot2(a, b, c, d);
}
template <>
__device__ __forceinline__ df64x2 dot2_t<df64x2>(df64x2 a, df64x2 b, df64x2 c, df64x2 d)
{
    return pair_dot2(a, b, c, d);
}
template <> __device__ __forceinline__ pd dot2_t<pd>(pd a, pd b, pd c, pd d)
{
    return pair_dot2(a, b, c, d);
}
template <> __device__ __forceinline__ f32x2 shx<f32x2>(f32x2 v, int m) { return pair_shx(v, m); }
template <> __device__ __forceinline__ df64x2 shx<df64x2>(df64x2 v, int m) { return pair_shx(v, m); }
template <> __device__ __forceinline__ pd shx<pd>(pd v, int m) { return pair_shx(v, m); }
template <> __device__ __forceinline__ f32x2 cB1<f32x2>()
{
    return {make_float2((float)kB1, (float)kB1)};
}
template <> __device__ __forceinline__ f32x2 cB2<f32x2>()
{
    return {make_float2((float)kB2, (float)kB2)};
}
template <> __device__ __forceinline__ df64x2 cB1<df64x2>()
{
    return {make_float2(kB1h, kB1h), make_float2(kB1l, kB1l)};
}
template <> __device__ __forceinline__ df64x2 cB2<df64x2>()
{
    return {make_float2(kB2h, kB2h), make_float2(kB2l, kB2l)};
}
template <> __device__ __forceinline__ pd cB1<pd>() { return {kB1, kB1}; }
template <> __device__ __forceinline__ pd cB2<pd>() { return {kB2, kB2}; }

// one node record of storage type S as compute type T
template <typename T>
__device__ __forceinline__ vec4<T> load_c(const vec4<typename StorageOf<T>::type> *p)
{
    const auto v = ld4(p);
    if constexpr (std::is_same<T, df64>::value)
        return {df_split<true>(v.x), df_split<true>(v.y), df_split<true>(v.z), df_split<true>(v.w)};
    else return {to_c<T>(v.x), to_c<T>(v.y), to_c<T>(v.z), to_c<T>(v.w)};
}

template <typename T> struct VG {
    T v, gx, gy, gz;
};

// Value and physical gradient at this lane's Gauss point of the Q1 field whose
// value at this lane's node is u.  sx = sigma_x/h_x with sigma = +1 when the
// lane's node sits at the upper side along x (and likewise sy, sz).
template <typename T> __device__ __forceinline__ VG<T> eval_vg_body(T u, T sx, T sy, T sz)
{
    const T b1 = cB1<T>(), b2 = cB2<T>();
    T uo = shx(u, 1);
    T tB = dot2_t(b1, u, b2, uo);
    T tD = u - uo;
    T tBo = shx(tB, 2), tDo = shx(tD, 2);
    T tBB = dot2_t(b1, tB, b2, tBo);
    T tBD = tB - tBo;
    T tDB = dot2_t(b1, tD, b2, tDo);
    T tBBo = shx(tBB, 4), tBDo = shx(tBD, 4), tDBo = shx(tDB, 4);
    VG<T> r;
    r.v = dot2_t(b1, tBB, b2, tBBo);
    r.gz = sz * (tBB - tBBo);
    r.gy = sy * dot2_t(b1, tBD, b2, tBDo);
    r.gx = sx * dot2_t(b1, tDB, b2, tDBo);
    return r;
}

// Native FP64 (one FP64 instruction per multiply, add or FMA alike): with
// b1 + b2 = 1, b1 u + b2 uo = uo + b1 (u - uo), so each value-type output of a
// butterfly stage is one FMA on the difference that the gradient-type output
// needs anyway: 15 FP64 instructions per field instead of 18.
template <> __device__ __forceinline__ VG<double> eval_vg_body<double>(double u, double sx,
                                                                       double sy, double sz)
{
    const double b1 = kB1;
    const double uo = shx(u, 1);
    const double tD = u - uo;
    const double tB = fma(b1, tD, uo);
    const double tBo = shx(tB, 2), tDo = shx(tD, 2);
    const double tBD = tB - tBo;
    const double tBB = fma(b1, tBD, tBo);
    const double tDB = fma(b1, tD - tDo, tDo);
    const double tBBo = shx(tBB, 4), tBDo = shx(tBD, 4), tDBo = shx(tDB, 4);
    const double dz = tBB - tBBo;
    VG<double> r;
    r.v = fma(b1, dz, tBBo);
    r.gz = sz * dz;
    r.gy = sy * fma(b1, tBD - tBDo, tBDo);
    r.gx = sx * fma(b1, tDB - tDBo, tDBo);
    return r;
}

template <typename T> __device__ __forceinline__ T eval_v_body(T u)
{
    const T b1 = cB1<T>(), b2 = cB2<T>();
    T t = dot2_t(b1, u, b2, shx(u, 1));
    t = dot2_t(b1, t, b2, shx(t, 2));
    return dot2_t(b1, t, b2, shx(t, 4));
}

// Evaluation and projection entry points.  With OUT set, double-float calls
// one out-of-line copy of each body instead of inlining it: inlined at all 8 +
// 4 + 4 call sites the double-float Jacobian body outgrows what the
// instruction cache holds for its 16 warps per SM (out of line: -6 % at 64^3,
// -12 % at 128^3); the shorter residual body is faster inlined (+3-5 %
// out of line; 6 % on mapped grids, whose geometry comes from a table).
// float and double always inline.
template <typename T> __device__ __noinline__ VG<T> eval_vg_ool(T u, T sx, T sy, T sz)
{
    return eval_vg_body(u, sx, sy, sz);
}
template <typename T> __device__ __noinline__ T eval_v_ool(T u) { return eval_v_body(u); }
// which compute types take the out-of-line copies when OUT is set
template <typename T>
constexpr bool kOutline = std::is_same<T, df64>::value || std::is_same<T, df64x2>::value;

template <bool OUT, typename T> __device__ __forceinline__ VG<T> eval_vg(T u, T sx, T sy, T sz)
{
    if constexpr (OUT && kOutline<T>)
        return eval_vg_ool(u, sx, sy, sz);
    else
        return eval_vg_body(u, sx, sy, sz);
}
template <bool OUT, typename T> __device__ __forceinline__ T eval_v(T u)
{
    if constexpr (OUT && kOutline<T>)
        return eval_v_ool(u);
    else
        return eval_v_body(u);
}
// Four fields of a node record evaluated as two pairs (x, y) and (z, w):
// float and double-float pairs run on the paired FP32 instructions (3-7 %
// faster VMS kernels); double has no paired form and evaluates field by field.
template <bool OUT, typename T>
__device__ __forceinline__ void eval_vg4(const vec4<T> &u, T sx, T sy, T sz, VG<T> &e0, VG<T> &e1,
                                         VG<T> &e2, VG<T> &e3)
{
    if constexpr (std::is_same<T, double>::value) {
        e0 = eval_vg<OUT>(u.x, sx, sy, sz);
        e1 = eval_vg<OUT>(u.y, sx, sy, sz);
        e2 = eval_vg<OUT>(u.z, sx, sy, sz);
        e3 = eval_vg<OUT>(u.w, sx, sy, sz);
        return;
    }
    using PO = PairOf<T>;
    const auto px = PO::pack(sx, sx), py = PO::pack(sy, sy), pz = PO::pack(sz, sz);
    const auto a = eval_vg<OUT>(PO::pack(u.x, u.y), px, py, pz);
    const auto b = eval_vg<OUT>(PO::pack(u.z, u.w), px, py, pz);
    e0 = {PO::first(a.v), PO::first(a.gx), PO::first(a.gy), PO::first(a.gz)};
    e1 = {PO::second(a.v), PO::second(a.gx), PO::second(a.gy), PO::second(a.gz)};
    e2 = {PO::first(b.v), PO::first(b.gx), PO::first(b.gy), PO::first(b.gz)};
    e3 = {PO::second(b.v), PO::second(b.gx), PO::second(b.gy), PO::second(b.gz)};
}

// values of two fields at the Gauss point
template <bool OUT, typename T> __device__ __forceinline__ void eval_v2(T u, T w, T &ru, T &rw)
{
    if constexpr (std::is_same<T, double>::value) {
        ru = eval_v<OUT>(u);
        rw = eval_v<OUT>(w);
        return;
    }
    using PO = PairOf<T>;
    const auto r = eval_v<OUT>(PO::pack(u, w));
    ru = PO::first(r);
    rw = PO::second(r);
}

template <typename T> __device__ __forceinline__ T inv_t(T v) { return T(1) / v; }
template <> __device__ __forceinline__ df64 inv_t<df64>(df64 v) { return df_rcp(v); }

template <typename T> __device__ __forceinline__ T rsqrt_t(T v);
template <> __device__ __forceinline__ float rsqrt_t(float v) { return 1.0f / sqrtf(v); }
// within 1 ulp (the CUDA math library's bound), far inside the operators' 1e-12
template <> __device__ __forceinline__ double rsqrt_t(double v) { return rsqrt(v); }
template <> __device__ __forceinline__ df64 rsqrt_t(df64 v) { return df_rsqrt(v); }

// Base state of the VMS form at one Gauss point.
// a[] holds the acceleration minus the body force (a - f): the two enter the
// residual only as that difference; cup = -tau_M / rho (u' = cup r_M)
template <typename T> struct GP {
    T v[3], gv[3][3], p, gp[3], a[3], f[3], s;
    T rM[3], rC, conv[3], tauM, tauC, up[3], pp, vGv, cup;
};

template <typename T>
__device__ __forceinline__ void base_state(const VmsArgs<T> &P, GP<T> &q)
{
    for (int i = 0; i < 3; ++i) {
        q.conv[i] = dot3_t(q.v[0], q.gv[i][0], q.v[1], q.gv[i][1], q.v[2], q.gv[i][2]);
        q.rM[i] = fma_t(P.rho, q.a[i] + q.conv[i], q.gp[i]);
    }
    q.rC = q.gv[0][0] + q.gv[1][1] + q.gv[2][2];
    q.vGv = dot3_t(P.G0 * q.v[0], q.v[0], P.G1 * q.v[1], q.v[1], P.G2 * q.v[2], q.v[2]);
    const T S = q.s * (P.q0 + q.vGv);
    q.tauM = rsqrt_t(S);
    // tau_C = 1/(tau_M tr G) and 1/tau_M = S tau_M
    q.tauC = S * q.tauM * P.inv_trG;
    q.cup = -q.tauM * P.inv_rho;
    for (int i = 0; i < 3; ++i) q.up[i] = q.cup * q.rM[i];
    q.pp = -P.rho * q.tauC * q.rC;
}

// Geometry of one Gauss point on a mapped grid: Ji = (dx/dxi)^{-1}, det,
// the metric G = Ji^T Ji of Sec. 2.1 (full), tr G and the bracket constant.
template <typename T> struct Geo {
    T Ji[3][3], det, G[3][3], inv_trG, q0;
};

// base state with a per-Gauss-point metric (mapped grids)
template <typename T>
__device__ __forceinline__ void base_state_g(const VmsArgs<T> &P, const Geo<T> &geo, GP<T> &q)
{
    for (int i = 0; i < 3; ++i) {
        q.conv[i] = dot3_t(q.v[0], q.gv[i][0], q.v[1], q.gv[i][1], q.v[2], q.gv[i][2]);
        q.rM[i] = fma_t(P.rho, q.a[i] + q.conv[i], q.gp[i]);
    }
    q.rC = q.gv[0][0] + q.gv[1][1] + q.gv[2][2];
    T vGv = T(0);
    for (int i = 0; i < 3; ++i)
        vGv += q.v[i] * (geo.G[i][0] * q.v[0] + geo.G[i][1] * q.v[1] + geo.G[i][2] * q.v[2]);
    q.vGv = vGv;
    const T S = q.s * (geo.q0 + q.vGv);
    q.tauM = rsqrt_t(S);
    q.tauC = S * q.tauM * geo.inv_trG;
    q.cup = -q.tauM * P.inv_rho;
    for (int i = 0; i < 3; ++i) q.up[i] = q.cup * q.rM[i];
    q.pp = -P.rho * q.tauC * q.rC;
}

// physical gradient from the reference one: g_j = sum_k gref_k Ji[k][j]
template <typename T>
__device__ __forceinline__ void to_phys(const Geo<T> &geo, VG<T> &e)
{
    const T a = e.gx, b = e.gy, c = e.gz;
    e.gx = a * geo.Ji[0][0] + b * geo.Ji[1][0] + c * geo.Ji[2][0];
    e.gy = a * geo.Ji[0][1] + b * geo.Ji[1][1] + c * geo.Ji[2][1];
    e.gz = a * geo.Ji[0][2] + b * geo.Ji[1][2] + c * geo.Ji[2][2];
}

// Geometry at this lane's Gauss point from the node coordinates xc of the
// element (lane = node on entry): J = dx/dxi by the butterfly (sx, sy, sz the
// reference gradient signs +-1/2), Ji by cofactors, G = Ji^T Ji, G:G, 1/tr G.
template <bool OUT, typename T>
__device__ __forceinline__ void mapped_geometry(const vec4<T> &xc, T sx, T sy, T sz,
                                                T (&out)[kMapGeo])
{
    VG<T> cx, cy, cz, cw;
    eval_vg4<OUT>(xc, sx, sy, sz, cx, cy, cz, cw);
    const T J[3][3] = {{cx.gx, cx.gy, cx.gz}, {cy.gx, cy.gy, cy.gz}, {cz.gx, cz.gy, cz.gz}};
    const T c00 = J[1][1] * J[2][2] - J[1][2] * J[2][1];
    const T c01 = J[1][2] * J[2][0] - J[1][0] * J[2][2];
    const T c02 = J[1][0] * J[2][1] - J[1][1] * J[2][0];
    const T det = J[0][0] * c00 + J[0][1] * c01 + J[0][2] * c02;
    const T id = inv_t(det);
    T Ji[3][3];
    Ji[0][0] = c00 * id;
    Ji[0][1] = (J[0][2] * J[2][1] - J[0][1] * J[2][2]) * id;
    Ji[0][2] = (J[0][1] * J[1][2] - J[0][2] * J[1][1]) * id;
    Ji[1][0] = c01 * id;
    Ji[1][1] = (J[0][0] * J[2][2] - J[0][2] * J[2][0]) * id;
    Ji[1][2] = (J[0][2] * J[1][0] - J[0][0] * J[1][2]) * id;
    Ji[2][0] = c02 * id;
    Ji[2][1] = (J[0][1] * J[2][0] - J[0][0] * J[2][1]) * id;
    Ji[2][2] = (J[0][0] * J[1][1] - J[0][1] * J[1][0]) * id;
    T G[3][3], GG = T(0);
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) {
            const T gij = Ji[0][i] * Ji[0][j] + Ji[1][i] * Ji[1][j] + Ji[2][i] * Ji[2][j];
            G[i][j] = gij;
            GG += gij * gij;
        }
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) out[3 * i + j] = Ji[i][j];
    out[9] = G[0][0];
    out[10] = G[0][1];
    out[11] = G[0][2];
    out[12] = G[1][1];
    out[13] = G[1][2];
    out[14] = G[2][2];
    out[15] = GG;
    out[16] = inv_t(G[0][0] + G[1][1] + G[2][2]);
    out[17] = det;
}

// Test-function coefficients of the residual at one quadrature point: X
// multiplies N_A, Y[c][j] multiplies dN_A/dx_j for residual component c.
template <typename T>
__device__ __forceinline__ void gp_residual_terms(const VmsArgs<T> &P, const GP<T> &q, T (&X)[4],
                                                  T (&Y)[4][3])
{
    // X_i = rho (a - f + v.grad v_i + u'.grad v_i), the sums in FMA order
    for (int i = 0; i < 3; ++i) {
        T t = q.a[i] + q.conv[i];
        t = fma_t(q.up[0], q.gv[i][0], t);
        t = fma_t(q.up[1], q.gv[i][1], t);
        t = fma_t(q.up[2], q.gv[i][2], t);
        X[i] = P.rho * t;
    }
    // Y_ij = mu (d_j v_i + d_i v_j) - rho (v_j + u'_j) u'_i: the symmetric
    // viscous part once per pair
    T mw[3];
    for (int j = 0; j < 3; ++j) mw[j] = -P.rho * (q.v[j] + q.up[j]);
    for (int i = 0; i < 3; ++i)
        for (int j = i; j < 3; ++j) {
            const T muS = P.mu * (q.gv[i][j] + q.gv[j][i]);
            Y[i][j] = fma_t(mw[j], q.up[i], muS);
            if (j != i) Y[j][i] = fma_t(mw[i], q.up[j], muS);
        }
    for (int i = 0; i < 3; ++i) Y[i][i] -= q.p + q.pp;
    X[3] = q.rC;
    for (int j = 0; j < 3; ++j) Y[3][j] = -q.up[j];
}

// v . G dv with the full metric of a Gauss point
template <typename T>
__device__ __forceinline__ T vGdv_full(const Geo<T> &geo, const GP<T> &q, const T (&dv)[3])
{
    T vGdv = T(0);
    for (int i = 0; i < 3; ++i)
        vGdv += q.v[i] * (geo.G[i][0] * dv[0] + geo.G[i][1] * dv[1] + geo.G[i][2] * dv[2]);
    return vGdv;
}

// The same coefficients of the Jacobian in the direction (dv, grad dv, da, dp,
// grad dp) (physical gradients, chain factors applied); vGdv = v . G dv and
// q0 = C_T/dt^2 + C_I nu^2 G:G at this point.
template <typename T>
__device__ __forceinline__ void gp_jacobian_terms(const VmsArgs<T> &P, const GP<T> &q,
                                                  const T (&dv)[3], const T (&dgv)[3][3],
                                                  const T (&da)[3], T dp, const T (&dgp)[3],
                                                  T vGdv, T q0, T (&X)[4], T (&Y)[4][3])
{
    T dconv[3], drM[3], dup[3], dadc[3];
    for (int i = 0; i < 3; ++i) {
        // dv.grad v_i + v.grad dv_i, one product and five FMAs
        T t = q.v[0] * dgv[i][0];
        t = fma_t(q.v[1], dgv[i][1], t);
        t = fma_t(q.v[2], dgv[i][2], t);
        t = fma_t(dv[0], q.gv[i][0], t);
        t = fma_t(dv[1], q.gv[i][1], t);
        dconv[i] = fma_t(dv[2], q.gv[i][2], t);
        dadc[i] = da[i] + dconv[i];
        drM[i] = fma_t(P.rho, dadc[i], dgp[i]);
    }
    const T drC = dgv[0][0] + dgv[1][1] + dgv[2][2];
    const T dtauM = -q.tauM * q.tauM * q.tauM * q.s * vGdv;
    // d tau_C = -tau_C d tau_M / tau_M, 1/tau_M = s (q0 + vGv) tau_M
    const T dtauC = -q.tauC * dtauM * (q.s * (q0 + q.vGv) * q.tauM);
    // du' = -(d tau_M r_M + tau_M d r_M) / rho
    const T ka = -dtauM * P.inv_rho;
    for (int i = 0; i < 3; ++i) dup[i] = fma_t(ka, q.rM[i], q.cup * drM[i]);
    const T dpp = -P.rho * dot2_t(dtauC, q.rC, q.tauC, drC);
    for (int i = 0; i < 3; ++i) {
        T t = dadc[i];
        t = fma_t(dup[0], q.gv[i][0], t);
        t = fma_t(dup[1], q.gv[i][1], t);
        t = fma_t(dup[2], q.gv[i][2], t);
        t = fma_t(q.up[0], dgv[i][0], t);
        t = fma_t(q.up[1], dgv[i][1], t);
        t = fma_t(q.up[2], dgv[i][2], t);
        X[i] = P.rho * t;
    }
    // Y_ij = mu (d_j dv_i + d_i dv_j) - rho [(dv_j + du'_j) u'_i + (v_j + u'_j) du'_i]
    T mw[3], md[3];
    for (int j = 0; j < 3; ++j) {
        mw[j] = -P.rho * (q.v[j] + q.up[j]);
        md[j] = -P.rho * (dv[j] + dup[j]);
    }
    for (int i = 0; i < 3; ++i)
        for (int j = i; j < 3; ++j) {
            const T muS = P.mu * (dgv[i][j] + dgv[j][i]);
            Y[i][j] = fma_t(md[j], q.up[i], fma_t(mw[j], dup[i], muS));
            if (j != i) Y[j][i] = fma_t(md[i], q.up[j], fma_t(mw[i], dup[j], muS));
        }
    for (int i = 0; i < 3; ++i) Y[i][i] -= dp + dpp;
    X[3] = drC;
    for (int j = 0; j < 3; ++j) Y[3][j] = -dup[j];
}

// ---------------------------------------------------------------- bricks
// A brick is bx x by columns of bz elements; four lanes own a column and march
// up its elements.  Lane (gx, gy) is first "node (gx, gy) of the plane" and
// then "the two Gauss points above that corner" (gz = 0, 1), so
//
//   evaluation  the x and y stages of the butterfly run once per node plane
//               (and serve the element below and the one above it), the z stage
//               combines the two planes of an element in the lane's own
//               registers, both Gauss points at once;
//   algebra     both Gauss points of a lane as one pair: float and double-float
//               on the paired FP32 instructions;
//   projection  the transposed z stage leaves a lower and an upper part, the
//               upper one is carried to the element above and added to its
//               lower part, and the transposed y and x stages run once per plane.
//
// Against eight lanes per element (one per node and Gauss point, three shuffle
// stages per field and element) this takes a quarter fewer floating-point
// operations per Gauss point, a third of the shuffles and half of the node
// loads.  Pressure and body force enter per unit of density (p/rho and a - f at
// the nodes), rho and det J once per plane at the end.
//
// Bound: FP64 by its pipe (86 % active), FP32 by issue (70 %, FMA pipe 63 %),
// double-float by the FP32 pipe and the latency of its dependent sequences.
// Against eight lanes per element (GB300, brick and gather kernels, default
// schedules): FP64 both operators at 64^3 2,073 -> 1,541 us; FP32 Jacobian apply
// at 128^3 370 -> 228 us, residual 283 -> 177 us; double-float residual at 128^3
// 1,524 -> 1,237 us, Jacobian apply 2,640 -> 2,230 us.  Tried and not kept: a
// barrier and the node sums after every plane (less shared memory, taller
// bricks) took the FP32 Jacobian apply from 296 to 376 us.

// storage cell of a compute type in shared memory (double-float: one 8-byte pair)
template <typename T> struct SmCell {
    using type = T;
};
template <> struct SmCell<df64> {
    using type = float2;
};
template <typename T> __device__ __forceinline__ T cell_ld(typename SmCell<T>::type v) { return v; }
template <> __device__ __forceinline__ df64 cell_ld<df64>(float2 v) { return df64(v.x, v.y); }
template <typename T> __device__ __forceinline__ typename SmCell<T>::type cell_st(T v) { return v; }
template <> __device__ __forceinline__ float2 cell_st<df64>(df64 v) { return make_float2(v.hi, v.lo); }

// Shared memory of a brick: rel[op][component][plane][corner][column], the
// columns padded so that a warp's 8 columns x 4 corners fall on different
// banks (4-byte cells: stride = 8 or 24 mod 32, 8-byte cells: 4 or 12 mod 16);
// then, for the types whose lower plane and carried parts do not fit the
// registers, lane[value][thread].
__host__ __device__ __forceinline__ int rel_stride(int ncol, int cell)
{
    if (cell == 4) {
        const int s = (ncol + 7) / 8 * 8;
        return s % 16 == 8 ? s : s + 8;
    }
    const int s = (ncol + 3) / 4 * 4;
    return s % 8 == 4 ? s : s + 4;
}
constexpr int kPlaneU = 16;  // plane values of U (4 x 3), A (3) and s
constexpr int kPlaneX = 12;  // plane values of x (4 x 3)
constexpr int kCarry = 12;   // carried values per operator (4 components x 3)
constexpr int kAsyncRecs = 4;  // node records of U, A, x and f
// 8-byte types: plane and carried values; float: two planes of node records
__host__ __device__ __forceinline__ int lane_values(int cell, bool jac, bool fused)
{
    return cell == 4 ? 2 * kAsyncRecs * 4 : kPlaneU + (jac ? kPlaneX : 0) + kCarry * (fused ? 2 : 1);
}
__host__ __device__ __forceinline__ size_t brick_smem(int bx, int by, int bz, int threads, int cell,
                                                      bool jac, bool fused)
{
    const size_t rel = (size_t)(fused ? 2 : 1) * 4 * (bz + 1) * 4 * rel_stride(bx * by, cell);
    return cell * (rel + (size_t)lane_values(cell, jac, fused) * threads);
}

// x and y stages at one node plane: value and in-plane gradient (scaled by sx,
// sy) above this lane's corner.  F: one field, or a pair of fields.
template <typename F> struct Face {
    F b, dx, dy;
};
template <typename F> __device__ __forceinline__ Face<F> face_body(F u, F sx, F sy)
{
    const F b1 = cB1<F>(), b2 = cB2<F>();
    const F uo = shx(u, 1);
    const F tB = dot2_t(b1, u, b2, uo), tD = u - uo;
    const F tBo = shx(tB, 2), tDo = shx(tD, 2);
    return {dot2_t(b1, tB, b2, tBo), sx * dot2_t(b1, tD, b2, tDo), sy * (tB - tBo)};
}
// native FP64 (one instruction per multiply, add or FMA alike): each
// value-type output is one FMA on the difference the gradient needs anyway
template <> __device__ __forceinline__ Face<double> face_body<double>(double u, double sx, double sy)
{
    const double b1 = kB1;
    const double uo = shx(u, 1);
    const double tD = u - uo, tB = fma(b1, tD, uo);
    const double tBo = shx(tB, 2), tDo = shx(tD, 2);
    const double d = tB - tBo;
    return {fma(b1, d, tBo), sx * fma(b1, tD - tDo, tDo), sy * d};
}
template <typename F> __device__ __forceinline__ F face_v_body(F u)
{
    const F b1 = cB1<F>(), b2 = cB2<F>();
    const F t = dot2_t(b1, u, b2, shx(u, 1));
    return dot2_t(b1, t, b2, shx(t, 2));
}
// transposed y and x stages: node contributions from the accumulated z parts
// (P1: value and z-gradient, P2 / P3: x- / y-gradient coefficients)
template <typename F>
__device__ __forceinline__ F face_project_body(F P1, F P2, F P3, F sx, F sy)
{
    const F b1 = cB1<F>(), b2 = cB2<F>();
    const F P1o = shx(P1, 2), P2o = shx(P2, 2), P3o = shx(P3, 2);
    const F Q1 = fma_t(sy, P3 + P3o, dot2_t(b1, P1, b2, P1o));
    const F Q2 = dot2_t(b1, P2, b2, P2o);
    const F Q1o = shx(Q1, 1), Q2o = shx(Q2, 1);
    return fma_t(sx, Q2 + Q2o, dot2_t(b1, Q1, b2, Q1o));
}
// one out-of-line copy of each for double-float pairs (instruction cache)
template <typename F> __device__ __noinline__ Face<F> face_ool(F u, F sx, F sy)
{
    return face_body(u, sx, sy);
}
template <typename F>
__device__ __noinline__ F face_project_ool(F P1, F P2, F P3, F sx, F sy)
{
    return face_project_body(P1, P2, P3, sx, sy);
}
template <typename F> __device__ __forceinline__ Face<F> face(F u, F sx, F sy)
{
    if constexpr (kOutline<F>)
        return face_ool(u, sx, sy);
    else
        return face_body(u, sx, sy);
}
template <typename F>
__device__ __forceinline__ F face_project(F P1, F P2, F P3, F sx, F sy)
{
    if constexpr (kOutline<F>)
        return face_project_ool(P1, P2, P3, sx, sy);
    else
        return face_project_body(P1, P2, P3, sx, sy);
}

// (a, b, c) times a 3 x 3 matrix m (row-major), or m times it (RIGHT), in the physical
// gradients and the projections of mapped grids: out of line for double-float pairs, as
// face_ool (128^3, both operators at once 5,835 -> 4,745 us; inline the eight uses
// outgrow the instruction cache)
template <typename F> struct Row3 {
    F x, y, z;
};
template <bool RIGHT, typename F>
__device__ __forceinline__ Row3<F> times3_body(F a, F b, F c, const F (&m)[9])
{
    if constexpr (RIGHT)
        return {dot3_t(m[0], a, m[1], b, m[2], c), dot3_t(m[3], a, m[4], b, m[5], c),
                dot3_t(m[6], a, m[7], b, m[8], c)};
    else
        return {dot3_t(a, m[0], b, m[3], c, m[6]), dot3_t(a, m[1], b, m[4], c, m[7]),
                dot3_t(a, m[2], b, m[5], c, m[8])};
}
template <bool RIGHT, typename F>
__device__ __noinline__ Row3<F> times3_ool(F a, F b, F c, F m0, F m1, F m2, F m3, F m4, F m5, F m6,
                                           F m7, F m8)
{
    const F m[9] = {m0, m1, m2, m3, m4, m5, m6, m7, m8};
    return times3_body<RIGHT>(a, b, c, m);
}
template <bool RIGHT, typename F>
__device__ __forceinline__ Row3<F> times3(F a, F b, F c, const F (&m)[9])
{
    if constexpr (kOutline<F>)
        return times3_ool<RIGHT>(a, b, c, m[0], m[1], m[2], m[3], m[4], m[5], m[6], m[7], m[8]);
    else
        return times3_body<RIGHT>(a, b, c, m);
}

// z stage: the two Gauss points between the plane values lo and hi
template <typename T> __device__ __forceinline__ typename PairOf<T>::type z_val(T lo, T hi)
{
    const T d = hi - lo;
    return PairOf<T>::pack(fma_t(cB2<T>(), d, lo), fma_t(cB1<T>(), d, lo));
}
template <> __device__ __forceinline__ df64x2 z_val<df64>(df64 lo, df64 hi)
{
    using PO = PairOf<df64>;
    return pair_dot2(PO::pack(cB1<df64>(), cB2<df64>()), PO::pack(lo, lo),
                     PO::pack(cB2<df64>(), cB1<df64>()), PO::pack(hi, hi));
}
// the same with the difference d = hi - lo at hand
template <typename T> __device__ __forceinline__ typename PairOf<T>::type z_val_d(T lo, T hi, T d)
{
    (void)hi;
    return PairOf<T>::pack(fma_t(cB2<T>(), d, lo), fma_t(cB1<T>(), d, lo));
}
template <> __device__ __forceinline__ df64x2 z_val_d<df64>(df64 lo, df64 hi, df64)
{
    return z_val(lo, hi);
}

// transposed z stage of one coefficient at the two Gauss points: tot = carry +
// b1 X0 + b2 X1 goes to the lower plane, up = b2 X0 + b1 X1 to the upper one
template <typename T>
__device__ __forceinline__ void z_part(typename PairOf<T>::type X, T carry, T &tot, T &up)
{
    const T X0 = PairOf<T>::first(X), X1 = PairOf<T>::second(X);
    const T d = X0 - X1;
    tot = fma_t(cB1<T>(), d, carry + X1);
    up = fma_t(-cB1<T>(), d, X0);
}
template <>
__device__ __forceinline__ void z_part<df64>(df64x2 X, df64 carry, df64 &tot, df64 &up)
{
    using PO = PairOf<df64>;
    const df64 X0 = PO::first(X), X1 = PO::second(X);
    const df64x2 r = pair_dot2(PO::pack(cB1<df64>(), cB2<df64>()), PO::pack(X0, X0),
                               PO::pack(cB2<df64>(), cB1<df64>()), PO::pack(X1, X1));
    tot = carry + PO::first(r);
    up = PO::second(r);
}

// 1/sqrt of both halves
template <> __device__ __forceinline__ f32x2 rsqrt_t(f32x2 v)
{
    // hardware estimate and one Newton step: within an ulp, in a fifth of the
    // instructions of an IEEE square root and division
    const f32x2 y = {make_float2(rsqrtf(v.v.x), rsqrtf(v.v.y))};
    const f32x2 one = {make_float2(1.0f, 1.0f)}, half = {make_float2(0.5f, 0.5f)};
    const f32x2 t = v * y;
    const f32x2 e = pair_fma({neg2(t.v)}, y, one);
    return pair_fma(half * y, e, y);
}
template <> __device__ __forceinline__ pd rsqrt_t(pd v) { return {rsqrt(v.a), rsqrt(v.b)}; }
template <> __device__ __forceinline__ df64x2 rsqrt_t(df64x2 x)
{
    // df_rsqrt on both halves
    const df64x2 r = {make_float2(rsqrtf(x.hi.x), rsqrtf(x.hi.y)), make_float2(0.0f, 0.0f)};
    const df64x2 one = {make_float2(1.0f, 1.0f), make_float2(0.0f, 0.0f)};
    const df64x2 half = {make_float2(0.5f, 0.5f), make_float2(0.0f, 0.0f)};
    const df64x2 corr = one - x * (r * r);
    return r + r * (corr * half);
}
__device__ __forceinline__ pd operator-(pd x) { return {-x.a, -x.b}; }
__device__ __forceinline__ f32x2 operator-(f32x2 x) { return {neg2(x.v)}; }

// 16 bytes to shared memory asynchronously (zeros when !ok)
__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool ok)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0)
                 : "memory");
}

// One brick: element contributions into rel (shared memory), then the node
// sums: nodes inside the brick straight into P.out, nodes shared with a
// neighbouring brick into the brick's node block in P.blocks (gather_node adds
// those up).  FUSED (with JAC): the residual at the same Gauss-point state goes
// to P.out2 / P.blocks2; the evaluation of U and A and the base state are
// shared by the two operators.
template <typename T, bool JAC, bool MAPPED = false, bool FUSED = false>
__device__ __forceinline__ void brick_body(const VmsArgs<T> &P, int brick, unsigned char *smem)
{
    static_assert(!FUSED || JAC, "the fused body computes the Jacobian apply too");
    using PO = PairOf<T>;
    using C = typename PO::type;
    using Cell = typename SmCell<T>::type;
    using S = typename StorageOf<T>::type;
    constexpr int kOps = FUSED ? 2 : 1;
    constexpr bool kLaneSm = sizeof(T) == 8;
    constexpr bool kAsync = sizeof(T) == 4;
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int bxi = brick % P.nbx, byi = (brick / P.nbx) % P.nby, bzi = brick / (P.nbx * P.nby);
    const int ex0 = bxi * P.bx, ey0 = byi * P.by, ez0 = bzi * P.bz;
    const int ncol = P.bx * P.by, stride = rel_stride(ncol, (int)sizeof(T));
    const int nl = min(P.bz, P.Nz - ez0);  // element layers of this brick
    const int plane_cells = 4 * stride, comp_cells = (P.bz + 1) * plane_cells;
    Cell *rel = reinterpret_cast<Cell *>(smem);
    Cell *lane = rel + kOps * 4 * comp_cells + tid;
    const int gx = tid & 1, gy = (tid >> 1) & 1;
    // gradient signs of the butterfly: physical (+-1/h) on the uniform grid,
    // reference (+-1/2 per unit of xi) on a mapped grid
    const T sx = MAPPED ? (gx ? T(0.5f) : T(-0.5f)) : (gx ? P.ih0 : -P.ih0);
    const T sy = MAPPED ? (gy ? T(0.5f) : T(-0.5f)) : (gy ? P.ih1 : -P.ih1);
    const T ihz = MAPPED ? T(0.5f) : P.ih2;
    const C sx2 = PO::pack(sx, sx), sy2 = PO::pack(sy, sy);
    const C nu = PO::pack(P.nu, P.nu), nu2 = PO::pack(P.nu2, P.nu2);
    const int NX1 = P.Nx + 1, NXY1 = (P.Nx + 1) * (P.Ny + 1);
    // rho det J and det J of the momentum and continuity rows (mapped grids:
    // det J per Gauss point)
    const T scale_m = MAPPED ? P.rho : P.rdetJ, scale_c = MAPPED ? T(1) : P.detJ;

    // plane values and carried parts: registers (float) or shared memory
    T Lr[kLaneSm ? 1 : kPlaneU + (JAC ? kPlaneX : 0)];
    T Cr[kLaneSm ? 1 : kCarry * kOps];
    auto getL = [&](int q) -> T {
        if constexpr (kLaneSm) return cell_ld<T>(lane[q * nthr]);
        else return Lr[q];
    };
    auto setL = [&](int q, T v) {
        if constexpr (kLaneSm) lane[q * nthr] = cell_st(v);
        else Lr[q] = v;
    };
    constexpr int kC0 = kPlaneU + (JAC ? kPlaneX : 0);
    auto getC = [&](int q) -> T {
        if constexpr (kLaneSm) return cell_ld<T>(lane[(kC0 + q) * nthr]);
        else return Cr[q];
    };
    auto setC = [&](int q, T v) {
        if constexpr (kLaneSm) lane[(kC0 + q) * nthr] = cell_st(v);
        else Cr[q] = v;
    };

    for (int base = 0; base < ncol; base += nthr >> 2) {
        const int col = base + (tid >> 2);
        const int lx = col % P.bx, ly = col / P.bx;
        const int ex = ex0 + lx, ey = ey0 + ly;
        const bool slot = col < ncol;
        const bool valid = slot && ex < P.Nx && ey < P.Ny;
        const int64_t node0 = valid ? (ex + gx) + (int64_t)NX1 * (ey + gy) + (int64_t)NXY1 * ez0 : 0;
        const vec4<T> zero = {T(0), T(0), T(0), T(0)};
        // in-plane stages of the four fields of a record, of three or four values
        auto faces4 = [&](const vec4<T> &u, Face<T> (&f)[4]) {
            if constexpr (std::is_same<T, double>::value) {
                f[0] = face(u.x, sx, sy);
                f[1] = face(u.y, sx, sy);
                f[2] = face(u.z, sx, sy);
                f[3] = face(u.w, sx, sy);
            } else {
                const Face<C> a = face(PO::pack(u.x, u.y), sx2, sy2);
                const Face<C> b = face(PO::pack(u.z, u.w), sx2, sy2);
                f[0] = {PO::first(a.b), PO::first(a.dx), PO::first(a.dy)};
                f[1] = {PO::second(a.b), PO::second(a.dx), PO::second(a.dy)};
                f[2] = {PO::first(b.b), PO::first(b.dx), PO::first(b.dy)};
                f[3] = {PO::second(b.b), PO::second(b.dx), PO::second(b.dy)};
            }
        };
        auto faces_v = [&](const vec4<T> &a, T (&v)[4]) {
            if constexpr (std::is_same<T, double>::value) {
                v[0] = face_v_body(a.x);
                v[1] = face_v_body(a.y);
                v[2] = face_v_body(a.z);
                v[3] = P.has_s ? face_v_body(a.w) : T(1);
            } else {
                const C p = face_v_body(PO::pack(a.x, a.y)), q = face_v_body(PO::pack(a.z, a.w));
                v[0] = PO::first(p);
                v[1] = PO::second(p);
                v[2] = PO::first(q);
                v[3] = PO::second(q);
            }
        };

        // float: the node records of the next plane are on their way to shared
        // memory (cp.async, each lane its own slots, no registers) while this
        // plane's element layer is computed; its layers are short against the
        // latency of the loads (Jacobian apply at 128^3: 290 us with plain loads,
        // 239 us so; prefetching into registers gained nothing).  Idle lanes get
        // zeros.
        float4 *slot4 = reinterpret_cast<float4 *>(rel + kOps * 4 * comp_cells) + tid;
        auto fetch = [&](int l) {
            if constexpr (kAsync) {
                if (l <= nl) {
                    const int64_t nd = node0 + (valid ? (int64_t)NXY1 * l : 0);
                    float4 *d = slot4 + (l & 1) * kAsyncRecs * nthr;
                    cp_async16(d, P.U + nd, valid);
                    cp_async16(d + nthr, P.A + nd, valid);
                    if constexpr (JAC) cp_async16(d + 2 * nthr, P.x + nd, valid);
                    if (P.f) cp_async16(d + 3 * nthr, P.f + nd, valid);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
        };
        auto fetched = [&](int l, int r) {
            const float4 v = slot4[((l & 1) * kAsyncRecs + r) * nthr];
            return vec4<T>{T(v.x), T(v.y), T(v.z), T(v.w)};
        };
        // records of plane l: scaled to per-unit-density pressure, chain factor
        auto load_u = [&](int l, int64_t nd) {
            vec4<T> u;
            if constexpr (kAsync) u = fetched(l, 0);
            else u = valid ? load_c<T>(P.U + nd) : zero;
            u.w = P.inv_rho * u.w;
            return u;
        };
        auto load_a = [&](int l, int64_t nd) {
            vec4<T> a, f;
            if constexpr (kAsync) a = fetched(l, 1);
            else a = valid ? load_c<T>(P.A + nd) : vec4<T>{T(0), T(0), T(0), T(1)};
            if (P.f) {
                if constexpr (kAsync) f = fetched(l, 3);
                else f = valid ? load_c<T>(P.f + nd) : zero;
                a.x = a.x - f.x;
                a.y = a.y - f.y;
                a.z = a.z - f.z;
            }
            return a;
        };
        auto load_x = [&](int l, int64_t nd) {
            vec4<T> x;
            if constexpr (kAsync) x = fetched(l, 2);
            else x = valid ? load_c<T>(P.x + nd) : zero;
            x.x = P.c_v * x.x;
            x.y = P.c_v * x.y;
            x.z = P.c_v * x.z;
            x.w = P.inv_rho * x.w;
            return x;
        };
        fetch(0);
        fetch(1);
        if constexpr (kAsync) asm volatile("cp.async.wait_group 1;" ::: "memory");

        // ---- the lowest plane
        {
            Face<T> f[4];
            T v[4];
            faces4(load_u(0, node0), f);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                setL(3 * c, f[c].b);
                setL(3 * c + 1, f[c].dx);
                setL(3 * c + 2, f[c].dy);
            }
            faces_v(load_a(0, node0), v);
#pragma unroll
            for (int c = 0; c < 4; ++c) setL(12 + c, v[c]);
            if constexpr (JAC) {
                faces4(load_x(0, node0), f);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    setL(kPlaneU + 3 * c, f[c].b);
                    setL(kPlaneU + 3 * c + 1, f[c].dx);
                    setL(kPlaneU + 3 * c + 2, f[c].dy);
                }
            }
#pragma unroll
            for (int q = 0; q < kCarry * kOps; ++q) setC(q, T(0));
        }

        // z parts of one component added to the carried ones; the totals of
        // the lower plane in t, the upper parts become the carried ones
        auto z_project = [&](int q0, const C &X, const C &Yx, const C &Yy, const C &Yz, T (&t)[3]) {
            T up;
            const T s = ihz * (PO::first(Yz) + PO::second(Yz));
            z_part<T>(X, getC(q0), t[0], up);
            t[0] = t[0] - s;
            setC(q0, up + s);
            z_part<T>(Yx, getC(q0 + 1), t[1], up);
            setC(q0 + 1, up);
            z_part<T>(Yy, getC(q0 + 2), t[2], up);
            setC(q0 + 2, up);
        };
        // transposed in-plane stages of components c and c + 1 (op o) of plane l
        auto put2 = [&](int o, int c, int l, const T (&t0)[3], const T (&t1)[3]) {
            T r0, r1;
            if constexpr (std::is_same<T, double>::value) {
                r0 = face_project(t0[0], t0[1], t0[2], sx, sy);
                r1 = face_project(t1[0], t1[1], t1[2], sx, sy);
            } else {
                const C r = face_project(PO::pack(t0[0], t1[0]), PO::pack(t0[1], t1[1]),
                                         PO::pack(t0[2], t1[2]), sx2, sy2);
                r0 = PO::first(r);
                r1 = PO::second(r);
            }
            r0 = scale_m * r0;
            r1 = (c == 2 ? scale_c : scale_m) * r1;
            if (slot) {
                Cell *d = rel + (4 * o + c) * comp_cells + l * plane_cells + (tid & 3) * stride + col;
                d[0] = cell_st(r0);
                d[comp_cells] = cell_st(r1);
            }
        };
        // projection of one operator's coefficients (continuity: X3, Y3) of layer l
        auto project_rows = [&](int o, int l, const C (&X)[4], const C (&Y)[4][3]) {
            T t0[3], t1[3];
#pragma unroll
            for (int c = 0; c < 4; c += 2) {
                z_project(kCarry * o + 3 * c, X[c], Y[c][0], Y[c][1], Y[c][2], t0);
                z_project(kCarry * o + 3 * c + 3, X[c + 1], Y[c + 1][0], Y[c + 1][1], Y[c + 1][2], t1);
                put2(o, c, l, t0, t1);
            }
        };

        // ---- the elements, bottom to top
        for (int l = 0; l < nl; ++l) {
            // the double-float body is long: a barrier per layer keeps the
            // CTA's warps on the same stretch of it (instruction cache)
            if constexpr (std::is_same<T, df64>::value) __syncthreads();
            const int64_t nd = node0 + (valid ? (int64_t)NXY1 * (l + 1) : 0);
            fetch(l + 2);
            if constexpr (kAsync) asm volatile("cp.async.wait_group 1;" ::: "memory");
            // geometry of the lane's two Gauss points (mapped grids); idle
            // lanes read element 0's
            const typename GeoStore<T>::type *gp = nullptr;
            if constexpr (MAPPED)
                gp = P.geo + (tid & 3) +
                     (valid ? (ex + (int64_t)P.Nx * (ey + (int64_t)P.Ny * (ez0 + l))) * (kMapGeo * 8)
                            : 0);
            auto geo = [&](int k) -> C {
                return PO::pack(geo_ld<T>(gp + 8 * k), geo_ld<T>(gp + 8 * k + 4));
            };
            // value and gradient at the two points of the field at plane slot q
            auto field = [&](int q, const Face<T> &h, C &v, C (&g)[3]) {
                const T lb = getL(q), d = h.b - lb, gz = ihz * d;
                v = z_val_d(lb, h.b, d);
                g[2] = PO::pack(gz, gz);
                g[0] = z_val(getL(q + 1), h.dx);
                g[1] = z_val(getL(q + 2), h.dy);
                setL(q, h.b);
                setL(q + 1, h.dx);
                setL(q + 2, h.dy);
            };
            auto to_physical = [&](C (&g)[3], const C (&Ji)[9]) {
                const Row3<C> t = times3<false>(g[0], g[1], g[2], Ji);
                g[0] = t.x;
                g[1] = t.y;
                g[2] = t.z;
            };
            C Ji[9];
            if constexpr (MAPPED)
#pragma unroll
                for (int k = 0; k < 9; ++k) Ji[k] = geo(k);

            // ---- base state: G[i][j] = d_j v_i, r = a + v.grad v + grad p / rho
            C v[3], G[3][3], pr, gpr[3], a[3], s;
            {
                Face<T> f[4];
                faces4(load_u(l + 1, nd), f);
#pragma unroll
                for (int i = 0; i < 3; ++i) field(3 * i, f[i], v[i], G[i]);
                field(9, f[3], pr, gpr);
                if constexpr (MAPPED) {
#pragma unroll
                    for (int i = 0; i < 3; ++i) to_physical(G[i], Ji);
                    to_physical(gpr, Ji);
                }
                T hv[4];
                faces_v(load_a(l + 1, nd), hv);
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    a[i] = z_val(getL(12 + i), hv[i]);
                    setL(12 + i, hv[i]);
                }
                if (P.has_s) {
                    s = z_val(getL(15), hv[3]);
                    setL(15, hv[3]);
                }
            }
            C rM[3], up[3], w[3], gv[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                C t = a[i] + gpr[i];
                t = fma_t(v[0], G[i][0], t);
                t = fma_t(v[1], G[i][1], t);
                rM[i] = fma_t(v[2], G[i][2], t);
            }
            const C rC = G[0][0] + G[1][1] + G[2][2];
            C q0, itrG;
            if constexpr (MAPPED) {
                const C g00 = geo(9), g01 = geo(10), g02 = geo(11), g11 = geo(12), g12 = geo(13),
                        g22 = geo(14);
                gv[0] = dot3_t(g00, v[0], g01, v[1], g02, v[2]);
                gv[1] = dot3_t(g01, v[0], g11, v[1], g12, v[2]);
                gv[2] = dot3_t(g02, v[0], g12, v[1], g22, v[2]);
                q0 = fma_t(PO::pack(P.CInu2, P.CInu2), geo(15), PO::pack(P.ct_dt2, P.ct_dt2));
                itrG = geo(16);
            } else {
                gv[0] = PO::pack(P.G0, P.G0) * v[0];
                gv[1] = PO::pack(P.G1, P.G1) * v[1];
                gv[2] = PO::pack(P.G2, P.G2) * v[2];
                q0 = PO::pack(P.q0, P.q0);
                itrG = PO::pack(P.inv_trG, P.inv_trG);
            }
            // S = s (q0 + v.G v), tau_M = S^-1/2, tau_C = S tau_M / tr G
            C Sq = q0 + dot3_t(gv[0], v[0], gv[1], v[1], gv[2], v[2]);
            if (P.has_s) Sq = s * Sq;
            const C tau = rsqrt_t(Sq);
            const C ntau = -tau;
            const C ntauC = Sq * ntau * itrG;
            // u' = -tau_M r, p'/rho = -tau_C r_C, w = v + u'
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                up[i] = ntau * rM[i];
                w[i] = v[i] + up[i];
            }
            const C pp = ntauC * rC;

            // Y[c] -> det (Ji Y[c]) and X[c] -> det X[c] on mapped grids
            auto to_reference = [&](C (&X)[4], C (&Y)[4][3]) {
                const C det = geo(17);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const Row3<C> t = times3<true>(Y[c][0], Y[c][1], Y[c][2], Ji);
                    Y[c][0] = det * t.x;
                    Y[c][1] = det * t.y;
                    Y[c][2] = det * t.z;
                    X[c] = det * X[c];
                }
            };
            // nu (g_ij + g_ji), both orders of the pair at once
            auto viscous = [&](const C (&g)[3][3], C (&Y)[4][3]) {
                Y[0][0] = nu2 * g[0][0];
                Y[1][1] = nu2 * g[1][1];
                Y[2][2] = nu2 * g[2][2];
                Y[0][1] = Y[1][0] = nu * (g[0][1] + g[1][0]);
                Y[0][2] = Y[2][0] = nu * (g[0][2] + g[2][0]);
                Y[1][2] = Y[2][1] = nu * (g[1][2] + g[2][1]);
            };
            if constexpr (!JAC || FUSED) {
                // residual: X_i = a_i + w.grad v_i,
                // Y_ij = nu (d_j v_i + d_i v_j) - w_j u'_i - (p + p') delta_ij
                C X[4], Y[4][3];
                viscous(G, Y);
                const C ptot = pr + pp;
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    C t = fma_t(w[0], G[i][0], a[i]);
                    t = fma_t(w[1], G[i][1], t);
                    X[i] = fma_t(w[2], G[i][2], t);
                    const C nup = -up[i];
#pragma unroll
                    for (int j = 0; j < 3; ++j) Y[i][j] = fma_t(w[j], nup, Y[i][j]);
                    Y[i][i] = Y[i][i] - ptot;
                    Y[3][i] = nup;
                }
                X[3] = rC;
                if constexpr (MAPPED) to_reference(X, Y);
                project_rows(FUSED ? 1 : 0, l, X, Y);
            }
            if constexpr (JAC) {
                C dv[3], dG[3][3], dp, dgp[3];
                {
                    Face<T> f[4];
                    faces4(load_x(l + 1, nd), f);
#pragma unroll
                    for (int i = 0; i < 3; ++i) field(kPlaneU + 3 * i, f[i], dv[i], dG[i]);
                    field(kPlaneU + 9, f[3], dp, dgp);
                    if constexpr (MAPPED) {
#pragma unroll
                        for (int i = 0; i < 3; ++i) to_physical(dG[i], Ji);
                        to_physical(dgp, Ji);
                    }
                }
                // d tau_M = -k tau_M and d tau_C = k tau_C with k = tau_M^2 s v.G dv
                const C vGdv = dot3_t(gv[0], dv[0], gv[1], dv[1], gv[2], dv[2]);
                C k = tau * tau * vGdv;
                if (P.has_s) k = s * k;
                const C drC = dG[0][0] + dG[1][1] + dG[2][2];
                const C cav = PO::pack(P.c_av, P.c_av);
                C da[3], dup[3], dw[3];
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    da[i] = cav * dv[i];
                    C t = da[i] + dgp[i];
                    t = fma_t(v[0], dG[i][0], t);
                    t = fma_t(v[1], dG[i][1], t);
                    t = fma_t(v[2], dG[i][2], t);
                    t = fma_t(dv[0], G[i][0], t);
                    t = fma_t(dv[1], G[i][1], t);
                    t = fma_t(dv[2], G[i][2], t);
                    // du' = -d tau_M r - tau_M dr = -k u' - tau_M dr
                    dup[i] = ntau * t - k * up[i];
                }
#pragma unroll
                for (int i = 0; i < 3; ++i) dw[i] = dv[i] + dup[i];
                // dp'/rho = -(d tau_C r_C + tau_C dr_C) = k p'/rho - tau_C dr_C
                const C dptot = dp + dot2_t(k, pp, ntauC, drC);
                C X[4], Y[4][3];
                viscous(dG, Y);
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    C t = da[i];
                    t = fma_t(dw[0], G[i][0], t);
                    t = fma_t(dw[1], G[i][1], t);
                    t = fma_t(dw[2], G[i][2], t);
                    t = fma_t(w[0], dG[i][0], t);
                    t = fma_t(w[1], dG[i][1], t);
                    X[i] = fma_t(w[2], dG[i][2], t);
                    const C nup = -up[i], ndup = -dup[i];
#pragma unroll
                    for (int j = 0; j < 3; ++j)
                        Y[i][j] = fma_t(dw[j], nup, fma_t(w[j], ndup, Y[i][j]));
                    Y[i][i] = Y[i][i] - dptot;
                    Y[3][i] = ndup;
                }
                X[3] = drC;
                if constexpr (MAPPED) to_reference(X, Y);
                project_rows(0, l, X, Y);
            }
        }
        // ---- the topmost plane: the carried parts alone
#pragma unroll
        for (int o = 0; o < kOps; ++o)
#pragma unroll
            for (int c = 0; c < 4; c += 2) {
                const int q = kCarry * o + 3 * c;
                const T t0[3] = {getC(q), getC(q + 1), getC(q + 2)};
                const T t1[3] = {getC(q + 3), getC(q + 4), getC(q + 5)};
                put2(o, c, nl, t0, t1);
            }
    }
    __syncthreads();

    // Node sums: each node of the brick's node block adds the contributions of
    // the (up to 4) columns around it in a fixed order.  A node that no other
    // brick holds is done; the others go to the node block.
    const int nx1 = P.bx + 1, ny1 = P.by + 1;
    const int nxv = min(P.bx, P.Nx - ex0), nyv = min(P.by, P.Ny - ey0);  // columns in the grid
    const int nin = (nxv + 1) * (nyv + 1) * (nl + 1);
    for (int q = tid; q < nin; q += nthr) {
        const int ix = q % (nxv + 1), iy = (q / (nxv + 1)) % (nyv + 1),
                  iz = q / ((nxv + 1) * (nyv + 1));
        const bool inner = (ix > 0 || ex0 == 0) && (ix < nxv || ex0 + nxv == P.Nx) &&
                           (iy > 0 || ey0 == 0) && (iy < nyv || ey0 + nyv == P.Ny) &&
                           (iz > 0 || ez0 == 0) && (iz < nl || ez0 + nl == P.Nz);
        const int64_t node = ex0 + ix + (int64_t)NX1 * (ey0 + iy) + (int64_t)NXY1 * (ez0 + iz);
        const size_t nb = (size_t)brick * (nx1 * ny1 * (P.bz + 1)) + ix + nx1 * (iy + ny1 * iz);
#pragma unroll
        for (int o = 0; o < kOps; ++o) {
            T acc[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int cx = ix - (c & 1), cy = iy - (c >> 1);
                if (cx < 0 || cy < 0 || cx >= nxv || cy >= nyv) continue;
                const Cell *r = rel + 4 * o * comp_cells + iz * plane_cells + c * stride + cy * P.bx + cx;
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[k] += cell_ld<T>(r[k * comp_cells]);
            }
            if (inner) {
                vec4<S> *out = FUSED && o ? P.out2 : P.out;
                out[node] = {to_s(acc[0]), to_s(acc[1]), to_s(acc[2]), to_s(acc[3])};
            } else {
                vec4<T> *blk = FUSED && o ? P.blocks2 : P.blocks;
                blk[nb] = {acc[0], acc[1], acc[2], acc[3]};
            }
        }
    }
}

// Candidate (brick, local index) pairs of node coordinate i along one axis,
// lower brick first.
static __device__ __forceinline__ int axis_candidates(int i, int b, int nb, int *cb, int *cl)
{
    int k = 0;
    const int q = i / b, r = i - q * b;
    if (r == 0 && q > 0) {
        cb[k] = q - 1;
        cl[k] = b;
        ++k;
    }
    if (q < nb) {
        cb[k] = q;
        cl[k] = r;
        ++k;
    }
    return k;
}

// Sum, for one node shared by several bricks, the (up to 8) brick node blocks
// that contain it, lower bricks first (FUSED: the residual's blocks into out2 as
// well): the node's candidate bricks along x and y, the plane k's along z.
struct AxisCandidates {
    int n, b[2] = {0, 0}, l[2] = {0, 0};  // count, bricks, local indices
    __device__ __forceinline__ AxisCandidates(int i, int size, int nb)
    {
        n = axis_candidates(i, size, nb, b, l);
    }
};
template <typename T, bool FUSED = false>
__device__ __forceinline__ void gather_node(const VmsArgs<T> &P, const AxisCandidates &cx,
                                            const AxisCandidates &cy, const AxisCandidates &cz,
                                            int64_t node)
{
    const int nx1 = P.bx + 1, ny1 = P.by + 1;
    const int nnodes = nx1 * ny1 * (P.bz + 1);
    constexpr int kOut = FUSED ? 2 : 1;
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
        const vec4<T> *blocks = o ? P.blocks2 : P.blocks;
        // all loads before the first sum: they are independent, and a branch
        // around each made the node wait for them one by one
        vec4<T> r[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int a = q & 1, b = (q >> 1) & 1, c = q >> 2;
            const bool in = a < cx.n && b < cy.n && c < cz.n;
            const int brick = in ? cx.b[a] + P.nbx * (cy.b[b] + P.nby * cz.b[c]) : 0;
            const int nl = in ? cx.l[a] + nx1 * (cy.l[b] + ny1 * cz.l[c]) : 0;
            r[q] = vec4<T>{T(0), T(0), T(0), T(0)};
            if (in) r[q] = ld4_blk(blocks + (int64_t)brick * nnodes + nl);
        }
        vec4<T> acc = r[0];  // the first candidate always exists
#pragma unroll
        for (int q = 1; q < 8; ++q) {
            // (an FP64 addition costs 16 cycles of an SM: none for a missing block)
            if (!((q & 1) < cx.n && ((q >> 1) & 1) < cy.n && (q >> 2) < cz.n)) continue;
            acc.x += r[q].x;
            acc.y += r[q].y;
            acc.z += r[q].z;
            acc.w += r[q].w;
        }
        (o ? P.out2 : P.out)[node] = {to_s(acc.x), to_s(acc.y), to_s(acc.z), to_s(acc.w)};
    }
}
// The nodes that several bricks share, numbered 0 .. shared_nodes() - 1 so that a
// thread per shared node does nothing else: (a) whole planes between bricks along
// z, (b) whole rows between bricks along y on the other planes, (c) the nodes
// between bricks along x in what is left.  (A thread per grid node spent 33 us at
// 129^3 finding out that its node was not shared; a warp per node row left too few
// loads in flight.)
template <typename T> __host__ __device__ __forceinline__ int64_t shared_nodes(const VmsArgs<T> &P)
{
    const int64_t nx = P.Nx + 1, ny = P.Ny + 1, nz = P.Nz + 1;
    const int sx = P.nbx - 1, sy = P.nby - 1, sz = P.nbz - 1;
    return sz * nx * ny + (nz - sz) * (sy * nx + (ny - sy) * sx);
}
// the r-th coordinate of an axis that no two of its bricks of b elements share
__device__ __forceinline__ int unshared_coord(int r, int b, int N)
{
    if (r == 0) return 0;
    const int g = b > 1 ? (r - 1) / (b - 1) : N;
    return min(g * b + r - g * (b - 1), N);
}
template <typename T, bool FUSED = false>
__device__ __forceinline__ void gather_shared(const VmsArgs<T> &P, int q)
{
    const int nx = P.Nx + 1, ny = P.Ny + 1;
    const int sx = P.nbx - 1, sy = P.nby - 1, sz = P.nbz - 1;
    int i, j, k;
    if (q < sz * nx * ny) {
        const int row = q / nx, pl = row / ny;
        i = q - row * nx;
        j = row - pl * ny;
        k = (pl + 1) * P.bz;
    } else {
        q -= sz * nx * ny;
        const int per = sy * nx + (ny - sy) * sx;  // of one plane
        const int pl = q / per;
        q -= pl * per;
        k = unshared_coord(pl, P.bz, P.Nz);
        if (q < sy * nx) {
            const int row = q / nx;
            i = q - row * nx;
            j = (row + 1) * P.by;
        } else {
            q -= sy * nx;
            const int row = q / sx;
            i = (q - row * sx + 1) * P.bx;
            j = unshared_coord(row, P.by, P.Ny);
        }
    }
    gather_node<T, FUSED>(P, AxisCandidates(i, P.bx, P.nbx), AxisCandidates(j, P.by, P.nby),
                          AxisCandidates(k, P.bz, P.nbz), i + (int64_t)nx * (j + (int64_t)ny * k));
}

// The schedule a kernel runs for a requested brick: the CTA no larger than the
// brick's lanes need, and the brick halved along its longest side until its
// shared memory fits.
constexpr int kBrickSmemMax = 200 * 1024;
constexpr int kBrickThreads = 128;  // CTA size limit of the brick kernels (their register caps)
inline Brick fit_brick(Brick b, int cell, bool jac, bool fused)
{
    for (;;) {
        const int lanes = (4 * b.bx * b.by + 31) / 32 * 32;
        if (b.threads > lanes) b.threads = lanes;
        if (b.threads > kBrickThreads) b.threads = kBrickThreads;
        if (brick_smem(b.bx, b.by, b.bz, b.threads, cell, jac, fused) <= kBrickSmemMax) return b;
        int &d = b.bz > 1 && b.bz >= b.bx && b.bz >= b.by ? b.bz : (b.bx >= b.by ? b.bx : b.by);
        if (d == 1) return b;  // a single element always fits
        d = (d + 1) / 2;
    }
}

template <typename T>
VmsArgs<T> make_args(const fsi_mesh *m, const Brick &b, const void *U, const void *A,
                     const void *f, const void *x, void *out)
{
    VmsArgs<T> P;
    P.Nx = m->grid.N[0];
    P.Ny = m->grid.N[1];
    P.Nz = m->grid.N[2];
    P.bx = b.bx;
    P.by = b.by;
    P.bz = b.bz;
    P.nbx = (P.Nx + b.bx - 1) / b.bx;
    P.nby = (P.Ny + b.by - 1) / b.by;
    P.nbz = (P.Nz + b.bz - 1) / b.bz;
    const double rho = m->phys.rho, mu = m->phys.mu, dt = m->phys.dt;
    const double *h = m->grid.h;
    double G[3], trG = 0.0, GG = 0.0;
    for (int k = 0; k < 3; ++k) {
        G[k] = 4.0 / (h[k] * h[k]);
        trG += G[k];
        GG += G[k] * G[k];
    }
    const double nu = mu / rho;
    P.rho = (T)rho;
    P.mu = (T)mu;
    P.inv_rho = (T)(1.0 / rho);
    P.nu = (T)nu;
    P.nu2 = (T)(2.0 * nu);
    P.G0 = (T)G[0];
    P.G1 = (T)G[1];
    P.G2 = (T)G[2];
    P.inv_trG = (T)(1.0 / trG);
    P.q0 = (T)(m->phys.C_T / (dt * dt) + m->phys.C_I * nu * nu * GG);
    P.ih0 = (T)(1.0 / h[0]);
    P.ih1 = (T)(1.0 / h[1]);
    P.ih2 = (T)(1.0 / h[2]);
    P.detJ = (T)(h[0] * h[1] * h[2] / 8.0);
    P.rdetJ = (T)(rho * (h[0] * h[1] * h[2] / 8.0));
    P.c_a = (T)m->alpha_m;
    P.c_v = (T)(m->alpha_f * m->gamma * dt);
    P.c_av = (T)(m->alpha_m / (m->alpha_f * m->gamma * dt));
    P.ct_dt2 = (T)(m->phys.C_T / (dt * dt));
    P.CInu2 = (T)(m->phys.C_I * nu * nu);
    P.has_s = m->phys.has_s != 0;
    using S = typename StorageOf<T>::type;
    P.Xc = (const vec4<S> *)(sizeof(S) == 8 ? m->coords64 : m->coords32);
    P.geo = nullptr;
    P.U = (const vec4<S> *)U;
    P.A = (const vec4<S> *)A;
    P.f = (const vec4<S> *)f;
    P.x = (const vec4<S> *)x;
    P.blocks = (vec4<T> *)m->vms_scratch;
    P.out = (vec4<S> *)out;
    P.blocks2 = nullptr;
    P.out2 = nullptr;
    return P;
}

}  // namespace vmsd
}  // namespace fsi
