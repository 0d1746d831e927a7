// tet.cu -- the hot path on unstructured meshes of linear tetrahedra (P1-P1,
// the element family of the paper's valve fluid mesh, Sec. 4): VMS residual
// and Jacobian apply (Sec. 2.1, 2.4), point location, interpolation and
// spreading (Sec. 2.3).
//
// VMS operators.  Four consecutive lanes own one tetrahedron: lane a first
// loads node a of the element (fields and coordinates) and then acts as
// quadrature point a of the symmetric 4-point rule (barycentric coordinates
// al at node a, be elsewhere).  The element geometry (J = [x1-x0, x2-x0,
// x3-x0], J^-1, the metric G = J^-T J^-1 of Sec. 2.1, G:G, 1/tr G, the weight)
// is a per-element table computed once per compute type (the mesh does not
// move; reading 72-144 B per element costs less than forming it in every
// lane of every apply); P1 gradients are constant per
// element, so a field's gradient is the group sum of u_a grad N_a and its
// value at point q is be * sum_a u_a + (al - be) u_q.  The Gauss-point
// algebra is the one the hexahedral kernels use (gp_residual_terms /
// gp_jacobian_terms with the full metric).  The projection onto test
// function a is w (be sum_q X_q + (al - be) X_a + grad N_a . sum_q Y_q) with
// w = |det J| / 24.  Each lane writes its node's contribution into a per-slot
// scratch [E][4]; a gather kernel sums, for every node, its slots in a fixed
// order (node -> slot lists built once at creation), so the result is
// deterministic and atomic-free.
//
// Location.  A uniform bucket grid over the mesh's bounding box lists, in
// increasing element order, the elements whose (padded) bounding box meets
// each bucket.  A point tests the candidates of its bucket in that order:
// an FP32 barycentric test discards elements it is clearly outside of (and
// stops the scan at one it is almost surely inside of), and the FP64
// barycentric coordinates, evaluated with round-to-nearest
// operations in the same order as the definition (no contraction), decide:
// the first element whose four coordinates are all >= -1e-12 holds the
// point.  That is the first element in element order, as a search over all
// elements would find.  The cell table (element -> points) is the stable
// counting sort of the grid path.
//
// Spreading.  Per element, four lanes sum the barycentric corner
// contributions w_B N_a(lam_B) lambda_B over the element's points (perm
// order, strided by lane), a fixed two-level transpose-reduce gives the 12
// corner sums; then every node sums the corner sums of its occupied elements
// in slot order.
#include <algorithm>
#include <cmath>
#include <new>
#include <type_traits>
#include <vector>

#include "fsi_internal.cuh"
#include "vms_device.cuh"

struct fsi_tetmesh {
    int device;
    cudaStream_t stream;
    int64_t n_nodes, n_elems;
    fsi_physics phys;
    double alpha_m, alpha_f, gamma;
    double4 *X64;
    float4 *X32;
    int4 *tets;
    int32_t *node_start, *node_slot;  // node -> slots e*4 + corner, increasing
    // location buckets
    int nb[3];
    double lo[3], inv_cell[3], box_lo[3], box_hi[3];
    int32_t *bucket_start, *bucket_tets;
    // scratch
    void *slot_scratch;    // [E][4] vec4 in the compute type (32 B per slot)
    void *corner_scratch;  // [E][4][3] spreading corner sums (8 B per value)
    int32_t *fill;         // [E+1]
    int32_t *scan_tmp;
    unsigned long long *nout;
    // distance-2 node colouring for probing the nodal diagonal blocks
    int32_t *colors;
    int n_colors;
    // per-element geometry (J^-1, G, G:G, 1/tr G, |det J|/24) in each compute
    // type [FSI_F64, FSI_F32, FSI_DF64], computed on first use
    void *geo[3];
};

namespace fsi {
namespace {

using namespace vmsd;

constexpr double kTetAl = 0.58541019662496845446;  // (5 + 3 sqrt 5) / 20
constexpr double kTetBe = 0.13819660112501051518;  // (5 - sqrt 5) / 20

template <typename T> __device__ __forceinline__ T tet_al();
template <typename T> __device__ __forceinline__ T tet_be();
template <> __device__ __forceinline__ double tet_al<double>() { return kTetAl; }
template <> __device__ __forceinline__ double tet_be<double>() { return kTetBe; }
template <> __device__ __forceinline__ float tet_al<float>() { return (float)kTetAl; }
template <> __device__ __forceinline__ float tet_be<float>() { return (float)kTetBe; }
constexpr float kTetAlH = static_cast<float>(kTetAl);
constexpr float kTetAlL = static_cast<float>(kTetAl - static_cast<double>(kTetAlH));
constexpr float kTetBeH = static_cast<float>(kTetBe);
constexpr float kTetBeL = static_cast<float>(kTetBe - static_cast<double>(kTetBeH));
template <> __device__ __forceinline__ df64 tet_al<df64>() { return df64(kTetAlH, kTetAlL); }
template <> __device__ __forceinline__ df64 tet_be<df64>() { return df64(kTetBeH, kTetBeL); }

// sum over the group of four lanes (butterfly; every lane gets the same value)
template <typename T> __device__ __forceinline__ T group_sum(T v)
{
    v = v + shx(v, 1);
    return v + shx(v, 2);
}

template <typename T> __device__ __forceinline__ T abs_t(T v) { return v < T(0) ? -v : v; }
template <> __device__ __forceinline__ df64 abs_t<df64>(df64 v) { return v.hi < 0.0f ? -v : v; }

// Element geometry from the four corner coordinates c[b][i]: J[i][k] =
// c[k+1][i] - c[0][i], J^-1 by cofactors, G = J^-T J^-1, G:G, 1/tr G and
// the quadrature weight |det J| / 24; it fills the per-element geometry table
// that the VMS kernels read.
constexpr int kTetGeo = 18;  // Ji[9], G00 G01 G02 G11 G12 G22, G:G, 1/trG, w

template <typename T> __device__ __forceinline__ void tet_geometry(const T (&c)[4][3], T (&out)[kTetGeo])
{
    T J[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) J[i][k] = c[k + 1][i] - c[0][i];
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
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            G[i][j] = dot3_t(Ji[0][i], Ji[0][j], Ji[1][i], Ji[1][j], Ji[2][i], Ji[2][j]);
            GG = fma_t(G[i][j], G[i][j], GG);
        }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) out[3 * i + k] = Ji[i][k];
    out[9] = G[0][0];
    out[10] = G[0][1];
    out[11] = G[0][2];
    out[12] = G[1][1];
    out[13] = G[1][2];
    out[14] = G[2][2];
    out[15] = GG;
    out[16] = inv_t(G[0][0] + G[1][1] + G[2][2]);
    out[17] = abs_t(det) * T(1.0 / 24.0);
}

template <typename T>
__global__ void tet_geo_kernel(int64_t E, const int4 *__restrict__ tets,
                               const vec4<typename StorageOf<T>::type> *__restrict__ X,
                               T *__restrict__ geo)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < E;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int4 t = tets[e];
        const int nd[4] = {t.x, t.y, t.z, t.w};
        T c[4][3];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const vec4<T> x = load_c<T>(X + nd[b]);
            c[b][0] = x.x;
            c[b][1] = x.y;
            c[b][2] = x.z;
        }
        T g[kTetGeo];
        tet_geometry(c, g);
#pragma unroll
        for (int k = 0; k < kTetGeo; ++k) geo[k * E + e] = g[k];
    }
}

template <typename T> struct TetArgs {
    using S = typename StorageOf<T>::type;
    VmsArgs<T> V;  // physics, chain factors and the field pointers U, A, f, x
    int64_t E;
    const vec4<S> *X;
    const int4 *tets;
    const T *geo;  // [kTetGeo][E]
    vec4<T> *slots;
};

// Four lanes per element (lane = node, then quadrature point): used on small
// meshes, where it spreads an element over four threads; every lane repeats the
// element's gradients (the rule: tet_by_element).
template <typename T, bool JAC> __global__ void __launch_bounds__(256) tet_vms_kernel(TetArgs<T> P)
{
    chain_trigger();
    using S = typename StorageOf<T>::type;
    const VmsArgs<T> &V = P.V;
    const int a = threadIdx.x & 3;
    const int lane = threadIdx.x & 31;
    // warp-uniform trip count: every lane of a warp shuffles in every pass
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t - lane < 4 * P.E;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = t >> 2;
        const bool valid = e < P.E;
        const vec4<T> zero = {T(0), T(0), T(0), T(0)};
        int node = 0;
        if (valid) {
            const int4 tt = P.tets[e];
            node = a == 0 ? tt.x : (a == 1 ? tt.y : (a == 2 ? tt.z : tt.w));
        }
        const vec4<T> u = valid ? load_c<T>(V.U + node) : zero;
        const vec4<T> ac = valid ? load_c<T>(V.A + node) : zero;
        const vec4<T> ff = (valid && V.f) ? load_c<T>(V.f + node) : zero;

        // element geometry from the table (idle lanes: the unit reference
        // tetrahedron, J = I)
        Geo<T> geo;
        T GG;
        if (valid) {
            auto g = [&](int k) { return P.geo[k * P.E + e]; };
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int k = 0; k < 3; ++k) geo.Ji[i][k] = g(3 * i + k);
            geo.G[0][0] = g(9);
            geo.G[0][1] = geo.G[1][0] = g(10);
            geo.G[0][2] = geo.G[2][0] = g(11);
            geo.G[1][1] = g(12);
            geo.G[1][2] = geo.G[2][1] = g(13);
            geo.G[2][2] = g(14);
            GG = g(15);
            geo.inv_trG = g(16);
            geo.det = g(17);  // holds the quadrature weight |det J| / 24
        } else {
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int k = 0; k < 3; ++k) geo.Ji[i][k] = geo.G[i][k] = T(i == k ? 1 : 0);
            GG = T(3);
            geo.inv_trG = inv_t(T(3));
            geo.det = T(1.0 / 24.0);
        }
        geo.q0 = fma_t(V.CInu2, GG, V.ct_dt2);
        // grad N of this lane's node
        T dN[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const T s3 = -(geo.Ji[0][j] + geo.Ji[1][j] + geo.Ji[2][j]);
            dN[j] = a == 0 ? s3 : (a == 1 ? geo.Ji[0][j] : (a == 2 ? geo.Ji[1][j] : geo.Ji[2][j]));
        }
        const T al = tet_al<T>(), be = tet_be<T>(), amb = al - be;
        // Values and gradients of two fields at a time: float and double-float
        // pairs run on the paired FP32 instructions (the double-float pair is
        // bit-identical to the scalar sequence); double pairs are two scalars.
        using PO = PairOf<T>;
        using PT = typename PO::type;
        const PT amb2 = PO::pack(amb, amb), be2 = PO::pack(be, be);
        PT dN2[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) dN2[j] = PO::pack(dN[j], dN[j]);
        auto value = [&](T w) { return fma_t(amb, w, be * group_sum(w)); };
        auto value2 = [&](T w1, T w2, T &r1, T &r2) {
            const PT w = PO::pack(w1, w2);
            const PT r = fma_t(amb2, w, be2 * group_sum(w));
            r1 = PO::first(r);
            r2 = PO::second(r);
        };
        auto grad2 = [&](T w1, T w2, T (&g1)[3], T (&g2)[3]) {
            const PT w = PO::pack(w1, w2);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const PT gs = group_sum(w * dN2[j]);
                g1[j] = PO::first(gs);
                g2[j] = PO::second(gs);
            }
        };

        GP<T> q;
        {
            value2(u.x, u.y, q.v[0], q.v[1]);
            value2(u.z, u.w, q.v[2], q.p);
            grad2(u.x, u.y, q.gv[0], q.gv[1]);
            grad2(u.z, u.w, q.gv[2], q.gp);
            T sv;
            value2(ac.x, ac.y, q.a[0], q.a[1]);
            value2(ac.z, ac.w, q.a[2], sv);
            q.s = V.has_s ? sv : T(1);
            if (V.f) {
                value2(ff.x, ff.y, q.f[0], q.f[1]);
                q.f[2] = value(ff.z);
                for (int i = 0; i < 3; ++i) q.a[i] = q.a[i] - q.f[i];
            } else {
                q.f[0] = q.f[1] = q.f[2] = T(0);
            }
            if (!valid) q.s = T(1);
        }
        base_state_g(V, geo, q);

        T X[4], Y[4][3];
        if (!JAC) {
            gp_residual_terms(V, q, X, Y);
        } else {
            const vec4<T> xx = valid ? load_c<T>(V.x + node) : zero;
            T val[3], dp, g[3][3], dgp[3];
            value2(xx.x, xx.y, val[0], val[1]);
            value2(xx.z, xx.w, val[2], dp);
            grad2(xx.x, xx.y, g[0], g[1]);
            grad2(xx.z, xx.w, g[2], dgp);
            T dv[3], da[3], dgv[3][3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                dv[i] = V.c_v * val[i];
                da[i] = V.c_a * val[i];
#pragma unroll
                for (int j = 0; j < 3; ++j) dgv[i][j] = V.c_v * g[i][j];
            }
            const T vGdv = vGdv_full(geo, q, dv);
            gp_jacobian_terms(V, q, dv, dgv, da, dp, dgp, vGdv, geo.q0, X, Y);
        }
        // projection onto this lane's test function, two components at a time
        const PT w2 = PO::pack(geo.det, geo.det);
        T r[4];
#pragma unroll
        for (int cc = 0; cc < 4; cc += 2) {
            const PT Xp = PO::pack(X[cc], X[cc + 1]);
            const PT gx = group_sum(PO::pack(Y[cc][0], Y[cc + 1][0]));
            const PT gy = group_sum(PO::pack(Y[cc][1], Y[cc + 1][1]));
            const PT gz = group_sum(PO::pack(Y[cc][2], Y[cc + 1][2]));
            const PT t0 = fma_t(amb2, Xp, be2 * group_sum(Xp));
            const PT rr = w2 * (t0 + dot3_t(dN2[0], gx, dN2[1], gy, dN2[2], gz));
            r[cc] = PO::first(rr);
            r[cc + 1] = PO::second(rr);
        }
        if (valid) P.slots[t] = vec4<T>{r[0], r[1], r[2], r[3]};
    }
}

// One thread per element.  On a linear tetrahedron the gradients, the divergence
// and the viscous stress are the same at all four quadrature points, so they are
// formed once: about 760 operations per Jacobian element against 1,400 of the
// four-lane kernel, and no shuffles.  float and double-float take their points two
// at a time on the paired FP32 instructions; float is fully unrolled, the 8-byte
// types run a rolled loop (their records come again from L1), which keeps the
// registers and the instruction footprint small.  Pressure enters per unit of
// density, rho at the end, as in the hexahedral kernels (vms_device.cuh, brick_body).
template <typename T> struct Points {  // quadrature points per pass
    static constexpr int n = 1;
    using C = T;
    static __device__ __forceinline__ C set(T a, T) { return a; }
    static __device__ __forceinline__ T first(C a) { return a; }
    static __device__ __forceinline__ T second(C) { return T(0); }
    static __device__ __forceinline__ T sum(C a) { return a; }
};
template <> struct Points<df64> {
    static constexpr int n = 2;
    using C = df64x2;
    static __device__ __forceinline__ C set(df64 a, df64 b) { return PairOf<df64>::pack(a, b); }
    static __device__ __forceinline__ df64 first(C a) { return PairOf<df64>::first(a); }
    static __device__ __forceinline__ df64 second(C a) { return PairOf<df64>::second(a); }
    static __device__ __forceinline__ df64 sum(C a) { return first(a) + second(a); }
};
template <> struct Points<float> {
    static constexpr int n = 2;
    using C = f32x2;
    static __device__ __forceinline__ C set(float a, float b) { return {make_float2(a, b)}; }
    static __device__ __forceinline__ float first(C a) { return a.v.x; }
    static __device__ __forceinline__ float second(C a) { return a.v.y; }
    static __device__ __forceinline__ float sum(C a) { return a.v.x + a.v.y; }
};

template <typename T, bool JAC>
__global__ void __launch_bounds__(128, sizeof(T) == 4 || (!JAC && std::is_same<T, df64>::value) ? 4 : 3)
    tet_vms_elem_kernel(TetArgs<T> P)
{
    chain_trigger();
    using S = typename StorageOf<T>::type;
    using PT = Points<T>;
    using C = typename PT::C;
    const VmsArgs<T> &V = P.V;
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= P.E) return;
    const int *nodes = reinterpret_cast<const int *>(P.tets + e);
    auto geo = [&](int k) -> T {
        return geo_ld<T>(reinterpret_cast<const typename GeoStore<T>::type *>(P.geo) + k * P.E + e);
    };
    auto load_u = [&](int n) {
        vec4<T> u = load_c<T>(V.U + n);
        u.w = V.inv_rho * u.w;
        return u;
    };
    auto load_a = [&](int n) {
        vec4<T> a = load_c<T>(V.A + n);
        if (V.f) {
            const vec4<T> f = load_c<T>(V.f + n);
            a.x = a.x - f.x;
            a.y = a.y - f.y;
            a.z = a.z - f.z;
        }
        return a;
    };
    auto load_x = [&](int n) {
        vec4<T> x = load_c<T>(V.x + n);
        x.x = V.c_v * x.x;
        x.y = V.c_v * x.y;
        x.z = V.c_v * x.z;
        x.w = V.inv_rho * x.w;
        return x;
    };
    // double-float: the records' values for the points' loop, converted once, in this
    // thread's column of shared memory (u, v, w, A and s, x)
    constexpr bool kKeep = std::is_same<T, df64>::value;
    constexpr int kVals = JAC ? 10 : 7;
    __shared__ float2 kept[kKeep ? 4 * kVals * 128 : 1];
    auto keep = [&](int node, int val, T t) {
        if constexpr (kKeep) kept[(node * kVals + val) * 128 + threadIdx.x] = make_float2(t.hi, t.lo);
    };
    auto keep3 = [&](int node, int val, const vec4<T> &t) {
        keep(node, val, t.x);
        keep(node, val + 1, t.y);
        keep(node, val + 2, t.z);
    };
    auto get3 = [&](int node, int val) {
        vec4<T> t;
        if constexpr (kKeep) {
            const float2 *q = kept + (node * kVals + val) * 128 + threadIdx.x;
            t = {T(q[0].x, q[0].y), T(q[128].x, q[128].y), T(q[256].x, q[256].y), T(0)};
        }
        return t;
    };
    auto get1 = [&](int node, int val) {
        T t;
        if constexpr (kKeep) {
            const float2 q = kept[(node * kVals + val) * 128 + threadIdx.x];
            t = T(q.x, q.y);
        }
        return t;
    };
    auto bc = [](T a) { return PT::set(a, a); };
    const T be = tet_be<T>(), amb = tet_al<T>() - be;
    T Ji[3][3];
#pragma unroll
    for (int k = 0; k < 9; ++k) Ji[k / 3][k % 3] = geo(k);

    // be x (sum over the nodes), and the gradients from the differences to
    // node 0: d_j w = sum_k Ji[k][j] (w_{k+1} - w_0)
    T su[4], sa[4], sx[4], G[4][3], dG[4][3];
    T Sp, Sdp;  // sums of the pressures over the points = over the nodes
    {
        const vec4<T> u0 = load_u(nodes[0]), a0 = load_a(nodes[0]);
        keep3(0, 0, u0);
        keep3(0, 3, a0);
        if (V.has_s) keep(0, 6, a0.w);
        const T w0[4] = {u0.x, u0.y, u0.z, u0.w};
        T x0[4] = {T(0), T(0), T(0), T(0)};
        if constexpr (JAC) {
            const vec4<T> v = load_x(nodes[0]);
            keep3(0, 7, v);
            x0[0] = v.x, x0[1] = v.y, x0[2] = v.z, x0[3] = v.w;
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) su[c] = w0[c], sx[c] = x0[c];
        sa[0] = a0.x, sa[1] = a0.y, sa[2] = a0.z, sa[3] = a0.w;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int n = nodes[k + 1];
            const vec4<T> uk = load_u(n), ak = load_a(n);
            keep3(k + 1, 0, uk);
            keep3(k + 1, 3, ak);
            if (V.has_s) keep(k + 1, 6, ak.w);
            const T w[4] = {uk.x, uk.y, uk.z, uk.w};
            sa[0] = sa[0] + ak.x;
            sa[1] = sa[1] + ak.y;
            sa[2] = sa[2] + ak.z;
            if (V.has_s) sa[3] = sa[3] + ak.w;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                su[c] = su[c] + w[c];
                const T d = w[c] - w0[c];
#pragma unroll
                for (int j = 0; j < 3; ++j) G[c][j] = k ? fma_t(Ji[k][j], d, G[c][j]) : Ji[k][j] * d;
            }
            if constexpr (JAC) {
                const vec4<T> xk = load_x(n);
                keep3(k + 1, 7, xk);
                const T y[4] = {xk.x, xk.y, xk.z, xk.w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    sx[c] = sx[c] + y[c];
                    const T d = y[c] - x0[c];
#pragma unroll
                    for (int j = 0; j < 3; ++j)
                        dG[c][j] = k ? fma_t(Ji[k][j], d, dG[c][j]) : Ji[k][j] * d;
                }
            }
        }
        Sp = su[3];
        Sdp = sx[3];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            su[c] = be * su[c];
            if (c < 3 || V.has_s) sa[c] = be * sa[c];
            if constexpr (JAC) sx[c] = be * sx[c];
        }
    }
    const T rC = G[0][0] + G[1][1] + G[2][2];
    const T drC = JAC ? dG[0][0] + dG[1][1] + dG[2][2] : T(0);
    const T q0 = fma_t(V.CInu2, geo(15), V.ct_dt2), itrG = geo(16);

    // sums over the points of the coefficients: Y without the viscous part and
    // with the pressures' sum apart; X at each point for the projection
    T SY[4][3], SX[3], Spp = T(0), Xp[4][3];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int j = 0; j < 3; ++j) SY[c][j] = T(0);
    SX[0] = SX[1] = SX[2] = T(0);
#pragma unroll(sizeof(T) == 4 ? 2 : 1)
    for (int g = 0; g < 4; g += PT::n) {
        [[maybe_unused]] const int n0 = nodes[g], n1 = nodes[g + PT::n - 1];
        auto at = [&](T s, T a, T b) { return fma_t(bc(amb), PT::set(a, b), bc(s)); };
        C v[3], r[3], a[3], s;
        {
            vec4<T> u0, a0, u1, a1;
            if constexpr (kKeep) {
                u0 = get3(g, 0), a0 = get3(g, 3), u1 = get3(g + 1, 0), a1 = get3(g + 1, 3);
                if (V.has_s) a0.w = get1(g, 6), a1.w = get1(g + 1, 6);
            } else {
                u0 = load_u(n0), a0 = load_a(n0);
                u1 = u0, a1 = a0;
                if constexpr (PT::n == 2) u1 = load_u(n1), a1 = load_a(n1);
            }
            v[0] = at(su[0], u0.x, u1.x);
            v[1] = at(su[1], u0.y, u1.y);
            v[2] = at(su[2], u0.z, u1.z);
            a[0] = at(sa[0], a0.x, a1.x);
            a[1] = at(sa[1], a0.y, a1.y);
            a[2] = at(sa[2], a0.z, a1.z);
            if (V.has_s) s = at(sa[3], a0.w, a1.w);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            C t = a[i] + bc(G[3][i]);
            t = fma_t(v[0], bc(G[i][0]), t);
            t = fma_t(v[1], bc(G[i][1]), t);
            r[i] = fma_t(v[2], bc(G[i][2]), t);
        }
        // S = s (q0 + v.G v), tau_M = S^-1/2, tau_C = S tau_M / tr G
        const C g01 = bc(geo(10)), g02 = bc(geo(11)), g12 = bc(geo(13));
        const C gv[3] = {dot3_t(bc(geo(9)), v[0], g01, v[1], g02, v[2]),
                         dot3_t(g01, v[0], bc(geo(12)), v[1], g12, v[2]),
                         dot3_t(g02, v[0], g12, v[1], bc(geo(14)), v[2])};
        C Sq = bc(q0) + dot3_t(gv[0], v[0], gv[1], v[1], gv[2], v[2]);
        if (V.has_s) Sq = s * Sq;
        const C tau = rsqrt_t(Sq), ntau = -tau, ntauC = Sq * ntau * bc(itrG);
        C up[3], w[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            up[i] = ntau * r[i];
            w[i] = v[i] + up[i];
        }
        const C pp = ntauC * bc(rC);
        C X[3];
        if constexpr (!JAC) {
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                C t = fma_t(w[0], bc(G[i][0]), a[i]);
                t = fma_t(w[1], bc(G[i][1]), t);
                X[i] = fma_t(w[2], bc(G[i][2]), t);
                const C nup = -up[i];
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    if constexpr (PT::n == 1) SY[i][j] = fma_t(w[j], nup, SY[i][j]);
                    else if constexpr (sizeof(T) == 8)
                        SY[i][j] = fma_t(PT::second(w[j]), PT::second(nup),
                                         fma_t(PT::first(w[j]), PT::first(nup), SY[i][j]));
                    else SY[i][j] = SY[i][j] + PT::sum(w[j] * nup);
                }
                SY[3][i] = SY[3][i] + PT::sum(nup);
            }
            Spp = Spp + PT::sum(pp);
        } else {
            C dv[3];
            {
                vec4<T> x0, x1;
                if constexpr (kKeep) {
                    x0 = get3(g, 7), x1 = get3(g + 1, 7);
                } else {
                    x0 = load_x(n0), x1 = x0;
                    if constexpr (PT::n == 2) x1 = load_x(n1);
                }
                dv[0] = at(sx[0], x0.x, x1.x);
                dv[1] = at(sx[1], x0.y, x1.y);
                dv[2] = at(sx[2], x0.z, x1.z);
            }
            const C vGdv = dot3_t(gv[0], dv[0], gv[1], dv[1], gv[2], dv[2]);
            C k = tau * tau * vGdv;
            if (V.has_s) k = s * k;
            C da[3], dup[3], dw[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                da[i] = bc(V.c_av) * dv[i];
                C t = da[i] + bc(dG[3][i]);
                t = fma_t(v[0], bc(dG[i][0]), t);
                t = fma_t(v[1], bc(dG[i][1]), t);
                t = fma_t(v[2], bc(dG[i][2]), t);
                t = fma_t(dv[0], bc(G[i][0]), t);
                t = fma_t(dv[1], bc(G[i][1]), t);
                t = fma_t(dv[2], bc(G[i][2]), t);
                dup[i] = ntau * t - k * up[i];
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) dw[i] = dv[i] + dup[i];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                C t = fma_t(dw[0], bc(G[i][0]), da[i]);
                t = fma_t(dw[1], bc(G[i][1]), t);
                t = fma_t(dw[2], bc(G[i][2]), t);
                t = fma_t(w[0], bc(dG[i][0]), t);
                t = fma_t(w[1], bc(dG[i][1]), t);
                X[i] = fma_t(w[2], bc(dG[i][2]), t);
                const C nup = -up[i], ndup = -dup[i];
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    if constexpr (PT::n == 1)
                        SY[i][j] = fma_t(dw[j], nup, fma_t(w[j], ndup, SY[i][j]));
                    else
                        SY[i][j] = SY[i][j] + PT::sum(fma_t(dw[j], nup, w[j] * ndup));
                }
                SY[3][i] = SY[3][i] + PT::sum(ndup);
            }
            Spp = Spp + PT::sum(dot2_t(k, pp, ntauC, bc(drC)));
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            SX[i] = SX[i] + PT::sum(X[i]);
            if constexpr (kKeep) {  // over u, which these points no longer need
                keep(g, i, PT::first(X[i]));
                keep(g + 1, i, PT::second(X[i]));
            } else {
                Xp[g][i] = PT::first(X[i]);
                if constexpr (PT::n == 2) Xp[g + 1][i] = PT::second(X[i]);
            }
        }
    }
    // the parts that are the same at every point: viscous stress, pressure sums
    {
        const T(&H)[4][3] = JAC ? dG : G;
        const T nu4 = V.nu2 + V.nu2, nu8 = nu4 + nu4;  // 4 nu, 8 nu
        const T p = JAC ? Sdp + Spp : Sp + Spp;
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = i; j < 3; ++j) {
                if (i == j) {
                    SY[i][i] = fma_t(nu8, H[i][i], SY[i][i]) - p;
                } else {
                    const T m = H[i][j] + H[j][i];
                    SY[i][j] = fma_t(nu4, m, SY[i][j]);
                    SY[j][i] = fma_t(nu4, m, SY[j][i]);
                }
            }
    }
    // projection: node a gets amb X(a) + be sum X + grad N_a . SY, the continuity
    // row div + grad N_a . SY_3; grad N_0 = -(sum of the others)
    // (double-float reads Ji again: its 18 registers are worth more in the loop)
    if constexpr (kKeep)
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            float2 t;
            asm volatile("ld.global.v2.f32 {%0, %1}, [%2];"
                         : "=f"(t.x), "=f"(t.y)
                         : "l"(reinterpret_cast<const float2 *>(P.geo) + k * P.E + e));
            Ji[k / 3][k % 3] = T(t.x, t.y);
        }
    const T wc = geo(17), wm = V.rho * wc;
    T q[4][4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
#pragma unroll
        for (int k = 0; k < 3; ++k)
            q[k + 1][c] = dot3_t(Ji[k][0], SY[c][0], Ji[k][1], SY[c][1], Ji[k][2], SY[c][2]);
        q[0][c] = -(q[1][c] + q[2][c] + q[3][c]);
    }
    const T div = JAC ? drC : rC;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        T o[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) o[i] = wm * (fma_t(amb, kKeep ? get1(a, i) : Xp[a][i], fma_t(be, SX[i], q[a][i])));
        P.slots[4 * e + a] = vec4<T>{o[0], o[1], o[2], wc * (div + q[a][3])};
    }
}

// Which of the two kernels.  A thread per element needs enough elements to fill the
// chip: in FP32 the two are level below 10,000 elements, in FP64 a mesh of 3,072 takes
// 37.2 us by elements against 35.2 us by lanes, and double-float, with its long
// dependent operations, is level at 24,576 (10,368: 20.8 against 16.8 us).  At 279,936
// elements, residual / Jacobian with their gathers, by lanes -> by elements: FP32
// 36.1/43.5 -> 27.0/32.8 us, FP64 508/787 -> 291/466 us, double-float 126/181 ->
// 93/145 us.
template <typename T> bool tet_by_element(int64_t E)
{
    return E >= (std::is_same<T, df64>::value ? 25000 : 10000);
}

// Sums over the four lanes of a node of four values each: lane q ends with value q.
template <typename T> __device__ __forceinline__ T quad_sum4(const T (&v)[4], int q)
{
    const bool b1 = q & 2, b0 = q & 1;
    T h[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const T send = b1 ? v[k] : v[2 + k], keep = b1 ? v[2 + k] : v[k];
        h[k] = keep + shfl_x(send, 2);
    }
    const T send = b0 ? h[0] : h[1], keep = b0 ? h[1] : h[0];
    return keep + shfl_x(send, 1);
}

// Element slots to nodes: a node's slots (24 on average) in four lanes, four
// slots a lane in flight.  Bound by the latency of two dependent reads: one
// thread per node, slot after slot, took 23 us at
// 279,936 elements, this 14 us.
template <typename T>
__global__ void __launch_bounds__(256)
    tet_gather_kernel(int64_t n, const int32_t *__restrict__ start, const int32_t *__restrict__ slot,
                      const vec4<T> *__restrict__ in, typename StorageOf<T>::type *__restrict__ out)
{
    chain_wait(start, slot, in, out);
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, i = t >> 2;
    const int q = (int)(t & 3);
    int k = 0, k1 = 0;
    if (i < n) {
        k = start[i] + q;
        k1 = start[i + 1];
    }
    T acc[4] = {T(0), T(0), T(0), T(0)};
    for (; k < k1; k += 16) {
        int sl[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) sl[u] = k + 4 * u < k1 ? slot[k + 4 * u] : -1;
        vec4<T> v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (sl[u] >= 0) v[u] = ld4_blk(in + sl[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (sl[u] >= 0) {
                acc[0] += v[u].x;
                acc[1] += v[u].y;
                acc[2] += v[u].z;
                acc[3] += v[u].w;
            }
    }
    const T sum = quad_sum4<T>(acc, q);
    if (i < n) out[t] = to_s(sum);
}

// ------------------------------------------------------------------ location
struct BucketArgs {
    int nb[3];
    double lo[3], inv_cell[3], box_lo[3], box_hi[3];
};

// barycentric coordinates, round-to-nearest operations in the order of the
// definition (e_k = x_k - x_0, d = P - x_0, D = e1.(e2 x e3), ...)
__device__ __forceinline__ void barycentric64(const double4 &x0, const double4 &x1,
                                              const double4 &x2, const double4 &x3,
                                              const double P[3], double lam[4])
{
    const double e1[3] = {__dsub_rn(x1.x, x0.x), __dsub_rn(x1.y, x0.y), __dsub_rn(x1.z, x0.z)};
    const double e2[3] = {__dsub_rn(x2.x, x0.x), __dsub_rn(x2.y, x0.y), __dsub_rn(x2.z, x0.z)};
    const double e3[3] = {__dsub_rn(x3.x, x0.x), __dsub_rn(x3.y, x0.y), __dsub_rn(x3.z, x0.z)};
    const double d[3] = {__dsub_rn(P[0], x0.x), __dsub_rn(P[1], x0.y), __dsub_rn(P[2], x0.z)};
    auto cross = [](const double *u, const double *v, double *w) {
        w[0] = __dsub_rn(__dmul_rn(u[1], v[2]), __dmul_rn(u[2], v[1]));
        w[1] = __dsub_rn(__dmul_rn(u[2], v[0]), __dmul_rn(u[0], v[2]));
        w[2] = __dsub_rn(__dmul_rn(u[0], v[1]), __dmul_rn(u[1], v[0]));
    };
    auto dot = [](const double *u, const double *v) {
        return __dadd_rn(__dadd_rn(__dmul_rn(u[0], v[0]), __dmul_rn(u[1], v[1])),
                         __dmul_rn(u[2], v[2]));
    };
    double c[3], a[3], b[3];
    cross(e2, e3, c);
    const double D = dot(e1, c);
    const double l1 = __ddiv_rn(dot(d, c), D);
    cross(d, e3, a);
    const double l2 = __ddiv_rn(dot(e1, a), D);
    cross(e2, d, b);
    const double l3 = __ddiv_rn(dot(e1, b), D);
    lam[1] = l1;
    lam[2] = l2;
    lam[3] = l3;
    lam[0] = __dsub_rn(__dsub_rn(__dsub_rn(1.0, l1), l2), l3);
}

// FP32 screen: 0 where the point is clearly outside (some barycentric
// coordinate below -1e-2), 2 where it is almost surely inside (all above
// -1e-5), 1 in between
__device__ __forceinline__ int screen32(const float4 &x0, const float4 &x1, const float4 &x2,
                                        const float4 &x3, const float P[3])
{
    const float e1[3] = {x1.x - x0.x, x1.y - x0.y, x1.z - x0.z};
    const float e2[3] = {x2.x - x0.x, x2.y - x0.y, x2.z - x0.z};
    const float e3[3] = {x3.x - x0.x, x3.y - x0.y, x3.z - x0.z};
    const float d[3] = {P[0] - x0.x, P[1] - x0.y, P[2] - x0.z};
    const float c0 = e2[1] * e3[2] - e2[2] * e3[1], c1 = e2[2] * e3[0] - e2[0] * e3[2],
                c2 = e2[0] * e3[1] - e2[1] * e3[0];
    const float D = e1[0] * c0 + e1[1] * c1 + e1[2] * c2;
    const float iD = 1.0f / D;
    const float l1 = (d[0] * c0 + d[1] * c1 + d[2] * c2) * iD;
    const float a0 = d[1] * e3[2] - d[2] * e3[1], a1 = d[2] * e3[0] - d[0] * e3[2],
                a2 = d[0] * e3[1] - d[1] * e3[0];
    const float l2 = (e1[0] * a0 + e1[1] * a1 + e1[2] * a2) * iD;
    const float b0 = e2[1] * d[2] - e2[2] * d[1], b1 = e2[2] * d[0] - e2[0] * d[2],
                b2 = e2[0] * d[1] - e2[1] * d[0];
    const float l3 = (e1[0] * b0 + e1[1] * b1 + e1[2] * b2) * iD;
    const float l0 = 1.0f - l1 - l2 - l3;
    const float lmin = fminf(fminf(l0, l1), fminf(l2, l3));
    if (lmin < -1e-2f) return 0;  // (a NaN falls through to the exact test)
    return lmin >= -1e-5f ? 2 : 1;
}

// A warp takes npw points (4, 8 or 16, few enough to fill the chip), each in a lane.
// Screening: eight lanes test eight
// elements of a point's list at a time in FP32, until every point has an element
// that holds it almost surely, four candidates, or no list left.  Then the exact FP64
// test runs over all (point, candidate) pairs of the warp, packed over the lanes, and
// a point takes its first candidate that passes, in list order.  Bound by the
// FP64 unit (about 120 operations a test, 16 cycles each) and by the latency of
// the screening's dependent reads; with a point's screening and tests in its own
// lane, lists of unequal length and candidate numbers left most lanes idle (50,000 points in
// 279,936 elements: 76 us, now 46 us).
constexpr int kLocThreads = 128, kLocCand = 4;
__global__ void __launch_bounds__(kLocThreads)
    tet_locate_kernel(int64_t m, BucketArgs B, const double4 *__restrict__ X64,
                      const float4 *__restrict__ X32, const int4 *__restrict__ tets,
                      const int32_t *__restrict__ bstart, const int32_t *__restrict__ btets,
                      const double *__restrict__ P, int npw, int32_t *__restrict__ elem,
                      double *__restrict__ lam_out, int32_t *__restrict__ count,
                      unsigned long long *n_out)
{
    chain_trigger();
    constexpr unsigned kAll = 0xffffffffu;
    __shared__ int cand_s[kLocThreads / 32][32 * kLocCand], pair_s[kLocThreads / 32][32 * kLocCand];
    __shared__ uint8_t owner_s[kLocThreads / 32][32 * kLocCand];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int *cand = cand_s[wid] + lane * kLocCand, *pairs = pair_s[wid];
    uint8_t *owners = owner_s[wid];
    const int64_t step = (int64_t)gridDim.x * (kLocThreads / 32) * npw;
    for (int64_t i0 = (blockIdx.x * (int64_t)(kLocThreads / 32) + wid) * npw; i0 < m; i0 += step) {
        const int64_t i = lane < npw ? i0 + lane : m;
        double p[3] = {0.0, 0.0, 0.0};
        int found = -1, c = 0, cend = 0;
        double l1 = 0.0, l2 = 0.0, l3 = 0.0;
        if (i < m) {
            bool inbox = true;
            for (int k = 0; k < 3; ++k) {
                p[k] = P[3 * i + k];
                inbox = inbox && p[k] >= B.box_lo[k] && p[k] <= B.box_hi[k];  // NaN: outside
            }
            if (inbox) {
                int bi[3];
                for (int k = 0; k < 3; ++k) {
                    int v = (int)floor((p[k] - B.lo[k]) * B.inv_cell[k]);
                    bi[k] = v < 0 ? 0 : (v >= B.nb[k] ? B.nb[k] - 1 : v);
                }
                const int64_t bk = bi[0] + (int64_t)B.nb[0] * (bi[1] + (int64_t)B.nb[1] * bi[2]);
                c = bstart[bk];
                cend = bstart[bk + 1];
            }
        }
        const float pf[3] = {(float)p[0], (float)p[1], (float)p[2]};
        while (__any_sync(kAll, found < 0 && c < cend)) {
            int nc = 0;
            bool more = found < 0 && c < cend;
            while (unsigned need = __ballot_sync(kAll, more)) {
#pragma unroll 2
                for (int g = 0; g < npw / 4; ++g) {
                    if (!((need >> (4 * g)) & 15u)) continue;  // none of these four points
                    const int src = 4 * g + (lane >> 3);
                    const int k = __shfl_sync(kAll, c, src) + (lane & 7);
                    const int ke = __shfl_sync(kAll, cend, src);
                    const float q[3] = {__shfl_sync(kAll, pf[0], src), __shfl_sync(kAll, pf[1], src),
                                        __shfl_sync(kAll, pf[2], src)};
                    int sc = 0;
                    if (((need >> src) & 1u) && k < ke) {
                        const int4 t = tets[btets[k]];
                        sc = screen32(X32[t.x], X32[t.y], X32[t.z], X32[t.w], q);
                    }
                    const unsigned some = __ballot_sync(kAll, sc > 0), sure = __ballot_sync(kAll, sc == 2);
                    if (more && (lane >> 2) == g) {
                        unsigned m1 = (some >> (8 * (lane & 3))) & 255u;
                        const unsigned m2 = (sure >> (8 * (lane & 3))) & 255u;
                        int next = c + 8;
                        if (m2) {
                            const int f = __ffs((int)m2);  // up to and with the first sure one
                            m1 &= (1u << f) - 1u;
                            next = c + f;
                            more = false;
                        }
                        while (m1) {
                            const int f = __ffs((int)m1);
                            m1 &= m1 - 1u;
                            cand[nc++] = c + f - 1;
                            if (nc == kLocCand) {
                                next = c + f;
                                more = false;
                                break;
                            }
                        }
                        c = next < cend ? next : cend;
                        more = more && c < cend;
                    }
                }
            }
            // the pairs of all points, point by point
            int first = nc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(kAll, first, o);
                if (lane >= o) first += v;
            }
            const int total = __shfl_sync(kAll, first, 31);
            first -= nc;
            for (int k = 0; k < nc; ++k) {
                pairs[first + k] = cand[k];
                owners[first + k] = (uint8_t)lane;
            }
            __syncwarp();
            for (int b = 0; b < total; b += 32) {
                const bool live = b + lane < total;
                const int own = live ? owners[b + lane] : lane, e = live ? btets[pairs[b + lane]] : 0;
                const double pp[3] = {__shfl_sync(kAll, p[0], own), __shfl_sync(kAll, p[1], own),
                                      __shfl_sync(kAll, p[2], own)};
                double lam[4] = {0.0, 0.0, 0.0, 0.0};
                bool ok = false;
                if (live) {
                    const int4 t = tets[e];
                    barycentric64(X64[t.x], X64[t.y], X64[t.z], X64[t.w], pp, lam);
                    ok = lam[0] >= -1e-12 && lam[1] >= -1e-12 && lam[2] >= -1e-12 && lam[3] >= -1e-12;
                }
                // this point's pairs among these 32
                const int lo = max(first - b, 0), hi = min(first + nc - b, 32);
                unsigned hit = __ballot_sync(kAll, ok);
                hit = lo < hi ? (hit >> lo) << lo & (kAll >> (32 - hi)) : 0u;
                const bool take = found < 0 && hit;
                const int src = take ? __ffs((int)hit) - 1 : lane;
                const int fe = __shfl_sync(kAll, e, src);
                const double f1 = __shfl_sync(kAll, lam[1], src), f2 = __shfl_sync(kAll, lam[2], src),
                             f3 = __shfl_sync(kAll, lam[3], src);
                if (take) {
                    found = fe;
                    l1 = f1;
                    l2 = f2;
                    l3 = f3;
                }
            }
            __syncwarp();
        }
        if (i >= m) continue;
        elem[i] = found;
        lam_out[3 * i] = l1;
        lam_out[3 * i + 1] = l2;
        lam_out[3 * i + 2] = l3;
        if (found < 0) atomicAdd(n_out, 1ull);
        else if (count) atomicAdd(count + found, 1);
    }
}

// ------------------------------------------------------------ interp / spread
template <typename T, typename S = typename StorageOf<T>::type>
__global__ void tet_interp_kernel(int64_t m, int64_t E, const int4 *__restrict__ tets,
                                  const int32_t *__restrict__ elem, const S *__restrict__ lam,
                                  const vec4<S> *__restrict__ U, S *__restrict__ u)
{
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < m;
         b += (int64_t)gridDim.x * blockDim.x) {
        const int e = elem[b];
        T ux = T(0), uy = T(0), uz = T(0);
        if (e >= 0 && e < E) {
            const int4 t = tets[e];
            const T l1 = to_c<T>(lam[3 * b]), l2 = to_c<T>(lam[3 * b + 1]),
                    l3 = to_c<T>(lam[3 * b + 2]);
            const T Nv[4] = {T(1) - l1 - l2 - l3, l1, l2, l3};
            const int nd[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const auto v = ld4(U + nd[a]);
                ux = madd(Nv[a], to_c<T>(v.x), ux);
                uy = madd(Nv[a], to_c<T>(v.y), uy);
                uz = madd(Nv[a], to_c<T>(v.z), uz);
            }
        }
        u[3 * b] = to_s(ux);
        u[3 * b + 1] = to_s(uy);
        u[3 * b + 2] = to_s(uz);
    }
}

// corner sums S[e][4][3] of the points of each element: a warp takes 8
// elements, four lanes per element; lane k sums the element's points k, k+4,
// ... in perm order, then a two-level transpose-reduce leaves corner 2 b1 + b0
// (3 values) in the lane with bits (b1, b0)
// (a point's inputs are loaded while the one before it is summed, and its index one
// earlier still, as in spread_run: elements of many points are bound by that latency and
// by the length of a double-float split, 300,000 points in 3,072 elements 767 -> 384 us;
// four CTAs an SM: at three, meshes with few points lose)
template <typename S> struct TetPoint {
    S l[3], f[3], w;
};
template <typename T, typename S = typename StorageOf<T>::type>
__global__ void __launch_bounds__(256, sizeof(S) == 8 ? 4 : 6) tet_spread_cells_kernel(int64_t E, const S *__restrict__ lam,
                                        const int32_t *__restrict__ start,
                                        const int32_t *__restrict__ perm,
                                        const S *__restrict__ lamv, const S *__restrict__ w,
                                        T *__restrict__ Ssum)
{
    chain_trigger();
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t e0 = warp * 8; e0 < E; e0 += nwarps * 8) {
        const int64_t e = e0 + (lane >> 2);
        int lo = 0, hi = 0;
        if (e < E) {
            lo = start[e];
            hi = start[e + 1];
        }
        if (__all_sync(0xffffffffu, hi == lo)) continue;
        T acc[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) acc[k] = T(0);
        auto load = [&](int b) {
            TetPoint<S> q;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                q.l[k] = lam[3 * b + k];
                q.f[k] = lamv[3 * b + k];
            }
            q.w = w ? w[b] : S(1);
            return q;
        };
        int p = lo + (lane & 3), b = 0;
        TetPoint<S> next;
        if (p < hi) {
            next = load(perm[p]);
            if (hi - p > 4) b = perm[p + 4];
        }
        for (; p < hi; p += 4) {
            const TetPoint<S> q = next;
            if (hi - p > 4) next = load(b);
            if (hi - p > 8) b = perm[p + 8];
            const T l1 = to_c<T>(q.l[0]), l2 = to_c<T>(q.l[1]), l3 = to_c<T>(q.l[2]);
            const T s = w ? to_c<T>(q.w) : T(1);
            const T Nv[4] = {(T(1) - l1 - l2 - l3) * s, l1 * s, l2 * s, l3 * s};
            const T f0 = to_c<T>(q.f[0]), f1 = to_c<T>(q.f[1]), f2 = to_c<T>(q.f[2]);
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                acc[3 * a] = madd(Nv[a], f0, acc[3 * a]);
                acc[3 * a + 1] = madd(Nv[a], f1, acc[3 * a + 1]);
                acc[3 * a + 2] = madd(Nv[a], f2, acc[3 * a + 2]);
            }
        }
        const bool b1 = lane & 2, b0 = lane & 1;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const T send = b1 ? acc[k] : acc[6 + k];
            const T keep = b1 ? acc[6 + k] : acc[k];
            acc[k] = keep + shfl_x(send, 2);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const T send = b0 ? acc[k] : acc[3 + k];
            const T keep = b0 ? acc[3 + k] : acc[k];
            acc[k] = keep + shfl_x(send, 1);
        }
        if (hi > lo) {
            T *dst = Ssum + e * 12 + (b1 ? 6 : 0) + (b0 ? 3 : 0);
            dst[0] = acc[0];
            dst[1] = acc[1];
            dst[2] = acc[2];
        }
    }
}

template <typename T, typename S = typename StorageOf<T>::type>
__global__ void __launch_bounds__(256)
    tet_spread_nodes_kernel(int64_t n, const int32_t *__restrict__ nstart,
                            const int32_t *__restrict__ nslot, const int32_t *__restrict__ start,
                            const T *__restrict__ Ssum, S *__restrict__ F, int accumulate)
{
    chain_wait(nstart, nslot, start, Ssum, F);
    // four lanes per node, four slots a lane in flight, as in tet_gather_kernel
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, i = t >> 2;
    const int q = (int)(t & 3);
    int k = 0, k1 = 0;
    if (i < n) {
        k = nstart[i] + q;
        k1 = nstart[i + 1];
    }
    T acc[4] = {T(0), T(0), T(0), T(0)};
    for (; k < k1; k += 16) {
        int sl[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) sl[u] = k + 4 * u < k1 ? nslot[k + 4 * u] : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = sl[u] >= 0 ? sl[u] >> 2 : 0;
            if (start[e + 1] == start[e]) sl[u] = -1;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (sl[u] >= 0) {
                const T *src = Ssum + 3 * (int64_t)sl[u];
                acc[0] += src[0];
                acc[1] += src[1];
                acc[2] += src[2];
            }
    }
    const T sum = quad_sum4<T>(acc, q);
    if (i < n && q < 3) F[t] = to_s(accumulate ? to_c<T>(F[t]) + sum : sum);
}

__global__ void pad_tet_coords_kernel(int64_t n, const double *X, double4 *X64, float4 *X32)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double x = X[3 * i], y = X[3 * i + 1], z = X[3 * i + 2];
        X64[i] = make_double4(x, y, z, 0.0);
        X32[i] = make_float4((float)x, (float)y, (float)z, 0.0f);
    }
}

int grid_for(int64_t n, int threads, int cap = sm_count() * 32)
{
    int64_t b = (n + threads - 1) / threads;
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

fsi_status validate_tetmesh(const fsi_tetmesh *m)
{
    if (!m) return set_error(FSI_ERR_ARG, "tet mesh is NULL");
    return FSI_OK;
}

template <typename T>
TetArgs<T> tet_args(fsi_tetmesh *m, const void *U, const void *A, const void *f, const void *x)
{
    using S = typename StorageOf<T>::type;
    TetArgs<T> P;
    memset((void *)&P.V, 0, sizeof P.V);
    const double rho = m->phys.rho, mu = m->phys.mu, dt = m->phys.dt, nu = mu / rho;
    P.V.rho = T(rho);
    P.V.mu = T(mu);
    P.V.inv_rho = T(1.0 / rho);
    P.V.c_a = T(m->alpha_m);
    P.V.c_v = T(m->alpha_f * m->gamma * dt);
    P.V.c_av = T(m->alpha_m / (m->alpha_f * m->gamma * dt));
    P.V.nu = T(nu);
    P.V.nu2 = T(2.0 * nu);
    P.V.ct_dt2 = T(m->phys.C_T / (dt * dt));
    P.V.CInu2 = T(m->phys.C_I * nu * nu);
    P.V.has_s = m->phys.has_s != 0;
    P.V.U = (const vec4<S> *)U;
    P.V.A = (const vec4<S> *)A;
    P.V.f = (const vec4<S> *)f;
    P.V.x = (const vec4<S> *)x;
    P.E = m->n_elems;
    P.X = (const vec4<S> *)(sizeof(S) == 8 ? (const void *)m->X64 : (const void *)m->X32);
    P.tets = m->tets;
    P.slots = (vec4<T> *)m->slot_scratch;
    return P;
}

template <typename T> constexpr int geo_slot()
{
    return std::is_same<T, double>::value ? 0 : (std::is_same<T, float>::value ? 1 : 2);
}

// the per-element geometry table of compute type T, built on first use
template <typename T> fsi_status ensure_geo(fsi_tetmesh *m)
{
    using S = typename StorageOf<T>::type;
    void *&g = m->geo[geo_slot<T>()];
    if (g) return FSI_OK;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    FSI_CUDA(cudaStreamIsCapturing(m->stream, &cap), "cudaStreamIsCapturing");
    if (cap != cudaStreamCaptureStatusNone)
        return set_error(FSI_ERR_ARG, "tetrahedral geometry table: first apply of this compute "
                                      "type inside a stream capture");
    if (cudaMalloc(&g, (size_t)m->n_elems * kTetGeo * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        g = nullptr;
        return set_error(FSI_ERR_OOM, "tetrahedral geometry table: cudaMalloc failed");
    }
    const vec4<S> *X = (const vec4<S> *)(sizeof(S) == 8 ? (const void *)m->X64
                                                         : (const void *)m->X32);
    tet_geo_kernel<T><<<grid_for(m->n_elems, 256), 256, 0, m->stream>>>(m->n_elems, m->tets, X,
                                                                        (T *)g);
    return check_launch("tet geometry kernel");
}

template <typename T, bool JAC>
fsi_status tet_vms(fsi_tetmesh *m, const void *U, const void *A, const void *f, const void *x,
                   void *out)
{
    using S = typename StorageOf<T>::type;
    FSI_TRY(ensure_geo<T>(m));
    TetArgs<T> P = tet_args<T>(m, U, A, f, x);
    P.geo = (const T *)m->geo[geo_slot<T>()];
    if (tet_by_element<T>(m->n_elems)) {
        tet_vms_elem_kernel<T, JAC><<<(int)((m->n_elems + 127) / 128), 128, 0, m->stream>>>(P);
    } else {
        const int64_t threads = 4 * m->n_elems;
        tet_vms_kernel<T, JAC><<<grid_for(threads, 256, sm_count() * 64), 256, 0, m->stream>>>(P);
    }
    FSI_TRY(check_launch("tet vms kernel"));
    launch_chain(tet_gather_kernel<T>, (int)((4 * m->n_nodes + 255) / 256), 256, 0, m->stream,
        m->n_nodes, m->node_start, m->node_slot, P.slots, (S *)out);
    return check_launch("tet gather kernel");
}

}  // namespace

void tet_set_stream(fsi_tetmesh *t, cudaStream_t s) { t->stream = s; }

void tet_set_physics(fsi_tetmesh *t, const fsi_physics *p)
{
    t->phys = *p;
    const double r = p->rho_inf;
    t->alpha_m = 0.5 * (3.0 - r) / (1.0 + r);
    t->alpha_f = 1.0 / (1.0 + r);
    t->gamma = 0.5 + t->alpha_m - t->alpha_f;
}

const int32_t *tet_colors(const fsi_tetmesh *t, int *n_colors)
{
    *n_colors = t->n_colors;
    return t->colors;
}

fsi_status tet_download(fsi_tetmesh *t, std::vector<double> &X, std::vector<int32_t> &tets,
                        double box_lo[3], double box_hi[3])
{
    std::vector<double4> x4((size_t)t->n_nodes);
    tets.resize((size_t)t->n_elems * 4);
    FSI_CUDA(cudaMemcpyAsync(x4.data(), t->X64, x4.size() * sizeof(double4), cudaMemcpyDeviceToHost,
                             t->stream),
             "memcpy");
    FSI_CUDA(cudaMemcpyAsync(tets.data(), t->tets, tets.size() * sizeof(int32_t),
                             cudaMemcpyDeviceToHost, t->stream),
             "memcpy");
    FSI_CUDA(cudaStreamSynchronize(t->stream), "sync");
    X.resize((size_t)t->n_nodes * 3);
    for (int k = 0; k < 3; ++k) {
        box_lo[k] = INFINITY;
        box_hi[k] = -INFINITY;
    }
    for (int64_t i = 0; i < t->n_nodes; ++i) {
        const double v[3] = {x4[i].x, x4[i].y, x4[i].z};
        for (int k = 0; k < 3; ++k) {
            X[3 * i + k] = v[k];
            box_lo[k] = std::min(box_lo[k], v[k]);
            box_hi[k] = std::max(box_hi[k], v[k]);
        }
    }
    return FSI_OK;
}

}  // namespace fsi

using namespace fsi;

extern "C" {

fsi_status fsi_mesh_create_tet(int64_t n_nodes, const double *X, int64_t n_tets,
                               const int32_t *tets, const fsi_physics *phys, int device,
                               void *cuda_stream, fsi_mesh **out)
{
    if (!out) return set_error(FSI_ERR_ARG, "out is NULL");
    *out = nullptr;
    fsi_tetmesh *t = nullptr;
    FSI_TRY(fsi_tetmesh_create(n_nodes, X, n_tets, tets, phys, device, cuda_stream, &t));
    fsi_mesh *m = new (std::nothrow) fsi_mesh();
    if (!m) {
        fsi_tetmesh_destroy(t);
        return set_error(FSI_ERR_OOM, "host allocation of the mesh handle failed");
    }
    m->phys = *phys;
    m->device = device;
    m->stream = (cudaStream_t)cuda_stream;
    m->n_nodes = n_nodes;
    m->n_elems = n_tets;
    m->alpha_m = t->alpha_m;
    m->alpha_f = t->alpha_f;
    m->gamma = t->gamma;
    m->tet = t;
    if (cudaMalloc(&m->dev_counters, 8 * sizeof(int64_t)) != cudaSuccess) {
        cudaGetLastError();
        fsi_mesh_destroy(m);
        return set_error(FSI_ERR_OOM, "fsi_mesh_create_tet: cudaMalloc failed");
    }
    *out = m;
    return FSI_OK;
}


fsi_status fsi_tetmesh_create(int64_t n_nodes, const double *X, int64_t n_tets,
                              const int32_t *tets, const fsi_physics *phys, int device,
                              void *cuda_stream, fsi_tetmesh **out)
{
    if (!out) return set_error(FSI_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (n_nodes < 4 || n_nodes >= INT32_MAX || n_tets < 1 || n_tets >= INT32_MAX / 4)
        return set_error(FSI_ERR_ARG, "fsi_tetmesh_create: bad sizes");
    if (!X || !tets || !phys) return set_error(FSI_ERR_ARG, "fsi_tetmesh_create: NULL argument");
    if (!(phys->rho > 0.0) || !(phys->mu >= 0.0) || !(phys->dt > 0.0) || !(phys->C_I >= 0.0) ||
        !(phys->C_T >= 0.0) || !(phys->rho_inf >= 0.0 && phys->rho_inf <= 1.0))
        return set_error(FSI_ERR_ARG, "invalid physics");
    FSI_DEVICE(device);
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // host copies for the set-up structures
    std::vector<int32_t> ht((size_t)n_tets * 4);
    std::vector<double> hx((size_t)n_nodes * 3);
    FSI_CUDA(cudaMemcpyAsync(ht.data(), tets, ht.size() * sizeof(int32_t), cudaMemcpyDeviceToHost,
                             s), "copy tets");
    FSI_CUDA(cudaMemcpyAsync(hx.data(), X, hx.size() * sizeof(double), cudaMemcpyDeviceToHost, s),
             "copy coordinates");
    FSI_CUDA(cudaStreamSynchronize(s), "sync");
    for (int32_t v : ht)
        if (v < 0 || v >= n_nodes) return set_error(FSI_ERR_ARG, "tet node index out of range");
    // node -> slots, increasing slot order
    std::vector<int32_t> nstart((size_t)n_nodes + 1, 0), nslot(ht.size());
    for (int32_t v : ht) nstart[(size_t)v + 1] += 1;
    for (int64_t i = 0; i < n_nodes; ++i) nstart[i + 1] += nstart[i];
    {
        std::vector<int32_t> cur(nstart.begin(), nstart.end() - 1);
        for (size_t sl = 0; sl < ht.size(); ++sl) nslot[cur[ht[sl]]++] = (int32_t)sl;
    }
    // greedy distance-2 colouring in node order: a node takes the smallest
    // colour no node of its elements holds yet
    std::vector<int32_t> hcol((size_t)n_nodes, -1);
    int ncol = 0;
    {
        std::vector<int64_t> seen;  // per colour: last node that saw it
        for (int64_t v = 0; v < n_nodes; ++v) {
            for (int k = nstart[v]; k < nstart[v + 1]; ++k) {
                const int64_t e = nslot[k] >> 2;
                for (int a = 0; a < 4; ++a) {
                    const int c = hcol[ht[4 * e + a]];
                    if (c >= 0) {
                        if ((size_t)c >= seen.size()) seen.resize(c + 1, -1);
                        seen[c] = v;
                    }
                }
            }
            int c = 0;
            while ((size_t)c < seen.size() && seen[c] == v) ++c;
            hcol[v] = c;
            ncol = std::max(ncol, c + 1);
        }
    }
    // bucket grid: about two elements per bucket, cells as cubic as the box allows
    double lo[3], hi[3];
    for (int k = 0; k < 3; ++k) {
        lo[k] = INFINITY;
        hi[k] = -INFINITY;
    }
    for (int64_t i = 0; i < n_nodes; ++i)
        for (int k = 0; k < 3; ++k) {
            const double v = hx[3 * i + k];
            if (!std::isfinite(v)) return set_error(FSI_ERR_ARG, "non-finite node coordinate");
            lo[k] = std::min(lo[k], v);
            hi[k] = std::max(hi[k], v);
        }
    double ext[3], vol = 1.0;
    for (int k = 0; k < 3; ++k) {
        ext[k] = std::max(hi[k] - lo[k], 1e-300);
        vol *= ext[k];
    }
    const double cell = std::cbrt(vol / std::max(1.0, n_tets / 2.0));
    int nb[3];
    for (int k = 0; k < 3; ++k)
        nb[k] = (int)std::min<double>(1024.0, std::max(1.0, std::ceil(ext[k] / cell)));
    double inv_cell[3];
    for (int k = 0; k < 3; ++k) inv_cell[k] = nb[k] / ext[k];
    const int64_t nbk = (int64_t)nb[0] * nb[1] * nb[2];
    std::vector<int32_t> bstart((size_t)nbk + 1, 0);
    std::vector<int> brange((size_t)n_tets * 6);
    for (int64_t e = 0; e < n_tets; ++e) {
        for (int k = 0; k < 3; ++k) {
            double mn = INFINITY, mx = -INFINITY;
            for (int a = 0; a < 4; ++a) {
                const double v = hx[3 * (size_t)ht[4 * e + a] + k];
                mn = std::min(mn, v);
                mx = std::max(mx, v);
            }
            const double pad = 1e-9 * ext[k];
            int i0 = (int)std::floor((mn - pad - lo[k]) * inv_cell[k]);
            int i1 = (int)std::floor((mx + pad - lo[k]) * inv_cell[k]);
            brange[6 * e + 2 * k] = std::max(0, std::min(nb[k] - 1, i0));
            brange[6 * e + 2 * k + 1] = std::max(0, std::min(nb[k] - 1, i1));
        }
        for (int z = brange[6 * e + 4]; z <= brange[6 * e + 5]; ++z)
            for (int y = brange[6 * e + 2]; y <= brange[6 * e + 3]; ++y)
                for (int x = brange[6 * e]; x <= brange[6 * e + 1]; ++x)
                    bstart[(size_t)(x + (int64_t)nb[0] * (y + (int64_t)nb[1] * z)) + 1] += 1;
    }
    for (int64_t b = 0; b < nbk; ++b) bstart[b + 1] += bstart[b];
    if ((int64_t)bstart[nbk] >= INT32_MAX) return set_error(FSI_ERR_ARG, "bucket lists too long");
    std::vector<int32_t> btets(bstart[nbk]);
    {
        std::vector<int32_t> cur(bstart.begin(), bstart.end() - 1);
        for (int64_t e = 0; e < n_tets; ++e)
            for (int z = brange[6 * e + 4]; z <= brange[6 * e + 5]; ++z)
                for (int y = brange[6 * e + 2]; y <= brange[6 * e + 3]; ++y)
                    for (int x = brange[6 * e]; x <= brange[6 * e + 1]; ++x)
                        btets[cur[x + (int64_t)nb[0] * (y + (int64_t)nb[1] * z)]++] = (int32_t)e;
    }

    fsi_tetmesh *m = new fsi_tetmesh();
    m->device = device;
    m->stream = s;
    m->n_nodes = n_nodes;
    m->n_elems = n_tets;
    m->phys = *phys;
    const double r = phys->rho_inf;
    m->alpha_m = 0.5 * (3.0 - r) / (1.0 + r);
    m->alpha_f = 1.0 / (1.0 + r);
    m->gamma = 0.5 + m->alpha_m - m->alpha_f;
    for (int k = 0; k < 3; ++k) {
        m->nb[k] = nb[k];
        m->lo[k] = lo[k];
        m->inv_cell[k] = inv_cell[k];
        m->box_lo[k] = lo[k] - 1e-9 * ext[k];
        m->box_hi[k] = hi[k] + 1e-9 * ext[k];
    }
    const int64_t ntmp = cell_table_scan_ints(n_tets) + 16;
    bool ok = cudaMalloc(&m->X64, n_nodes * sizeof(double4)) == cudaSuccess &&
              cudaMalloc(&m->X32, n_nodes * sizeof(float4)) == cudaSuccess &&
              cudaMalloc(&m->tets, n_tets * sizeof(int4)) == cudaSuccess &&
              cudaMalloc(&m->node_start, nstart.size() * sizeof(int32_t)) == cudaSuccess &&
              cudaMalloc(&m->node_slot, nslot.size() * sizeof(int32_t)) == cudaSuccess &&
              cudaMalloc(&m->bucket_start, bstart.size() * sizeof(int32_t)) == cudaSuccess &&
              cudaMalloc(&m->bucket_tets, std::max<size_t>(1, btets.size()) * sizeof(int32_t)) ==
                  cudaSuccess &&
              cudaMalloc(&m->slot_scratch, (size_t)n_tets * 4 * 32) == cudaSuccess &&
              cudaMalloc(&m->corner_scratch, (size_t)n_tets * 12 * 8) == cudaSuccess &&
              cudaMalloc(&m->fill, (size_t)(n_tets + 1) * sizeof(int32_t)) == cudaSuccess &&
              cudaMalloc(&m->scan_tmp, (size_t)ntmp * sizeof(int32_t)) == cudaSuccess &&
              cudaMalloc(&m->nout, sizeof(unsigned long long)) == cudaSuccess &&
              cudaMalloc(&m->colors, (size_t)n_nodes * sizeof(int32_t)) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        fsi_tetmesh_destroy(m);
        return set_error(FSI_ERR_OOM, "fsi_tetmesh_create: cudaMalloc failed");
    }
    auto up = [&](void *dst, const void *src, size_t bytes) {
        return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, s) == cudaSuccess;
    };
    ok = cudaMemcpyAsync(m->tets, tets, n_tets * sizeof(int4), cudaMemcpyDeviceToDevice, s) ==
             cudaSuccess &&
         cudaMemsetAsync(m->scan_tmp, 0, (size_t)ntmp * sizeof(int32_t), s) == cudaSuccess &&
         up(m->node_start, nstart.data(), nstart.size() * sizeof(int32_t)) &&
         up(m->node_slot, nslot.data(), nslot.size() * sizeof(int32_t)) &&
         up(m->bucket_start, bstart.data(), bstart.size() * sizeof(int32_t)) &&
         (btets.empty() || up(m->bucket_tets, btets.data(), btets.size() * sizeof(int32_t))) &&
         up(m->colors, hcol.data(), hcol.size() * sizeof(int32_t));
    m->n_colors = ncol;
    if (!ok) {
        fsi_tetmesh_destroy(m);
        return set_error(FSI_ERR_CUDA, "fsi_tetmesh_create: copy failed");
    }
    pad_tet_coords_kernel<<<grid_for(n_nodes, 256), 256, 0, s>>>(n_nodes, X, m->X64, m->X32);
    fsi_status st = check_launch("pad coordinates kernel");
    if (st == FSI_OK) st = check_cuda(cudaStreamSynchronize(s), "sync");
    if (st != FSI_OK) {
        fsi_tetmesh_destroy(m);
        return st;
    }
    *out = m;
    return FSI_OK;
}

void fsi_tetmesh_destroy(fsi_tetmesh *m)
{
    if (!m) return;
    fsi::DeviceGuard _fsi_device_guard(m->device);
    if (m->stream) cudaStreamSynchronize(m->stream);
    cudaFree(m->X64);
    cudaFree(m->X32);
    cudaFree(m->tets);
    cudaFree(m->node_start);
    cudaFree(m->node_slot);
    cudaFree(m->bucket_start);
    cudaFree(m->bucket_tets);
    cudaFree(m->slot_scratch);
    cudaFree(m->corner_scratch);
    cudaFree(m->fill);
    cudaFree(m->scan_tmp);
    cudaFree(m->nout);
    cudaFree(m->colors);
    for (void *g : m->geo) cudaFree(g);
    delete m;
}

fsi_status fsi_tet_residual(fsi_tetmesh *m, fsi_prec prec, const void *U, const void *A,
                            const void *f, void *R)
{
    FSI_TRY(validate_tetmesh(m));
    if (!U || !A || !R) return set_error(FSI_ERR_ARG, "fsi_tet_residual: NULL argument");
    FSI_DEVICE(m->device);
    if (prec == FSI_F64) return tet_vms<double, false>(m, U, A, f, nullptr, R);
    if (prec == FSI_DF64) return tet_vms<df64, false>(m, U, A, f, nullptr, R);
    if (prec == FSI_F32) return tet_vms<float, false>(m, U, A, f, nullptr, R);
    return set_error(FSI_ERR_ARG, "bad precision");
}

fsi_status fsi_tet_jacobian_apply(fsi_tetmesh *m, fsi_prec prec, const void *U, const void *A,
                                  const void *f, const void *x, void *Jx)
{
    FSI_TRY(validate_tetmesh(m));
    if (!U || !A || !x || !Jx) return set_error(FSI_ERR_ARG, "fsi_tet_jacobian_apply: NULL argument");
    FSI_DEVICE(m->device);
    if (prec == FSI_F64) return tet_vms<double, true>(m, U, A, f, x, Jx);
    if (prec == FSI_DF64) return tet_vms<df64, true>(m, U, A, f, x, Jx);
    if (prec == FSI_F32) return tet_vms<float, true>(m, U, A, f, x, Jx);
    return set_error(FSI_ERR_ARG, "bad precision");
}

fsi_status fsi_tet_locate(fsi_tetmesh *m, int64_t np, const double *P, int32_t *elem,
                          double *lam, int32_t *cell_start, int32_t *perm, int64_t *n_outside)
{
    FSI_TRY(validate_tetmesh(m));
    if (np < 0 || np >= INT32_MAX) return set_error(FSI_ERR_ARG, "fsi_tet_locate: bad m");
    if (np > 0 && (!P || !elem || !lam))
        return set_error(FSI_ERR_ARG, "fsi_tet_locate: NULL P, elem or lam");
    if (perm != nullptr && cell_start == nullptr)
        return set_error(FSI_ERR_ARG, "fsi_tet_locate: perm given without cell_start");
    if (cell_start != nullptr && perm == nullptr && np > 0)
        return set_error(FSI_ERR_ARG, "fsi_tet_locate: cell_start given without perm");
    FSI_DEVICE(m->device);
    cudaStream_t s = m->stream;
    const int64_t E = m->n_elems;
    const bool table = cell_start != nullptr;
    FSI_CUDA(cudaMemsetAsync(m->nout, 0, sizeof(unsigned long long), s), "memset");
    if (table) FSI_CUDA(cudaMemsetAsync(m->fill, 0, (E + 1) * sizeof(int32_t), s), "memset");
    if (np > 0) {
        BucketArgs B;
        for (int k = 0; k < 3; ++k) {
            B.nb[k] = m->nb[k];
            B.lo[k] = m->lo[k];
            B.inv_cell[k] = m->inv_cell[k];
            B.box_lo[k] = m->box_lo[k];
            B.box_hi[k] = m->box_hi[k];
        }
        int npw = 4;
        while (npw < 16 && np > (int64_t)npw * 16 * sm_count()) npw *= 2;
        // (16 CTAs an SM, warps striding: 300,000 points in 24,576 elements 201 us with 32, 188)
        tet_locate_kernel<<<grid_for((np + npw - 1) / npw * 32, kLocThreads, sm_count() * 16),
                            kLocThreads, 0, s>>>(
            np, B, m->X64, m->X32, m->tets, m->bucket_start, m->bucket_tets, P, npw, elem, lam,
            table ? m->fill : nullptr, m->nout);
        FSI_TRY(check_launch("tet locate kernel"));
    }
    if (table) FSI_TRY(build_cell_table(s, E, np, elem, m->fill, m->scan_tmp, cell_start, perm));
    if (n_outside) {
        unsigned long long h = 0;
        FSI_CUDA(cudaMemcpyAsync(&h, m->nout, sizeof h, cudaMemcpyDeviceToHost, s), "memcpy");
        FSI_CUDA(cudaStreamSynchronize(s), "stream sync");
        *n_outside = (int64_t)h;
    }
    return FSI_OK;
}

fsi_status fsi_tet_interp(fsi_tetmesh *m, fsi_prec prec, int64_t np, const int32_t *elem,
                          const void *lam, const void *U, void *u)
{
    FSI_TRY(validate_tetmesh(m));
    if (np < 0 || np >= INT32_MAX) return set_error(FSI_ERR_ARG, "fsi_tet_interp: bad m");
    if (np == 0) return FSI_OK;
    if (!elem || !lam || !U || !u) return set_error(FSI_ERR_ARG, "fsi_tet_interp: NULL argument");
    FSI_DEVICE(m->device);
    const int g = grid_for(np, 256);
    if (prec == FSI_F64)
        tet_interp_kernel<double><<<g, 256, 0, m->stream>>>(np, m->n_elems, m->tets, elem,
                                                            (const double *)lam,
                                                            (const vec4<double> *)U, (double *)u);
    else if (prec == FSI_DF64)
        tet_interp_kernel<df64><<<g, 256, 0, m->stream>>>(np, m->n_elems, m->tets, elem,
                                                          (const double *)lam,
                                                          (const vec4<double> *)U, (double *)u);
    else if (prec == FSI_F32)
        tet_interp_kernel<float><<<g, 256, 0, m->stream>>>(np, m->n_elems, m->tets, elem,
                                                           (const float *)lam,
                                                           (const vec4<float> *)U, (float *)u);
    else
        return set_error(FSI_ERR_ARG, "bad precision");
    return check_launch("tet interp kernel");
}

fsi_status fsi_tet_spread(fsi_tetmesh *m, fsi_prec prec, int64_t np, const int32_t *elem,
                          const void *lam, const int32_t *cell_start, const int32_t *perm,
                          const void *lamv, const void *w, void *F, int accumulate)
{
    (void)elem;
    FSI_TRY(validate_tetmesh(m));
    if (np < 0 || np >= INT32_MAX) return set_error(FSI_ERR_ARG, "fsi_tet_spread: bad m");
    if (!F || !cell_start) return set_error(FSI_ERR_ARG, "fsi_tet_spread: NULL F or cell_start");
    if (np > 0 && (!lam || !perm || !lamv))
        return set_error(FSI_ERR_ARG, "fsi_tet_spread: NULL lam, perm or forces");
    FSI_DEVICE(m->device);
    const int64_t E = m->n_elems;
    const int cg = grid_for((E + 7) / 8 * 32, 256, sm_count() * 64);
    const int ng = (int)((4 * m->n_nodes + 255) / 256);
    cudaStream_t s = m->stream;
    if (prec == FSI_F64) {
        tet_spread_cells_kernel<double><<<cg, 256, 0, s>>>(E, (const double *)lam, cell_start, perm,
                                                           (const double *)lamv,
                                                           (const double *)w,
                                                           (double *)m->corner_scratch);
        FSI_TRY(check_launch("tet spread cells kernel"));
        launch_chain(tet_spread_nodes_kernel<double>, ng, 256, 0, s, m->n_nodes, m->node_start, m->node_slot,
                                                           cell_start,
                                                           (const double *)m->corner_scratch,
                                                           (double *)F, accumulate);
    } else if (prec == FSI_DF64) {
        tet_spread_cells_kernel<df64><<<cg, 256, 0, s>>>(E, (const double *)lam, cell_start, perm,
                                                         (const double *)lamv, (const double *)w,
                                                         (df64 *)m->corner_scratch);
        FSI_TRY(check_launch("tet spread cells kernel"));
        launch_chain(tet_spread_nodes_kernel<df64>, ng, 256, 0, s, m->n_nodes, m->node_start, m->node_slot,
                                                         cell_start,
                                                         (const df64 *)m->corner_scratch,
                                                         (double *)F, accumulate);
    } else if (prec == FSI_F32) {
        tet_spread_cells_kernel<float><<<cg, 256, 0, s>>>(E, (const float *)lam, cell_start, perm,
                                                          (const float *)lamv, (const float *)w,
                                                          (float *)m->corner_scratch);
        FSI_TRY(check_launch("tet spread cells kernel"));
        launch_chain(tet_spread_nodes_kernel<float>, ng, 256, 0, s, m->n_nodes, m->node_start, m->node_slot,
                                                          cell_start,
                                                          (const float *)m->corner_scratch,
                                                          (float *)F, accumulate);
    } else {
        return set_error(FSI_ERR_ARG, "bad precision");
    }
    return check_launch("tet spread nodes kernel");
}

}  // extern "C"
