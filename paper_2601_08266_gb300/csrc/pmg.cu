// pmg.cu -- pressure block of the Schur-complement block preconditioner
// (Sec. 2.4 solves the reduced system with block preconditioners built from
// its sub-matrices).  For the saddle-point blocks [[A, B], [C, D]] of the
// linearised fluid system with a mass-dominated velocity block
// A ~ alpha_m rho M, the pressure Schur complement D - C A^{-1} B acts like
// sigma K, K the Q1 stiffness matrix of the pressure space and
// sigma = alpha_f gamma dt / (alpha_m rho).  The preconditioner replaces it by
// sigma (K + kappa M), kappa = (pi / (2 L))^2 with L the largest extent of the
// grid (M the Q1 mass matrix; the shift keeps the operator non-singular where
// only Neumann conditions bound the pressure).  On faces of the box where the
// velocity is free (traction-free outflow) the true Schur complement acts like
// a Dirichlet problem for the pressure, so the nodes of such faces are
// eliminated (rows and columns dropped, diagonal kept; the restricted
// right-hand side is zeroed there).  The approximation is inverted with one
// geometric multigrid V-cycle on the uniform grid:
//
//   levels     the mesh grid, then every other node while all N_d are even and
//              the grid has more than 125 nodes;
//   operator   K + kappa M applied matrix-free: on a uniform grid both are
//              tensor products of the 1D linear-element matrices
//              M1 = h/6 [1 4 1] (h/3 on boundary nodes) and
//              K1 = 1/h [-1 2 -1] (1/h on boundary nodes):
//              K = K1 x M1 x M1 + M1 x K1 x M1 + M1 x M1 x K1;
//   transfer   trilinear interpolation P, restriction P^T (weights 1, 1/2);
//              the coarse operators equal P^T A P (Galerkin) exactly;
//   smoother   Chebyshev semi-iteration of degree 2 on D^{-1} A over
//              [hi/4, hi], hi = 1.1 x the largest symbol/diagonal ratio over
//              the modes theta_d in {0, pi} (pre- and post-smoothing);
//   coarsest   a dense inverse (<= 1000 nodes, built once on the host in
//              FP64) or, on grids that do not coarsen, Chebyshev degree 8 over
//              [hi/30, hi].
//
// The V-cycle is a fixed linear operator (symmetric), so it can precondition
// plain GMRES.  The stencil and transfer kernels march up columns of nodes, a thread
// or lane each; the FP32 levels of at most 17^3 nodes run as one cluster of CTAs
// (coarse_cycle_kernel); the rest is a thread per node.  Deterministic; FP64 or FP32
// arithmetic follows the caller's precision.
#include <algorithm>
#include <cmath>
#include <cooperative_groups.h>
#include <cuda_pipeline.h>
#include <type_traits>
#include <vector>

#include "fsi_internal.cuh"

namespace fsi {

constexpr int kPmgMaxLevels = 16;
constexpr int kPmgNu = 2;
constexpr int kPmgCoarseDegree = 8;
constexpr int64_t kPmgDirectMax = 1000;
constexpr int64_t kPmgMinCoarsen = 125;

struct PmgLevel {
    int N[3];
    double h[3];
    int64_t n;
    double hi;          // Chebyshev upper bound of D^{-1} A
    // level vectors, 8 bytes per entry (either precision fits): right-hand
    // side, solution, residual (also the second x buffer of the smoother),
    // pre-smoothed iterate, two smoother directions, one more x buffer
    void *b, *x, *r, *t, *d0, *d1, *xa;
};

struct PressureMG {
    int nlev = 0;
    PmgLevel lev[kPmgMaxLevels];
    double kappa = 0.0;
    int faces[6] = {0, 0, 0, 0, 0, 0};  // eliminated faces x0, x1, y0, y1, z0, z1
    bool direct = false;
    int64_t nc = 0;
    double *inv64 = nullptr;  // [nc][nc]
    float *inv32 = nullptr;
};

namespace {

// 1D coefficients of a level in the working type: mass and stiffness
// entries of interior / boundary diagonals and of the off-diagonals.
namespace cg = cooperative_groups;

template <typename T> struct Axis {
    int N;
    T m_in, m_bd, m_off, k_in, k_bd, k_off;
};

template <typename T> struct LevelArgs {
    Axis<T> a[3];
    T kappa;
    int NX1, NY1, NZ1;
    int faces[6];
};

template <typename T> LevelArgs<T> level_args(const PressureMG &P, int l)
{
    const PmgLevel &L = P.lev[l];
    LevelArgs<T> A;
    for (int d = 0; d < 3; ++d) {
        const double h = L.h[d];
        A.a[d] = {L.N[d], (T)(2.0 * h / 3.0), (T)(h / 3.0), (T)(h / 6.0),
                  (T)(2.0 / h), (T)(1.0 / h), (T)(-1.0 / h)};
    }
    A.kappa = (T)P.kappa;
    A.NX1 = L.N[0] + 1;
    A.NY1 = L.N[1] + 1;
    A.NZ1 = L.N[2] + 1;
    for (int f = 0; f < 6; ++f) A.faces[f] = P.faces[f];
    return A;
}

// node (i, j, k) lies on an eliminated face
template <typename T>
__device__ __forceinline__ bool eliminated(const LevelArgs<T> &L, int i, int j, int k)
{
    return (L.faces[0] && i == 0) || (L.faces[1] && i == L.NX1 - 1) ||
           (L.faces[2] && j == 0) || (L.faces[3] && j == L.NY1 - 1) ||
           (L.faces[4] && k == 0) || (L.faces[5] && k == L.NZ1 - 1);
}

// entries (mass, stiffness) of row i, column i + d (|d| <= 1, in range)
template <typename T>
__device__ __forceinline__ void coef(const Axis<T> &a, int i, int d, T &m, T &k)
{
    if (d == 0) {
        const bool bd = (i == 0) || (i == a.N);
        m = bd ? a.m_bd : a.m_in;
        k = bd ? a.k_bd : a.k_in;
    } else {
        m = a.m_off;
        k = a.k_off;
    }
}

template <typename T> __device__ __forceinline__ T diag_of(const LevelArgs<T> &L, int i, int j, int k)
{
    T mx, kx, my, ky, mz, kz;
    coef(L.a[0], i, 0, mx, kx);
    coef(L.a[1], j, 0, my, ky);
    coef(L.a[2], k, 0, mz, kz);
    return kx * my * mz + mx * ky * mz + mx * my * kz + L.kappa * mx * my * mz;
}

// v = x + d at a node (x == null: v = d; d == null: v = x)
template <typename T>
__device__ __forceinline__ T val(const T *__restrict__ x, const T *__restrict__ d, int64_t q)
{
    return x ? (d ? x[q] + d[q] : x[q]) : d[q];
}

// One thread per (i, j) column on a 3D launch, x and y from the block and
// thread indices, striding over the planes k from the grid's z index (no
// per-node division; a CTA does several planes, so tiny CTAs do not make the
// CTA launches the limit).
#define NODE3(L, i, j, k)                                                                   \
    const int i = blockIdx.x * blockDim.x + threadIdx.x;                                 \
    const int j = blockIdx.y * blockDim.y + threadIdx.y;                                 \
    if (i >= (L).NX1 || j >= (L).NY1) return;                                            \
    for (int k = blockIdx.z; k < (L).NZ1; k += gridDim.z)

// Chebyshev, first direction from x = 0: d0 = D^{-1} b / theta, or with
// x_out (degree 1) x_out = d0.  (From a nonzero x the first direction needs
// A x: march_kernel in kMarchCheb0 mode.)
template <typename T>
__global__ void cheb0_kernel(LevelArgs<T> L, const T *__restrict__ b, T inv_theta,
                             T *__restrict__ d_out, T *__restrict__ x_out)
{
    NODE3(L, i, j, k)
    {
        const int64_t node = i + (int64_t)L.NX1 * (j + (int64_t)L.NY1 * k);
        const T d0 = inv_theta * b[node] / diag_of(L, i, j, k);
        if (x_out)
            x_out[node] = d0;
        else
            d_out[node] = d0;
    }
}

// ---------------------------------------------------------------- z-marching stencil
// The operator A = K + kappa M of a level is a tensor product of symmetric 1D Q1
// rows (stiffness k, mass m per axis), so with S_0 the node's value, S_x the sum of
// its two x neighbours, S_y of the y neighbours and S_xy of the four diagonal ones
// in a plane, (A v)(k) = PA(k) + PB(k - 1) + PB(k + 1), PA = sum_c A_c S_c and PB =
// sum_c B_c S_c.  The 8 weights depend on the node's place along x only: a
// boundary node's own 1D entries are exactly half of an inner one's, so on a
// boundary row S_0 and S_x, and on a boundary plane PA, count half, and 1/D takes
// factors of two.
//
// A lane owns a column in x, a warp 32 of them (the outer two are halo: 30 give
// results) by R rows, and marches up kz planes: x neighbours come by shuffles, y
// neighbours are the lane's own rows, the z fold is held in registers; the next
// plane's loads are in flight while a plane is folded.  No shared memory and no
// barrier: with both (x rows formed once per CTA, three barriers a plane) the four
// passes of a smoothing at 129^3 took 145 us in FP32, now 88 us.  v is zero
// outside the grid and on eliminated nodes (whose columns A does not have); rows of
// eliminated nodes keep only the diagonal.  Fixed order of sums (deterministic).
constexpr int kMarchOut = 30;    // columns of results per warp
constexpr int kMarchWarps = 4;   // warps per CTA, one row group each

template <typename T> struct March {
    const T *x, *d;  // v = x + d (VX selects which are present)
    const T *b;
    T c1, c2, inv_theta;
    T *y, *x_next, *d_next, *x_final;
    int kz;          // planes per warp
    // with z4 (a step's x_final): the result goes to z4[4 node + 3] as
    // x_final * inv_sigma, or v4[4 node + 3] where m4[4 node + 3] is set
    T *z4;
    const T *v4;
    const uint8_t *m4;
    T inv_sigma;
};

enum MarchMode { kMarchApply = 0, kMarchCheb0 = 1, kMarchStep = 2 };
// the vector v the stencil acts on: d alone, x alone, x + d, or (kVb) the
// first Chebyshev direction from x = 0, d0 = b / (theta D), formed from b at
// every staged node (so no pass writes d0 first)
enum MarchSource { kVd = 0, kVx = 1, kVxd = 2, kVb = 3 };

template <typename T>
__device__ __forceinline__ T md_of(const Axis<T> &a, int i)
{
    return (i == 0 || i == a.N) ? a.m_bd : a.m_in;
}
template <typename T>
__device__ __forceinline__ T kd_of(const Axis<T> &a, int i)
{
    return (i == 0 || i == a.N) ? a.k_bd : a.k_in;
}
template <typename T, int MODE, int VX, int R>
__global__ void __launch_bounds__(32 * kMarchWarps) march_kernel(LevelArgs<T> L, March<T> M)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x;
    const int i = blockIdx.x * kMarchOut + lane - 1, j0 = (blockIdx.y * kMarchWarps + threadIdx.y) * R;
    const int k0 = blockIdx.z * M.kz, k1 = min(k0 + M.kz, L.NZ1);  // planes k0 .. k1-1 are output
    if (j0 >= L.NY1) return;
    const Axis<T> &ax = L.a[0], &ay = L.a[1], &az = L.a[2];
    const int64_t plane_n = (int64_t)L.NX1 * L.NY1;
    const bool inx = i >= 0 && i < L.NX1;
    const bool elx = (L.faces[0] && i == 0) || (L.faces[1] && i == L.NX1 - 1);
    // rows j0 - 1 .. j0 + R: in the grid, not eliminated, half weights
    bool in[R + 2], ok[R + 2];
#pragma unroll
    for (int r = 0; r < R + 2; ++r) {
        const int j = j0 - 1 + r;
        in[r] = inx && j >= 0 && j < L.NY1;
        ok[r] = in[r] && !elx && !((L.faces[2] && j == 0) || (L.faces[3] && j == L.NY1 - 1));
    }
    auto bdy = [&](int r) { const int j = j0 - 1 + r; return j == 0 || j == L.NY1 - 1; };
    T A[4], B[4];
    {
        const T mx = md_of(ax, i), kx = kd_of(ax, i);
        const T ky = ay.k_in + L.kappa * ay.m_in, kyo = ay.k_off + L.kappa * ay.m_off;
        const T P[4] = {kx * ay.m_in + mx * ky, ax.k_off * ay.m_in + ax.m_off * ky,
                        kx * ay.m_off + mx * kyo, ax.k_off * ay.m_off + ax.m_off * kyo};
        const T Q[4] = {mx * ay.m_in, ax.m_off * ay.m_in, mx * ay.m_off, ax.m_off * ay.m_off};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            A[c] = P[c] * az.m_in + Q[c] * az.k_in;
            B[c] = P[c] * az.m_off + Q[c] * az.k_off;
        }
    }
    const T iA0 = T(1) / A[0];
    const int64_t off = i + (int64_t)L.NX1 * (j0 - 1);
    auto elz = [&](int k) { return (L.faces[4] && k == 0) || (L.faces[5] && k == L.NZ1 - 1); };
    auto bdz = [&](int k) { return k == 0 || k == L.NZ1 - 1; };

    // a plane as loaded: x (or b, VX = kVb) and d
    struct Raw {
        T x[R + 2], d[R + 2];
    };
    auto load = [&](int k, Raw &w) {
        const bool inz = k >= 0 && k < L.NZ1;
        const int64_t q = off + plane_n * k;
#pragma unroll
        for (int r = 0; r < R + 2; ++r) {
            const bool g = inz && in[r];
            if constexpr (VX != kVd) w.x[r] = g ? __ldcg((VX == kVb ? M.b : M.x) + q + (int64_t)L.NX1 * r) : T(0);
            if constexpr (VX == kVd || VX == kVxd) w.d[r] = g ? __ldcg(M.d + q + (int64_t)L.NX1 * r) : T(0);
        }
    };
    // v from a loaded plane's row
    auto value = [&](const Raw &w, int r, T gz) {
        if constexpr (VX == kVd) return w.d[r];
        else if constexpr (VX == kVx) return w.x[r];
        else if constexpr (VX == kVxd) return w.x[r] + w.d[r];
        else return M.inv_theta * w.x[r] * (iA0 * (bdy(r) ? gz + gz : gz));
    };

    // per output row: fz PA(k) + PB(k - 1) and PB(k) of the plane k below the
    // current one, and that plane's v, d and b at the node
    T acc[R], PBk[R], vk[R], dk[R], bk[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = PBk[r] = vk[r] = dk[r] = bk[r] = T(0);
    Raw nx;
    // A call's last kernel (a smoothing's, or y = A x for a caller) lets the next start
    // only when those before it are done: that one is the caller's choice, and
    // applications in a row that were all let in at once shared the SMs unevenly (FP64,
    // 25^3 nodes 12.8 -> 8.4 us, 65^3 44.9 -> 38.3 us).
    const bool last = M.x_final || M.z4 || (MODE == kMarchApply && !M.b);
    if (!last) chain_trigger();
    chain_wait(M.x, M.d, M.b, M.y, M.x_next, M.d_next, M.x_final, M.z4, M.v4, M.m4);
    if (last) chain_trigger();
    load(k0 - 1, nx);
    for (int kk = k0 - 1; kk <= k1; ++kk) {
        const Raw w = nx;
        if (kk < k1) load(kk + 1, nx);
        const bool zb = bdz(kk), vz = kk >= 0 && kk < L.NZ1 && !elz(kk);
        const T gz = zb ? T(2) : T(1), fz = zb ? T(0.5) : T(1);
        // the node inputs of this plane's results, used one plane later
        T bn[R];
        const bool mine = kk >= k0 && kk < k1;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            bn[r] = T(0);
            if constexpr (VX == kVb) bn[r] = w.x[r + 1];
            else if (M.b && mine && in[r + 1])
                bn[r] = __ldcg(M.b + off + plane_n * kk + (int64_t)L.NX1 * (r + 1));
        }
        T v[R + 2], X[R + 2];
#pragma unroll
        for (int r = 0; r < R + 2; ++r) {
            v[r] = vz && ok[r] ? value(w, r, gz) : T(0);
            X[r] = __shfl_up_sync(kAll, v[r], 1) + __shfl_down_sync(kAll, v[r], 1);
        }
        const int k = kk - 1;  // the plane that is complete now
        const bool out = k >= k0 && inx && lane >= 1 && lane <= kMarchOut;
        const bool kb = bdz(k), kel = elz(k);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const T fy = bdy(r + 1) ? T(0.5) : T(1);
            const T S0 = fy * v[r + 1], Sx = fy * X[r + 1], Sy = v[r] + v[r + 2], Sxy = X[r] + X[r + 2];
            const T PA = A[0] * S0 + A[1] * Sx + A[2] * Sy + A[3] * Sxy;
            const T PB = B[0] * S0 + B[1] * Sx + B[2] * Sy + B[3] * Sxy;
            if (out && in[r + 1]) {
                const int64_t node = off + plane_n * k + (int64_t)L.NX1 * (r + 1);
                const T g = (kb ? T(2) : T(1)) * (bdy(r + 1) ? T(2) : T(1)), inv_D = iA0 * g;
                const T Av = ok[r + 1] && !kel ? acc[r] + PB : A[0] * (fy * (kb ? T(0.5) : T(1))) * vk[r];
                if constexpr (MODE == kMarchApply) {
                    M.y[node] = M.b ? bk[r] - Av : Av;
                } else if constexpr (MODE == kMarchCheb0) {
                    // first Chebyshev direction from x (not null here)
                    const T d0 = M.inv_theta * (bk[r] - Av) * inv_D;
                    if (M.x_final)
                        M.x_final[node] = vk[r] + d0;
                    else
                        M.d_next[node] = d0;
                } else {
                    const T dn = M.c1 * dk[r] + M.c2 * ((bk[r] - Av) * inv_D);
                    if (M.z4) {
                        M.z4[4 * node + 3] = (M.m4 && M.m4[4 * node + 3]) ? __ldcg(M.v4 + 4 * node + 3)
                                                                         : (vk[r] + dn) * M.inv_sigma;
                    } else if (M.x_final) {
                        M.x_final[node] = vk[r] + dn;
                    } else {
                        M.x_next[node] = vk[r];
                        M.d_next[node] = dn;
                    }
                }
            }
            acc[r] = fz * PA + PBk[r];
            PBk[r] = PB;
            vk[r] = value(w, r + 1, gz);  // also where it is eliminated
            if constexpr (MODE == kMarchStep) dk[r] = VX == kVb ? vk[r] : w.d[r + 1];
            bk[r] = bn[r];
        }
    }
}

template <typename T, int MODE, int VX, int R>
fsi_status march_rows(const PressureMG &P, int l, cudaStream_t s, March<T> M)
{
    const PmgLevel &L = P.lev[l];
    const int nz1 = L.N[2] + 1;
    const int gx = (L.N[0] + kMarchOut) / kMarchOut, gy = (L.N[1] + R) / R;
    // planes per warp: 12 warps an SM (a warp reads two planes more than it
    // writes, and its planes are a serial chain), 1 to 16
    M.kz = (int)std::max<int64_t>(1, std::min<int64_t>(16, (int64_t)nz1 * gx * gy / (12 * sm_count())));
    const dim3 grid((unsigned)gx, (unsigned)((gy + kMarchWarps - 1) / kMarchWarps),
                    (unsigned)((nz1 + M.kz - 1) / M.kz));
    launch_chain(march_kernel<T, MODE, VX, R>, grid, dim3(32, kMarchWarps), 0, s, level_args<T>(P, l), M);
    return check_launch("pressure stencil");
}
// Rows per warp: more rows share their neighbours' loads, fewer give short vectors
// more warps (a mixed step at 32^3 with 4, 2, 1 rows: 7.93, 7.77, 7.65 ms; FP64 at
// 24^3: 37.2, 33.2, 31.1 ms; 129^3 gains from 4, 65^3 is level between 2 and 4)
template <typename T, int MODE, int VX>
fsi_status march_launch(const PressureMG &P, int l, cudaStream_t s, const March<T> &M)
{
    if (P.lev[l].n >= 400000) return march_rows<T, MODE, VX, 4>(P, l, s, M);
    if (P.lev[l].n >= 100000) return march_rows<T, MODE, VX, 2>(P, l, s, M);
    return march_rows<T, MODE, VX, 1>(P, l, s, M);
}

// the stencil pass in MODE: on v = M.x (apply, first Chebyshev direction) or
// v = M.x + M.d (Chebyshev step; M.x null after a zero start; both null: the
// first step from x = 0, v = d0 = b / (theta D) formed in the pass)
template <typename T, int MODE>
fsi_status march(const PressureMG &P, int l, cudaStream_t s, const March<T> &M)
{
    if constexpr (MODE == kMarchStep) {
        if (M.x) return march_launch<T, MODE, kVxd>(P, l, s, M);
        if (M.d) return march_launch<T, MODE, kVd>(P, l, s, M);
        if (!M.b) return FSI_ERR_ARG;
        return march_launch<T, MODE, kVb>(P, l, s, M);  // the first step from x = 0
    } else {
        if (!M.x) return FSI_ERR_ARG;
        return march_launch<T, MODE, kVx>(P, l, s, M);
    }
}

// y = A x (b == null) or y = b - A x on level l
template <typename T>
fsi_status level_apply(const PressureMG &P, int l, cudaStream_t s, const T *x, const T *b, T *y)
{
    March<T> M{};
    M.x = x;
    M.b = b;
    M.y = y;
    return march<T, kMarchApply>(P, l, s, M);
}

// b_c = P^T r: each coarse node gathers the fine nodes within one fine cell,
// weights 1 (coincident) and 1/2 (neighbour) per axis; zero on eliminated nodes.
// A thread has a coarse column (I, J) and goes up kz coarse planes: a fine plane's
// 3 x 3 sum is formed once for the two coarse planes that it belongs to
template <typename T>
__global__ void restrict_kernel(LevelArgs<T> F, LevelArgs<T> C, int kz, const T *__restrict__ r,
                                T *__restrict__ bc)
{
    const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
    if (I >= C.NX1 || J >= C.NY1) return;
    const int K0 = blockIdx.z * kz, K1 = min(K0 + kz, C.NZ1);
    const int xl = I > 0 ? 1 : 0, xr = 2 * I + 1 < F.NX1 ? 1 : 0, yl = J > 0 ? F.NX1 : 0,
              yr = 2 * J + 1 < F.NY1 ? F.NX1 : 0;
    const T wl = xl ? T(0.5) : T(0), wr = xr ? T(0.5) : T(0), vl = yl ? T(0.5) : T(0),
            vr = yr ? T(0.5) : T(0);
    const int64_t plane_n = (int64_t)F.NX1 * F.NY1, off = 2 * I + (int64_t)F.NX1 * (2 * J);
    auto plane = [&](int k) {
        if (k < 0 || k >= F.NZ1) return T(0);
        const T *q = r + off + plane_n * k;
        auto at = [&](int o) { return __ldcg(q + o); };
        const T a = at(0) + wl * at(-xl) + wr * at(xr);
        const T b = at(-yl) + wl * at(-yl - xl) + wr * at(xr - yl);
        const T c = at(yr) + wl * at(yr - xl) + wr * at(yr + xr);
        return a + vl * b + vr * c;
    };
    chain_trigger();
    chain_wait(r, bc);
    T below = plane(2 * K0 - 1);
#pragma unroll 2
    for (int K = K0; K < K1; ++K) {
        const T at = plane(2 * K), above = plane(2 * K + 1);
        bc[I + (int64_t)C.NX1 * (J + (int64_t)C.NY1 * K)] =
            eliminated(C, I, J, K) ? T(0) : at + T(0.5) * (below + above);
        below = above;
    }
}

// x += P x_c: trilinear interpolation of the coarse correction.  A thread has a
// fine column (i, j) and goes up kz coarse planes, two fine nodes for each: the mean
// of the (one, two or four) coarse values around the column in a plane is formed
// once per coarse plane.  (A node at a time with its loops over the coarse
// neighbours took 22 us at 129^3 in FP32, now 12 us.)
template <typename T>
__global__ void prolong_kernel(LevelArgs<T> F, LevelArgs<T> C, int kz, const T *__restrict__ xc,
                               T *__restrict__ x)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= F.NX1 || j >= F.NY1) return;
    const int K0 = blockIdx.z * kz, K1 = min(K0 + kz, C.NZ1);
    const int dx = i & 1, dy = (j & 1) ? C.NX1 : 0;
    const int64_t plane_n = (int64_t)F.NX1 * F.NY1, plane_c = (int64_t)C.NX1 * C.NY1;
    const T *c = xc + (i >> 1) + (int64_t)C.NX1 * (j >> 1);
    T *f = x + i + (int64_t)F.NX1 * j;
    auto plane = [&](int K) {
        const T *q = c + plane_c * K;
        return T(0.25) * ((__ldcg(q) + __ldcg(q + dx)) + (__ldcg(q + dy) + __ldcg(q + dy + dx)));
    };
    chain_trigger();
    chain_wait(c, f);
    T at = plane(K0);
#pragma unroll 2
    for (int K = K0; K < K1; ++K) {
        f[plane_n * (2 * K)] = __ldcg(f + plane_n * (2 * K)) + at;
        if (2 * K + 1 < F.NZ1) {
            const T above = plane(K + 1);
            f[plane_n * (2 * K + 1)] = __ldcg(f + plane_n * (2 * K + 1)) + T(0.5) * (at + above);
            at = above;
        }
    }
}

template <typename T> __global__ void copy_kernel(int64_t n, const T *a, T *b)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n;
         q += (int64_t)gridDim.x * blockDim.x)
        b[q] = a[q];
}

// x = Ainv b on the coarsest grid: one warp per row, fixed reduction order
template <typename T>
__global__ void dense_apply_kernel(int64_t nc, const T *__restrict__ Ainv, const T *__restrict__ b,
                                   T *__restrict__ x)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t row = warp; row < nc; row += nwarps) {
        T s = T(0);
        for (int64_t c = lane; c < nc; c += 32) s += Ainv[row * nc + c] * b[c];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) x[row] = s;
    }
}

int grid_for(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, sm_count() * 16)); }

// transfers: CTAs of 32 nodes along x by 4 along y of L (at 129 nodes per row:
// 81 % of the lanes busy, against 50 % for 128-node rows of CTAs), and along z the
// coarse planes, up to four per thread where that leaves 8 CTAs per SM
const dim3 kRowBlock(32, 4);
dim3 transfer_grid(const PmgLevel &L, const PmgLevel &Lc, int &kz)
{
    const int gx = (L.N[0] + 1 + 31) / 32, gy = (L.N[1] + 1 + 3) / 4;
    kz = (int)std::max<int64_t>(1, std::min<int64_t>(4, (int64_t)gx * gy * (Lc.N[2] + 1) / (8 * sm_count())));
    return dim3((unsigned)gx, (unsigned)gy, (unsigned)((Lc.N[2] + kz) / kz));
}
// node kernels with about 16 CTAs per SM in all, each striding over planes (the
// purely pointwise first smoother direction: 13 -> 8 us at 129^3)
dim3 grid3_strided(const PmgLevel &L)
{
    const int gx = (L.N[0] + 1 + 31) / 32, gy = (L.N[1] + 1 + 3) / 4;
    const int64_t gz = std::max<int64_t>(1, std::min<int64_t>(L.N[2] + 1,
                                                              16 * sm_count() / ((int64_t)gx * gy)));
    return dim3((unsigned)gx, (unsigned)gy, (unsigned)gz);
}

double spectrum_bound(const double h[3], double kappa)
{
    double diag = kappa;
    for (int d = 0; d < 3; ++d) diag *= 2.0 * h[d] / 3.0;
    for (int d = 0; d < 3; ++d) {
        double t = 2.0 / h[d];
        for (int e = 0; e < 3; ++e)
            if (e != d) t *= 2.0 * h[e] / 3.0;
        diag += t;
    }
    double best = 0.0;
    for (int s = 0; s < 8; ++s) {
        double k[3], m[3];
        for (int d = 0; d < 3; ++d) {
            const bool pi = (s >> d) & 1;
            k[d] = pi ? 4.0 / h[d] : 0.0;
            m[d] = pi ? h[d] / 3.0 : h[d];
        }
        const double sym = k[0] * m[1] * m[2] + m[0] * k[1] * m[2] + m[0] * m[1] * k[2] +
                           kappa * m[0] * m[1] * m[2];
        best = std::max(best, sym / diag);
    }
    return 1.1 * best;
}

// Dense K + kappa M of a (small) level from the same 1D coefficients, then
// its inverse by Gauss-Jordan with partial pivoting (FP64, host).
bool dense_inverse(const PmgLevel &L, double kappa, const int faces[6], std::vector<double> &inv)
{
    auto elim = [&](int i, int j, int k) {
        return (faces[0] && i == 0) || (faces[1] && i == L.N[0]) || (faces[2] && j == 0) ||
               (faces[3] && j == L.N[1]) || (faces[4] && k == 0) || (faces[5] && k == L.N[2]);
    };
    const int nx = L.N[0] + 1, ny = L.N[1] + 1, nz = L.N[2] + 1;
    const int64_t n = L.n;
    auto c1 = [&](int d, int i, int off, double &m, double &k) {
        const double h = L.h[d];
        if (off == 0) {
            const bool bd = i == 0 || i == L.N[d];
            m = bd ? h / 3.0 : 2.0 * h / 3.0;
            k = bd ? 1.0 / h : 2.0 / h;
        } else {
            m = h / 6.0;
            k = -1.0 / h;
        }
    };
    std::vector<double> a((size_t)n * 2 * n, 0.0);
    const int64_t w = 2 * n;
    for (int k = 0; k < nz; ++k)
        for (int j = 0; j < ny; ++j)
            for (int i = 0; i < nx; ++i) {
                const int64_t row = i + (int64_t)nx * (j + (int64_t)ny * k);
                for (int dk = -1; dk <= 1; ++dk)
                    for (int dj = -1; dj <= 1; ++dj)
                        for (int di = -1; di <= 1; ++di) {
                            const int ii = i + di, jj = j + dj, kk = k + dk;
                            if (ii < 0 || ii >= nx || jj < 0 || jj >= ny || kk < 0 || kk >= nz)
                                continue;
                            double mx, kx, my, ky, mz, kz;
                            c1(0, i, di, mx, kx);
                            c1(1, j, dj, my, ky);
                            c1(2, k, dk, mz, kz);
                            const int64_t col = ii + (int64_t)nx * (jj + (int64_t)ny * kk);
                            if (col != row && (elim(i, j, k) || elim(ii, jj, kk))) continue;
                            a[row * w + col] = kx * my * mz + mx * ky * mz + mx * my * kz +
                                               kappa * mx * my * mz;
                        }
                a[row * w + n + row] = 1.0;
            }
    for (int64_t c = 0; c < n; ++c) {
        int64_t p = c;
        for (int64_t r = c + 1; r < n; ++r)
            if (std::fabs(a[r * w + c]) > std::fabs(a[p * w + c])) p = r;
        if (!(std::fabs(a[p * w + c]) > 0.0)) return false;
        if (p != c)
            for (int64_t q = 0; q < w; ++q) std::swap(a[p * w + q], a[c * w + q]);
        const double piv = 1.0 / a[c * w + c];
        for (int64_t q = 0; q < w; ++q) a[c * w + q] *= piv;
        for (int64_t r = 0; r < n; ++r)
            if (r != c) {
                const double f = a[r * w + c];
                if (f != 0.0)
                    for (int64_t q = 0; q < w; ++q) a[r * w + q] -= f * a[c * w + q];
            }
    }
    inv.assign((size_t)n * n, 0.0);
    for (int64_t r = 0; r < n; ++r)
        for (int64_t c = 0; c < n; ++c) inv[r * n + c] = a[r * w + n + c];
    return true;
}

template <typename T> T *vec(void *p) { return static_cast<T *>(p); }

// Chebyshev semi-iteration of `degree` on level l for A x = b over [lo, hi],
// from x_in (null: zero) into x_out; x_out may equal x_in only for degree 1.
// One kernel per step: step k reads (x_{k-1}, d_{k-1}) and writes
// (x_k, d_k) to the other buffers of a ping-pong pair; the last step writes
// x_m = x_{m-1} + d_{m-1} straight into x_out.
// the Schur preconditioner's output of the V-cycle (see March::z4)
template <typename T> struct SchurOut {
    T *z4;
    const T *v4;
    const uint8_t *m4;
    T inv_sigma;
};

template <typename T>
fsi_status chebyshev(fsi_mesh *m, int l, int degree, double lo, double hi, const T *b,
                     const T *x_in, T *x_out, const SchurOut<T> *so = nullptr)
{
    PressureMG &P = *m->pmg;
    PmgLevel &L = P.lev[l];
    const LevelArgs<T> A = level_args<T>(P, l);
    cudaStream_t s = m->stream;
    const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo), s1 = theta / delta;
    T *dbuf[2] = {vec<T>(L.d0), vec<T>(L.d1)}, *xbuf[2] = {vec<T>(L.xa), vec<T>(L.r)};
    // first direction (degree 1: x_out = x + d0 directly)
    if (x_in) {
        March<T> M{};
        M.x = x_in;
        M.b = b;
        M.inv_theta = (T)(1.0 / theta);
        M.d_next = degree == 1 ? nullptr : dbuf[0];
        M.x_final = degree == 1 ? x_out : nullptr;
        FSI_TRY((march<T, kMarchCheb0>(P, l, s, M)));
    } else if (degree == 1) {
        cheb0_kernel<T><<<grid3_strided(L), kRowBlock, 0, s>>>(A, b, (T)(1.0 / theta), nullptr,
                                                               x_out);
        FSI_TRY(check_launch("pressure smoother"));
    }
    if (degree == 1) return FSI_OK;
    // from x = 0 the first step forms d0 = b / (theta D) itself (no d0 pass)
    const T *xc = x_in;
    const T *dc = x_in ? dbuf[0] : nullptr;
    double rho = 1.0 / s1;
    for (int it = 1; it < degree; ++it) {
        const double rho_new = 1.0 / (2.0 * s1 - rho);
        const T c1 = (T)(rho_new * rho), c2 = (T)(2.0 * rho_new / delta);
        const bool last = it == degree - 1;
        T *xn = xbuf[it & 1], *dn = dbuf[it & 1];
        March<T> M{};
        M.x = xc;
        M.d = dc;
        M.b = b;
        M.c1 = c1;
        M.c2 = c2;
        M.inv_theta = (T)(1.0 / theta);
        M.x_next = last ? nullptr : xn;
        M.d_next = last ? nullptr : dn;
        M.x_final = last ? x_out : nullptr;
        if (last && so) {
            M.z4 = so->z4;
            M.v4 = so->v4;
            M.m4 = so->m4;
            M.inv_sigma = so->inv_sigma;
        }
        FSI_TRY((march<T, kMarchStep>(P, l, s, M)));
        xc = xn;
        dc = dn;
        rho = rho_new;
    }
    return check_launch("pressure smoother");
}

// ---------------------------------------------------------------- coarse levels
// The V-cycle's FP32 levels of at most kCoarseNodes nodes, down to and with the
// dense coarsest solve, as one cluster of CTAs: every vector of those levels lives
// in shared memory and passes are separated by barriers.  As launches of their own
// these passes are 6 per level of 3 to 5 us each, nearly all latency: at 32^3 a
// mixed step with 56 V-cycles took 12.2 ms with them, and about 46 us a cycle less with this
// kernel (24.6 us).  In FP64 (two
// operations per SM and clock) they stay spread over the chip, pass by pass.
//
// A pass is bound by the length of one thread's instruction stream (a kernel of
// this form with a marching stencil, a thread per column piece, took 41 us), so a
// thread has one node and its weights stay in registers from pass to pass:
// the operator is symmetric along every axis, so a row is 8 weights times sums of
// neighbours (none, along x, along y, both; in the plane and off it).  Vectors
// that a stencil reads are padded by zeros, and they are zero at eliminated nodes,
// whose rows are their diagonal alone.
//
// The first (largest) level is split into slabs of planes, one per CTA; a CTA has
// the whole level's indexes, but only its slab and the plane on either side hold
// values: what the neighbours read is stored into their shared memory as well.
// Rank 0 alone does the levels below: at most an eighth of the work, and a pass over
// the cluster costs a cluster barrier.
constexpr int kCoarseNodes = 4913;  // 17^3
constexpr int kCoarseThreads = 1024;
constexpr int kCoarseCtas = 8;
constexpr int kCoarseSmemMax = 224 * 1024;
constexpr int kCoarseSplit = 1000;  // nodes from which the first level is split
constexpr int kCoarseMaxLevels = 8;
struct CoarseLevel {
    LevelArgs<float> A;
    int n;
    float inv_theta, c1, c2;  // Chebyshev degree 2 over [hi/4, hi]
    int sy, sz;               // strides of the padded vectors
    int b, e, v, t;           // places in shared memory: b, e [n], v, t padded
};
struct CoarseCycle {
    int nlev;  // smoothed levels; the dense level follows
    CoarseLevel lev[kCoarseMaxLevels];
    LevelArgs<float> Ad;  // the dense level
    int nd, off_d;        // its nodes and the place of its b, x
    int off_inv;          // of the dense inverse in shared memory; 0: left in global
    int pads0, pads1;     // the padded vectors' range
    const float *inv;
    const float *b;  // right-hand side of the first level
    float *x;        // result
};

// One node of a level and its row of the operator: A v = sum_c wA[c] S_c + wB[c] Z_c,
// S_c the neighbours' sum of class c (0: the node, 1: along x, 2: along y, 3: both) in
// the node's plane, Z_c in the two planes beside it
struct CoarseNode {
    int q;  // which (-1: none yet)
    int k, p;
    float wA[4], wB[4], iD;
};

__device__ __forceinline__ void coarse_node(const CoarseLevel &L, int q, CoarseNode &N)
{
    const LevelArgs<float> &A = L.A;
    const Axis<float> &ax = A.a[0], &ay = A.a[1], &az = A.a[2];
    const int row = q / A.NX1, i = q - row * A.NX1, k = row / A.NY1, j = row - k * A.NY1;
    N.q = q;
    N.k = k;
    N.p = (i + 1) + L.sy * (j + 1) + L.sz * (k + 1);
    const float mx = md_of(ax, i), kx = kd_of(ax, i), my = md_of(ay, j), mz = md_of(az, k), kz = kd_of(az, k);
    const float ky = kd_of(ay, j) + A.kappa * my, kyo = ay.k_off + A.kappa * ay.m_off;
    const float P[4] = {kx * my + mx * ky, ax.k_off * my + ax.m_off * ky, kx * ay.m_off + mx * kyo,
                        ax.k_off * ay.m_off + ax.m_off * kyo};
    const float Q[4] = {mx * my, ax.m_off * my, mx * ay.m_off, ax.m_off * ay.m_off};
    const bool el = eliminated(A, i, j, k);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        N.wA[c] = el && c ? 0.f : P[c] * mz + Q[c] * kz;
        N.wB[c] = el ? 0.f : P[c] * az.m_off + Q[c] * az.k_off;
    }
    N.iD = 1.f / N.wA[0];
}

// f(node) for this thread's nodes of the planes [z0, z1); N is kept from pass to
// pass (a thread has one node unless a plane has more than kCoarseThreads)
template <typename F>
__device__ __forceinline__ void coarse_nodes(const CoarseLevel &L, int z0, int z1, CoarseNode &N, F f)
{
    const int plane = L.A.NX1 * L.A.NY1;
    for (int q = z0 * plane + threadIdx.x; q < z1 * plane; q += kCoarseThreads) {
        if (q != N.q) coarse_node(L, q, N);
        f(N);
    }
}

__device__ __forceinline__ float coarse_row(const CoarseLevel &L, const CoarseNode &N, const float *v)
{
    float S[3][3], Z[3][3];  // [y][x]
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float *r = v + N.p + (d - 1) * L.sy;
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            S[d][x] = r[x - 1];
            Z[d][x] = r[x - 1 - L.sz] + r[x - 1 + L.sz];
        }
    }
    const float a0 = N.wA[0] * S[1][1] + N.wB[0] * Z[1][1];
    const float a1 = N.wA[1] * (S[1][0] + S[1][2]) + N.wB[1] * (Z[1][0] + Z[1][2]);
    const float a2 = N.wA[2] * (S[0][1] + S[2][1]) + N.wB[2] * (Z[0][1] + Z[2][1]);
    const float a3 = N.wA[3] * ((S[0][0] + S[0][2]) + (S[2][0] + S[2][2])) +
                     N.wB[3] * ((Z[0][0] + Z[0][2]) + (Z[2][0] + Z[2][2]));
    return (a0 + a1) + (a2 + a3);
}

__global__ void __launch_bounds__(kCoarseThreads, 1) coarse_cycle_kernel(const __grid_constant__ CoarseCycle C)
{
    extern __shared__ __align__(16) float cs[];
    cg::cluster_group cl = cg::this_cluster();
    const int tid = threadIdx.x;
    const int nr = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    // this CTA's planes [s0, s1) of the first level
    const int NZ = C.lev[0].A.NZ1, zl = (NZ + nr - 1) / nr;
    const int s0 = min(rank * zl, NZ), s1 = min(s0 + zl, NZ);
    auto sync = [&](bool split) {
        if (split && nr > 1) cl.sync();
        else __syncthreads();
    };
    // a value of plane k, with split also into the neighbours' halo planes
    auto put = [&](bool split, float *at, int k, float val) {
        *at = val;
        if (split && nr > 1) {
            if (k == s0 && s0 > 0) *cl.map_shared_rank(at, rank - 1) = val;
            if (k == s1 - 1 && s1 < NZ) *cl.map_shared_rank(at, rank + 1) = val;
        }
    };
    for (int q = C.pads0 + tid; q < C.pads1; q += kCoarseThreads) cs[q] = 0.f;
    CoarseNode N;
    N.q = -1;
    coarse_nodes(C.lev[0], s0, s1, N, [&](const CoarseNode &) {});  // the weights
    const float *gb = C.b, *ginv = C.inv;
    float *gx = C.x;
    chain_trigger();
    chain_wait(gb, ginv, gx);
    // the dense inverse on its way (see off_inv)
    if (rank == 0 && C.off_inv)
        for (int q = tid; q < C.nd * C.nd; q += kCoarseThreads)
            __pipeline_memcpy_async(cs + C.off_inv + q, ginv + q, 4);
    __pipeline_commit();
    coarse_nodes(C.lev[0], s0, s1, N, [&](const CoarseNode &N) { cs[C.lev[0].b + N.q] = __ldcg(gb + N.q); });
    sync(true);
    // down: pre-smoothing from zero into t, residual into v, its restriction
    for (int l = 0; l < C.nlev; ++l) {
        const bool split = l == 0;
        if (!split && rank > 0) break;
        const CoarseLevel &L = C.lev[l];
        const int z0 = l ? 0 : s0, z1 = l ? L.A.NZ1 : s1;
        const float *b = cs + L.b;
        float *v = cs + L.v, *t = cs + L.t;
        if (!split) N.q = -1;
        coarse_nodes(L, z0, z1, N, [&](const CoarseNode &N) {  // d0
            put(split, v + N.p, N.k, L.inv_theta * b[N.q] * N.iD);
        });
        sync(split);
        coarse_nodes(L, z0, z1, N, [&](const CoarseNode &N) {
            const float d0 = v[N.p];
            put(split, t + N.p, N.k, d0 + (L.c1 * d0 + L.c2 * ((b[N.q] - coarse_row(L, N, v)) * N.iD)));
        });
        sync(split);
        coarse_nodes(L, z0, z1, N, [&](const CoarseNode &N) {
            put(split, v + N.p, N.k, b[N.q] - coarse_row(L, N, t));
        });
        sync(split);
        // restriction of the coarse planes whose fine plane is in the slab, to rank 0
        const bool last = l + 1 == C.nlev;
        const LevelArgs<float> &B = last ? C.Ad : C.lev[l + 1].A;
        float *bc = cs + (last ? C.off_d : C.lev[l + 1].b);
        if (rank > 0) bc = cl.map_shared_rank(bc, 0);
        const int cplane = B.NX1 * B.NY1, K0 = (z0 + 1) / 2, K1 = z0 < z1 ? (z1 - 1) / 2 + 1 : 0;
        for (int q = K0 * cplane + tid; q < K1 * cplane; q += kCoarseThreads) {
            const int row = q / B.NX1, I = q - row * B.NX1, K = row / B.NY1, J = row - K * B.NY1;
            const float *c = v + (2 * I + 1) + L.sy * (2 * J + 1) + L.sz * (2 * K + 1);
            float acc[3];
#pragma unroll
            for (int dk = -1; dk <= 1; ++dk) {
                float r[3];
#pragma unroll
                for (int dj = -1; dj <= 1; ++dj) {
                    const float *rw = c + dk * L.sz + dj * L.sy;
                    r[dj + 1] = rw[0] + 0.5f * (rw[-1] + rw[1]);
                }
                acc[dk + 1] = r[1] + 0.5f * (r[0] + r[2]);
            }
            bc[q] = eliminated(B, I, J, K) ? 0.f : acc[1] + 0.5f * (acc[0] + acc[2]);
        }
        sync(split);
    }
    // the dense inverse: eight threads per row
    if (rank == 0) {
        const float *b = cs + C.off_d;
        float *x = cs + C.off_d + C.nd;
        const float *inv = C.off_inv ? cs + C.off_inv : ginv;
        __pipeline_wait_prior(0);
        __syncthreads();
        for (int r0 = 0; r0 < C.nd; r0 += kCoarseThreads / 8) {
            const int row = r0 + (tid >> 3);
            float s0 = 0.f, s1 = 0.f;
            if (row < C.nd) {
                const float *m = inv + row * C.nd;
                int c = tid & 7;
                for (; c + 8 < C.nd; c += 16) {
                    s0 += m[c] * b[c];
                    s1 += m[c + 8] * b[c + 8];
                }
                if (c < C.nd) s0 += m[c] * b[c];
            }
            s0 += s1;
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
            if (row < C.nd && (tid & 7) == 0) x[row] = s0;
        }
        __syncthreads();
    }
    // up: prolongation into t, post-smoothing from t
    for (int l = C.nlev - 1; l >= 0; --l) {
        const bool split = l == 0;
        if (!split && rank > 0) continue;
        const CoarseLevel &L = C.lev[l];
        const int z0 = l ? 0 : s0, z1 = l ? L.A.NZ1 : s1;
        const float *b = cs + L.b;
        float *e = cs + L.e, *v = cs + L.v, *t = cs + L.t;
        // the level below leaves its result in its t (the dense level after its b)
        const bool last = l + 1 == C.nlev;
        const LevelArgs<float> &B = last ? C.Ad : C.lev[l + 1].A;
        const int cy = last ? B.NX1 : C.lev[l + 1].sy, cz = last ? B.NX1 * B.NY1 : C.lev[l + 1].sz;
        const float *xc = cs + (last ? C.off_d + C.nd : C.lev[l + 1].t + 1 + cy + cz);
        if (split && nr > 1) {
            cl.sync();  // rank 0's result is there
            if (rank > 0) xc = cl.map_shared_rank(xc, 0);
        }
        if (!split || (rank == 0 && C.nlev > 1)) N.q = -1;
        coarse_nodes(L, z0, z1, N, [&](const CoarseNode &N) {
            // trilinear: the mean of the two (or, on a coarse line, twice the one) along each axis
            const int row = N.q / L.A.NX1, i = N.q - row * L.A.NX1, j = row - N.k * L.A.NY1;
            const float *r = xc + (i >> 1) + cy * (j >> 1) + cz * (N.k >> 1);
            const int dx = i & 1, dy = (j & 1) ? cy : 0, dz = (N.k & 1) ? cz : 0;
            const float s = ((r[0] + r[dx]) + (r[dy] + r[dx + dy])) +
                            ((r[dz] + r[dx + dz]) + (r[dy + dz] + r[dx + dy + dz]));
            put(split, t + N.p, N.k, t[N.p] + 0.125f * s);
        });
        sync(split);
        // the first direction d0 from x = t; then v = t + d0, d0 kept in e
        coarse_nodes(L, z0, z1, N, [&](const CoarseNode &N) {
            const float d0 = L.inv_theta * (b[N.q] - coarse_row(L, N, t)) * N.iD;
            e[N.q] = d0;
            put(split, v + N.p, N.k, t[N.p] + d0);
        });
        sync(split);
        coarse_nodes(L, z0, z1, N, [&](const CoarseNode &N) {
            const float y = v[N.p] + (L.c1 * e[N.q] + L.c2 * ((b[N.q] - coarse_row(L, N, v)) * N.iD));
            if (l == 0) gx[N.q] = y;
            else t[N.p] = y;
        });
        __syncthreads();
    }
}

// The levels from l0 on as coarse_cycle_kernel's arguments; the shared memory they
// need in bytes
int coarse_plan(const PressureMG &P, int l0, CoarseCycle &C)
{
    C.nlev = P.nlev - 1 - l0;
    int off = 0;
    for (int l = 0; l < C.nlev; ++l) {
        const PmgLevel &L = P.lev[l0 + l];
        CoarseLevel &D = C.lev[l];
        const double hi = L.hi, lo = hi / 4.0, theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo),
                     s1 = theta / delta, rho = 1.0 / s1, rho_new = 1.0 / (2.0 * s1 - rho);
        D.A = level_args<float>(P, l0 + l);
        D.n = (int)L.n;
        D.inv_theta = (float)(1.0 / theta);
        D.c1 = (float)(rho_new * rho);
        D.c2 = (float)(2.0 * rho_new / delta);
        D.sy = D.A.NX1 + 2;
        D.sz = D.sy * (D.A.NY1 + 2);
        const int padded = D.sz * (D.A.NZ1 + 2);
        D.v = off;
        D.t = off + padded;
        off += 2 * padded;
    }
    C.pads0 = 0;
    C.pads1 = off;
    for (int l = 0; l < C.nlev; ++l) {
        C.lev[l].b = off;
        C.lev[l].e = off + C.lev[l].n;
        off += 2 * C.lev[l].n;
    }
    C.Ad = level_args<float>(P, P.nlev - 1);
    C.nd = (int)P.nc;
    C.off_d = off;
    off += 2 * C.nd;
    C.inv = P.inv32;
    if (C.nd <= 181 && (off + C.nd * C.nd) * (int)sizeof(float) <= kCoarseSmemMax) {
        C.off_inv = off;
        off += C.nd * C.nd;
    }
    return off * (int)sizeof(float);
}

// The first level of the FP32 V-cycle that coarse_cycle_kernel takes, or -1: a
// level below the finest, small enough, with the levels after it fitting the
// kernel and a dense coarsest solve
int coarse_first(const PressureMG &P)
{
    if (!P.direct) return -1;
    for (int l = 1; l < P.nlev - 1; ++l) {
        if (P.lev[l].n > kCoarseNodes || P.nlev - 1 - l > kCoarseMaxLevels) continue;
        CoarseCycle C{};
        if (coarse_plan(P, l, C) <= kCoarseSmemMax) return l;
    }
    return -1;
}

fsi_status coarse_cycle(fsi_mesh *m, int l0, const float *b, float *x)
{
    CoarseCycle C{};
    const int bytes = coarse_plan(*m->pmg, l0, C);
    C.b = b;
    C.x = x;
    FSI_TRY(set_smem_limit((const void *)coarse_cycle_kernel, kCoarseSmemMax));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = cfg.blockDim = dim3(1, 1, 1);
    cfg.gridDim.x = C.lev[0].n >= kCoarseSplit ? kCoarseCtas : 1;
    cfg.blockDim.x = kCoarseThreads;
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = m->stream;
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cfg.gridDim.x;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see launch_chain
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    FSI_CUDA(cudaLaunchKernelEx(&cfg, coarse_cycle_kernel, C), "pressure coarse levels");
    return check_launch("pressure coarse levels");
}

template <typename T> fsi_status coarse_solve(fsi_mesh *m, const T *b, T *x)
{
    PressureMG &P = *m->pmg;
    const int l = P.nlev - 1;
    if (P.direct) {
        const T *inv = std::is_same<T, double>::value ? (const T *)P.inv64 : (const T *)P.inv32;
        const int warps_per_block = 8;
        const int blocks = (int)std::min<int64_t>((P.nc + warps_per_block - 1) / warps_per_block, sm_count() * 8);
        dense_apply_kernel<T><<<blocks, 32 * warps_per_block, 0, m->stream>>>(P.nc, inv, b, x);
        return check_launch("pressure coarse solve");
    }
    return chebyshev<T>(m, l, kPmgCoarseDegree, P.lev[l].hi / 30.0, P.lev[l].hi, b, nullptr, x);
}

// x = V_l(b): pre-smoothing from zero into t, residual, restriction, the
// coarse cycle, prolongation into t, post-smoothing from t into x
// (so: level l's result goes to the Schur preconditioner's output instead of
// x; not on the coarsest level)
template <typename T>
fsi_status vcycle_level(fsi_mesh *m, int l, const T *b, T *x, const SchurOut<T> *so = nullptr)
{
    PressureMG &P = *m->pmg;
    if (l == P.nlev - 1) return coarse_solve<T>(m, b, x);
    if constexpr (std::is_same<T, float>::value)
        if (l == coarse_first(P)) return coarse_cycle(m, l, b, x);
    PmgLevel &L = P.lev[l], &Lc = P.lev[l + 1];
    const double hi = L.hi;
    T *t = vec<T>(L.t);
    FSI_TRY(chebyshev<T>(m, l, kPmgNu, hi / 4.0, hi, b, (const T *)nullptr, t));
    const LevelArgs<T> A = level_args<T>(P, l), Ac = level_args<T>(P, l + 1);
    int kz = 1;
    FSI_TRY(level_apply<T>(P, l, m->stream, t, b, vec<T>(L.r)));
    const dim3 gr = transfer_grid(Lc, Lc, kz);
    launch_chain(restrict_kernel<T>, gr, kRowBlock, 0, m->stream, A, Ac, kz, vec<T>(L.r), vec<T>(Lc.b));
    FSI_TRY(check_launch("pressure restrict"));
    FSI_TRY(vcycle_level<T>(m, l + 1, vec<T>(Lc.b), vec<T>(Lc.x)));
    const dim3 gp = transfer_grid(L, Lc, kz);
    launch_chain(prolong_kernel<T>, gp, kRowBlock, 0, m->stream, A, Ac, kz, vec<T>(Lc.x), t);
    FSI_TRY(check_launch("pressure prolong"));
    return chebyshev<T>(m, l, kPmgNu, hi / 4.0, hi, b, t, x, so);
}

fsi_status check_prec(fsi_prec p)
{
    if (p != FSI_F64 && p != FSI_F32) return set_error(FSI_ERR_ARG, "pressure operator: precision must be FSI_F64 or FSI_F32");
    return FSI_OK;
}

fsi_status check_level(fsi_mesh *m, int level, bool need_coarser)
{
    if (level < 0 || level >= m->pmg->nlev || (need_coarser && level + 1 >= m->pmg->nlev))
        return set_error(FSI_ERR_ARG, "pressure operator: level %d out of range", level);
    return FSI_OK;
}

}  // namespace

void destroy_pmg(fsi_mesh *m)
{
    if (!m->pmg) return;
    PressureMG &P = *m->pmg;
    for (int l = 0; l < P.nlev; ++l) {
        void *bufs[] = {P.lev[l].b, P.lev[l].x, P.lev[l].r, P.lev[l].t,
                        P.lev[l].d0, P.lev[l].d1, P.lev[l].xa};
        for (void *q : bufs) cudaFree(q);
    }
    cudaFree(P.inv64);
    cudaFree(P.inv32);
    delete m->pmg;
    m->pmg = nullptr;
}

// dense inverse of the coarsest level for the current faces (FP64 host
// Gauss-Jordan), copied to the device in FP64 and FP32
fsi_status build_coarse_inverse(fsi_mesh *m)
{
    PressureMG &P = *m->pmg;
    const PmgLevel &C = P.lev[P.nlev - 1];
    std::vector<double> inv;
    if (!dense_inverse(C, P.kappa, P.faces, inv))
        return set_error(FSI_ERR_ARG, "pressure hierarchy: singular coarse operator");
    std::vector<float> inv32(inv.begin(), inv.end());
    FSI_CUDA(cudaMemcpy(P.inv64, inv.data(), inv.size() * sizeof(double), cudaMemcpyHostToDevice),
             "memcpy");
    FSI_CUDA(cudaMemcpy(P.inv32, inv32.data(), inv32.size() * sizeof(float),
                        cudaMemcpyHostToDevice),
             "memcpy");
    return FSI_OK;
}

fsi_status pmg_ensure(fsi_mesh *m)
{
    FSI_TRY(require_structured(m, "the pressure multigrid"));
    if (m->pmg) return FSI_OK;
    PressureMG *P = new (std::nothrow) PressureMG();
    if (!P) return set_error(FSI_ERR_OOM, "host allocation of the pressure hierarchy failed");
    m->pmg = P;
    double Lmax = 0.0;
    for (int d = 0; d < 3; ++d) Lmax = std::max(Lmax, m->grid.N[d] * m->grid.h[d]);
    const double q = 3.14159265358979323846 / (2.0 * Lmax);
    P->kappa = q * q;
    if (m->grid.N[1] + 1 > 65535 || m->grid.N[2] + 1 > 65535) {
        destroy_pmg(m);
        return set_error(FSI_ERR_ARG, "pressure hierarchy: at most 65535 nodes along y and z");
    }
    PmgLevel cur{};
    for (int d = 0; d < 3; ++d) {
        cur.N[d] = m->grid.N[d];
        cur.h[d] = m->grid.h[d];
    }
    while (true) {
        cur.n = (int64_t)(cur.N[0] + 1) * (cur.N[1] + 1) * (cur.N[2] + 1);
        cur.hi = spectrum_bound(cur.h, P->kappa);
        P->lev[P->nlev++] = cur;
        const bool even = cur.N[0] % 2 == 0 && cur.N[1] % 2 == 0 && cur.N[2] % 2 == 0;
        if (!even || cur.n <= kPmgMinCoarsen || P->nlev == kPmgMaxLevels) break;
        for (int d = 0; d < 3; ++d) {
            cur.N[d] /= 2;
            cur.h[d] *= 2.0;
        }
    }
    for (int l = 0; l < P->nlev; ++l) {
        const size_t bytes = (size_t)P->lev[l].n * sizeof(double);
        void **bufs[] = {&P->lev[l].b,  &P->lev[l].x,  &P->lev[l].r, &P->lev[l].t,
                         &P->lev[l].d0, &P->lev[l].d1, &P->lev[l].xa};
        for (void **b : bufs) {
            *b = nullptr;
            if (cudaMalloc(b, bytes) != cudaSuccess) {
                cudaGetLastError();
                destroy_pmg(m);
                return set_error(FSI_ERR_OOM, "pressure hierarchy: cudaMalloc failed");
            }
        }
    }
    const PmgLevel &C = P->lev[P->nlev - 1];
    P->nc = C.n;
    P->direct = C.n <= kPmgDirectMax;
    if (P->direct) {
        if (cudaMalloc((void **)&P->inv64, (size_t)C.n * C.n * sizeof(double)) != cudaSuccess ||
            cudaMalloc((void **)&P->inv32, (size_t)C.n * C.n * sizeof(float)) != cudaSuccess) {
            cudaGetLastError();
            destroy_pmg(m);
            return set_error(FSI_ERR_OOM, "pressure hierarchy: cudaMalloc failed");
        }
        fsi_status st = build_coarse_inverse(m);
        if (st != FSI_OK) {
            destroy_pmg(m);
            return st;
        }
    }
    return FSI_OK;
}

fsi_status pmg_set_faces(fsi_mesh *m, const int faces[6])
{
    FSI_TRY(pmg_ensure(m));
    PressureMG &P = *m->pmg;
    bool same = true;
    for (int f = 0; f < 6; ++f) same = same && (P.faces[f] != 0) == (faces[f] != 0);
    if (same) return FSI_OK;
    for (int f = 0; f < 6; ++f) P.faces[f] = faces[f] != 0;
    // the coarse inverse is in use by work already queued on the stream
    FSI_CUDA(cudaStreamSynchronize(m->stream), "sync");
    return P.direct ? build_coarse_inverse(m) : FSI_OK;
}

template <typename T> fsi_status pmg_vcycle(fsi_mesh *m, const T *b, T *x)
{
    FSI_TRY(pmg_ensure(m));
    return vcycle_level<T>(m, 0, b, x);
}
template fsi_status pmg_vcycle<double>(fsi_mesh *, const double *, double *);
template fsi_status pmg_vcycle<float>(fsi_mesh *, const float *, float *);

template <typename T>
fsi_status pmg_vcycle_schur(fsi_mesh *m, const T *b, T *z, const T *v, const uint8_t *mask,
                            T inv_sigma, bool *done)
{
    FSI_TRY(pmg_ensure(m));
    *done = false;
    PressureMG &P = *m->pmg;
    if (P.nlev < 2) return FSI_OK;
    const SchurOut<T> so{z, v, mask, inv_sigma};
    FSI_TRY(vcycle_level<T>(m, 0, b, vec<T>(P.lev[0].x), &so));
    *done = true;
    return FSI_OK;
}
template fsi_status pmg_vcycle_schur<double>(fsi_mesh *, const double *, double *, const double *,
                                             const uint8_t *, double, bool *);
template fsi_status pmg_vcycle_schur<float>(fsi_mesh *, const float *, float *, const float *,
                                            const uint8_t *, float, bool *);

// level-0 right-hand side (which = 0) and solution (which = 1) buffers, n
// entries of either precision; the Newton preconditioner gathers into them
void *pmg_fine_buffer(fsi_mesh *m, int which) { return which == 0 ? m->pmg->lev[0].b : m->pmg->lev[0].x; }

}  // namespace fsi

// ---------------------------------------------------------------- C ABI
using namespace fsi;

extern "C" {

fsi_status fsi_pressure_levels(fsi_mesh *mesh, int32_t *n_levels, int32_t *N)
{
    FSI_TRY(validate_mesh(mesh));
    if (!n_levels) return set_error(FSI_ERR_ARG, "fsi_pressure_levels: n_levels is NULL");
    if (mesh->pressure_amg)
        return set_error(FSI_ERR_ARG, "fsi_pressure_levels: the pressure block is the algebraic "
                                      "multigrid (fsi_pressure_level_sizes)");
    FSI_DEVICE(mesh->device);
    FSI_TRY(pmg_ensure(mesh));
    *n_levels = mesh->pmg->nlev;
    if (N)
        for (int l = 0; l < mesh->pmg->nlev; ++l)
            for (int d = 0; d < 3; ++d) N[3 * l + d] = mesh->pmg->lev[l].N[d];
    return FSI_OK;
}

fsi_status fsi_pressure_level_sizes(fsi_mesh *mesh, int32_t *n_levels, int64_t *n)
{
    FSI_TRY(validate_mesh(mesh));
    if (!n_levels) return set_error(FSI_ERR_ARG, "fsi_pressure_level_sizes: n_levels is NULL");
    FSI_DEVICE(mesh->device);
    if (uses_amg(mesh)) return amg_level_sizes(mesh, n_levels, n);
    FSI_TRY(pmg_ensure(mesh));
    *n_levels = mesh->pmg->nlev;
    if (n)
        for (int l = 0; l < mesh->pmg->nlev; ++l) n[l] = mesh->pmg->lev[l].n;
    return FSI_OK;
}

fsi_status fsi_pressure_set_eliminated(fsi_mesh *mesh, const uint8_t *eliminated)
{
    FSI_TRY(validate_mesh(mesh));
    if (!uses_amg(mesh))
        return set_error(FSI_ERR_ARG, "fsi_pressure_set_eliminated: the pressure block is the "
                                      "geometric multigrid (it eliminates faces: "
                                      "fsi_pressure_set_faces; or fsi_pressure_use_amg)");
    FSI_DEVICE(mesh->device);
    std::vector<uint8_t> e((size_t)mesh->n_nodes, 0);
    if (eliminated) {
        FSI_CUDA(cudaMemcpyAsync(e.data(), eliminated, e.size(), cudaMemcpyDeviceToHost,
                                 mesh->stream),
                 "memcpy");
        FSI_CUDA(cudaStreamSynchronize(mesh->stream), "sync");
        for (uint8_t &v : e) v = v != 0;
    }
    return amg_set_eliminated(mesh, e);
}

fsi_status fsi_pressure_use_amg(fsi_mesh *mesh, int32_t on)
{
    FSI_TRY(validate_mesh(mesh));
    if (mesh->tet) {
        if (!on)
            return set_error(FSI_ERR_ARG, "fsi_pressure_use_amg: a tetrahedral mesh has only the "
                                          "algebraic multigrid");
        return FSI_OK;
    }
    FSI_DEVICE(mesh->device);
    if ((on != 0) == mesh->pressure_amg) return FSI_OK;
    // the hierarchy may be in use by work already queued on the stream
    FSI_CUDA(cudaStreamSynchronize(mesh->stream), "sync");
    destroy_amg(mesh);
    mesh->pressure_amg = on != 0;
    return FSI_OK;
}

fsi_status fsi_pressure_set_faces(fsi_mesh *mesh, const int32_t *faces)
{
    FSI_TRY(validate_mesh(mesh));
    if (!faces) return set_error(FSI_ERR_ARG, "fsi_pressure_set_faces: faces is NULL");
    if (mesh->pressure_amg)
        return set_error(FSI_ERR_ARG, "fsi_pressure_set_faces: the pressure block is the "
                                      "algebraic multigrid (fsi_pressure_set_eliminated)");
    FSI_DEVICE(mesh->device);
    int f[6];
    for (int q = 0; q < 6; ++q) f[q] = faces[q] != 0;
    return pmg_set_faces(mesh, f);
}

fsi_status fsi_pressure_apply(fsi_mesh *mesh, fsi_prec prec, int32_t level, const void *x, void *y)
{
    FSI_TRY(validate_mesh(mesh));
    FSI_TRY(check_prec(prec));
    if (!x || !y) return set_error(FSI_ERR_ARG, "fsi_pressure_apply: NULL argument");
    FSI_DEVICE(mesh->device);
    if (uses_amg(mesh)) return amg_apply(mesh, prec, level, x, y);
    FSI_TRY(pmg_ensure(mesh));
    FSI_TRY(check_level(mesh, level, false));
    if (prec == FSI_F64)
        return level_apply<double>(*mesh->pmg, level, mesh->stream, (const double *)x, nullptr,
                                   (double *)y);
    return level_apply<float>(*mesh->pmg, level, mesh->stream, (const float *)x, nullptr,
                              (float *)y);
}

fsi_status fsi_pressure_restrict(fsi_mesh *mesh, fsi_prec prec, int32_t level, const void *r,
                                 void *b)
{
    FSI_TRY(validate_mesh(mesh));
    FSI_TRY(check_prec(prec));
    if (!r || !b) return set_error(FSI_ERR_ARG, "fsi_pressure_restrict: NULL argument");
    FSI_DEVICE(mesh->device);
    if (uses_amg(mesh)) return amg_restrict(mesh, prec, level, r, b);
    FSI_TRY(pmg_ensure(mesh));
    FSI_TRY(check_level(mesh, level, true));
    PressureMG &P = *mesh->pmg;
    int kz = 1;
    const dim3 g = transfer_grid(P.lev[level + 1], P.lev[level + 1], kz);
    if (prec == FSI_F64)
        restrict_kernel<double><<<g, kRowBlock, 0, mesh->stream>>>(
            level_args<double>(P, level), level_args<double>(P, level + 1), kz, (const double *)r,
            (double *)b);
    else
        restrict_kernel<float><<<g, kRowBlock, 0, mesh->stream>>>(
            level_args<float>(P, level), level_args<float>(P, level + 1), kz, (const float *)r,
            (float *)b);
    return check_launch("pressure restrict");
}

fsi_status fsi_pressure_prolong_add(fsi_mesh *mesh, fsi_prec prec, int32_t level,
                                    const void *xc, void *x)
{
    FSI_TRY(validate_mesh(mesh));
    FSI_TRY(check_prec(prec));
    if (!xc || !x) return set_error(FSI_ERR_ARG, "fsi_pressure_prolong_add: NULL argument");
    FSI_DEVICE(mesh->device);
    if (uses_amg(mesh)) return amg_prolong_add(mesh, prec, level, xc, x);
    FSI_TRY(pmg_ensure(mesh));
    FSI_TRY(check_level(mesh, level, true));
    PressureMG &P = *mesh->pmg;
    int kz = 1;
    const dim3 g = transfer_grid(P.lev[level], P.lev[level + 1], kz);
    if (prec == FSI_F64)
        prolong_kernel<double><<<g, kRowBlock, 0, mesh->stream>>>(
            level_args<double>(P, level), level_args<double>(P, level + 1), kz, (const double *)xc,
            (double *)x);
    else
        prolong_kernel<float><<<g, kRowBlock, 0, mesh->stream>>>(
            level_args<float>(P, level), level_args<float>(P, level + 1), kz, (const float *)xc,
            (float *)x);
    return check_launch("pressure prolong");
}

fsi_status fsi_pressure_smooth(fsi_mesh *mesh, fsi_prec prec, int32_t level, int32_t degree,
                               const void *b, void *x, int32_t from_zero)
{
    FSI_TRY(validate_mesh(mesh));
    FSI_TRY(check_prec(prec));
    if (!b || !x) return set_error(FSI_ERR_ARG, "fsi_pressure_smooth: NULL argument");
    if (degree < 1 || degree > 64) return set_error(FSI_ERR_ARG, "fsi_pressure_smooth: degree 1..64");
    FSI_DEVICE(mesh->device);
    if (uses_amg(mesh)) return amg_smooth(mesh, prec, level, degree, b, x, from_zero);
    FSI_TRY(pmg_ensure(mesh));
    FSI_TRY(check_level(mesh, level, false));
    const double hi = mesh->pmg->lev[level].hi;
    const int64_t n = mesh->pmg->lev[level].n;
    // from a given x: the iteration reads x while it writes the result, so
    // it starts from a copy in the level's t buffer
    if (prec == FSI_F64) {
        const double *xin = nullptr;
        if (!from_zero) {
            copy_kernel<double><<<grid_for(n), 256, 0, mesh->stream>>>(
                n, (const double *)x, (double *)mesh->pmg->lev[level].t);
            xin = (const double *)mesh->pmg->lev[level].t;
        }
        return chebyshev<double>(mesh, level, degree, hi / 4.0, hi, (const double *)b, xin,
                                 (double *)x);
    }
    const float *xin = nullptr;
    if (!from_zero) {
        copy_kernel<float><<<grid_for(n), 256, 0, mesh->stream>>>(
            n, (const float *)x, (float *)mesh->pmg->lev[level].t);
        xin = (const float *)mesh->pmg->lev[level].t;
    }
    return chebyshev<float>(mesh, level, degree, hi / 4.0, hi, (const float *)b, xin, (float *)x);
}

fsi_status fsi_pressure_vcycle(fsi_mesh *mesh, fsi_prec prec, const void *b, void *x)
{
    FSI_TRY(validate_mesh(mesh));
    FSI_TRY(check_prec(prec));
    if (!b || !x) return set_error(FSI_ERR_ARG, "fsi_pressure_vcycle: NULL argument");
    if (b == x) return set_error(FSI_ERR_ARG, "fsi_pressure_vcycle: b and x must not alias");
    FSI_DEVICE(mesh->device);
    if (uses_amg(mesh)) {
        if (prec == FSI_F64) return amg_vcycle<double>(mesh, (const double *)b, (double *)x);
        return amg_vcycle<float>(mesh, (const float *)b, (float *)x);
    }
    if (prec == FSI_F64) return pmg_vcycle<double>(mesh, (const double *)b, (double *)x);
    return pmg_vcycle<float>(mesh, (const float *)b, (float *)x);
}

}  // extern "C"
