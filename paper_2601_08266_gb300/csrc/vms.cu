// vms.cu -- matrix-free VMS residual and Jacobian-vector product on the
// uniform Q1-Q1 hex grid (Sec. 2.1 / 2.4 of the paper; form of Bazilevs et
// al. 2007).
//
// Layout of the work:
//   * One CTA per brick of bx*by columns of bz elements, four lanes per column.
//     A lane is first a node of the column's current plane, then the two Gauss
//     points above it.  On the uniform grid the Q1 basis is a tensor product of
//     1D linear functions: the x and y stages of the evaluation are butterflies
//     over two lane bits, once per node plane; the z stage stays in the lane; the
//     test-function projection is the transposed sequence, with the upper plane's
//     part carried to the next element (brick_body in vms_device.cuh).
//   * Contributions go to shared memory per column and plane; after the brick is
//     done every node sums its (<= 4) columns' contributions in a fixed order (no
//     atomics) and is written out, or, on a face between bricks, kept in the
//     brick's node block.
//   * A second kernel sums, for every node that several bricks share, the blocks
//     that contain it in a fixed brick order.  The result is deterministic
//     (bitwise reproducible) and atomic-free.
#include <algorithm>
#include <vector>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "fsi_internal.cuh"

#include "vms_device.cuh"

namespace fsi {
namespace {

using namespace vmsd;

// CTAs of 128 threads per SM that the registers are held to.  FP32: 4 (128
// registers; 3 or 5 were within 1 %).  FP64: 2, since 8 warps keep its pipe busy
// (85 % active) and no value has to be spilled.  Double-float: 3 (168 registers),
// both operators at once 2 (254; at 3 it spills and takes 420 instead of 406 us at
// 64^3).  On mapped grids FP32 spills a little at 4 and is still faster than at 3, but
// for both operators at once: 3 (at 4 it spills 628 bytes; 128^3 812 -> 555 us).
template <typename T, bool FUSED, bool MAPPED>
constexpr int kBrickCtas = sizeof(T) == 4 ? (FUSED && MAPPED ? 3 : 4)
                                          : (std::is_same<T, double>::value || FUSED ? 2 : 3);

template <typename T, bool JAC, bool MAPPED, bool FUSED = false>
__global__ void __launch_bounds__(kBrickThreads, (kBrickCtas<T, FUSED, MAPPED>)) vms_brick_kernel(const VmsArgs<T> P)
{
    if (P.nbx * P.nby * P.nbz > 1) chain_trigger();  // the gather follows; else any kernel
    extern __shared__ __align__(32) unsigned char smem_raw[];
    brick_body<T, JAC, MAPPED, FUSED>(P, blockIdx.x, smem_raw);
}

// Geometry table of a mapped grid: 8 lanes per element (lane = node, then
// Gauss point), the same butterfly as the VMS kernels.  The loop bound is
// uniform over the block, so every lane reaches every shuffle.
template <typename T>
__global__ void __launch_bounds__(256) mapped_geo_kernel(const VmsArgs<T> P,
                                                         typename GeoStore<T>::type *tab)
{
    const int g = threadIdx.x & 7;
    const int gx = g & 1, gy = (g >> 1) & 1, gz = (g >> 2) & 1;
    const T sx = gx ? T(0.5f) : T(-0.5f), sy = gy ? T(0.5f) : T(-0.5f),
            sz = gz ? T(0.5f) : T(-0.5f);
    const int64_t E = (int64_t)P.Nx * P.Ny * P.Nz;
    const int64_t NX1 = P.Nx + 1, NXY1 = NX1 * (P.Ny + 1);
    const int64_t per_block = blockDim.x >> 3, stride = (int64_t)gridDim.x * per_block;
    for (int64_t base = blockIdx.x * per_block; base < E; base += stride) {
        const int64_t e = base + (threadIdx.x >> 3);
        const bool valid = e < E;
        const int64_t ex = valid ? e % P.Nx : 0, ey = valid ? (e / P.Nx) % P.Ny : 0,
                      ez = valid ? e / ((int64_t)P.Nx * P.Ny) : 0;
        const int64_t node = (ex + gx) + NX1 * (ey + gy) + NXY1 * (ez + gz);
        const vec4<T> xc = valid ? load_c<T>(P.Xc + node)
                                 : vec4<T>{gx ? T(1) : T(0), gy ? T(1) : T(0), gz ? T(1) : T(0), T(0)};
        T out[kMapGeo];
        mapped_geometry<false>(xc, sx, sy, sz, out);
        if (valid)
#pragma unroll
            for (int k = 0; k < kMapGeo; ++k) tab[e * (kMapGeo * 8) + 8 * k + g] = geo_st(out[k]);
    }
}

// index of the compute type in fsi_mesh::brick (its fsi_prec)
template <typename T> constexpr int prec_slot()
{
    return std::is_same<T, double>::value ? FSI_F64
                                          : (std::is_same<T, float>::value ? FSI_F32 : FSI_DF64);
}

template <typename T> constexpr int geo_slot()
{
    return std::is_same<T, double>::value ? 0 : (std::is_same<T, float>::value ? 1 : 2);
}

// the geometry table of compute type T for the current coordinates, built on
// first use (it allocates: not inside a stream capture)
template <typename T> fsi_status ensure_map_geo(fsi_mesh *m, const VmsArgs<T> &P)
{
    void *&tab = m->map_geo[geo_slot<T>()];
    if (tab) return FSI_OK;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    FSI_CUDA(cudaStreamIsCapturing(m->stream, &cap), "cudaStreamIsCapturing");
    if (cap != cudaStreamCaptureStatusNone)
        return set_error(FSI_ERR_ARG, "mapped-grid geometry table: first use of this compute "
                                      "type inside a stream capture");
    const size_t bytes = (size_t)m->n_elems * kMapGeo * 8 * sizeof(typename GeoStore<T>::type);
    if (cudaMalloc(&tab, bytes) != cudaSuccess) {
        cudaGetLastError();
        tab = nullptr;
        return set_error(FSI_ERR_OOM, "mapped-grid geometry table: cudaMalloc of %zu bytes failed",
                         bytes);
    }
    int64_t blocks = (m->n_elems + 31) / 32;
    if (blocks > sm_count() * 8) blocks = sm_count() * 8;
    mapped_geo_kernel<T><<<(int)blocks, 256, 0, m->stream>>>(P, (typename GeoStore<T>::type *)tab);
    return check_launch("mapped geometry kernel");
}

template <typename T, bool FUSED = false>
__global__ void __launch_bounds__(256) vms_gather_kernel(const VmsArgs<T> P, int n)
{
    const int q = blockIdx.x * 256 + threadIdx.x;
    VmsArgs<T> Q = P;
    chain_wait(Q.blocks, Q.blocks2, Q.out, Q.out2);
    chain_trigger();
    if (q < n) gather_shared<T, FUSED>(Q, q);
}

// FUSED: the residual (R) and the Jacobian apply (out) at the same state in
// one pass; the brick schedule is op 2's, the shared memory and the node-block
// scratch hold both operators' contributions
template <typename T, bool JAC, bool MAPPED, bool FUSED = false>
fsi_status launch_geo(fsi_mesh *m, const void *U, const void *A, const void *f, const void *x,
                      void *out, void *R = nullptr)
{
    using S = typename StorageOf<T>::type;
    const Brick b = fit_brick(m->brick[FUSED ? 2 : (JAC ? 1 : 0)][prec_slot<T>()],
                              (int)sizeof(T), JAC, FUSED);
    FSI_TRY(ensure_vms_scratch(m, b, (FUSED ? 2 : 1) * sizeof(T)));
    VmsArgs<T> P = make_args<T>(m, b, U, A, f, x, out);
    if constexpr (MAPPED) {
        FSI_TRY(ensure_map_geo<T>(m, P));
        P.geo = (const typename GeoStore<T>::type *)m->map_geo[geo_slot<T>()];
    }
    const int nbricks = P.nbx * P.nby * P.nbz;
    if constexpr (FUSED) {
        P.blocks2 = P.blocks + (size_t)nbricks * (b.bx + 1) * (b.by + 1) * (b.bz + 1);
        P.out2 = (vec4<S> *)R;
    }
    const size_t smem = brick_smem(b.bx, b.by, b.bz, b.threads, (int)sizeof(T), JAC, FUSED);
    void (*kernel)(const VmsArgs<T>) = vms_brick_kernel<T, JAC, MAPPED, FUSED>;
    FSI_TRY(set_smem_limit((const void *)kernel, kBrickSmemMax));
    kernel<<<nbricks, b.threads, smem, m->stream>>>(P);
    FSI_TRY(check_launch("vms brick kernel"));
    const int64_t shared = shared_nodes(P);
    if (shared == 0) return FSI_OK;
    launch_chain(vms_gather_kernel<T, FUSED>, (int)((shared + 255) / 256), 256, 0, m->stream, P, (int)shared);
    return check_launch("vms gather kernel");
}

// the mapped-grid kernels take the geometry of every Gauss point from a table
// built from the node coordinates (set by fsi_mesh_set_coordinates)
template <typename T, bool JAC>
fsi_status launch(fsi_mesh *m, const void *U, const void *A, const void *f, const void *x,
                  void *out)
{
    if (m->coords64) return launch_geo<T, JAC, true>(m, U, A, f, x, out);
    return launch_geo<T, JAC, false>(m, U, A, f, x, out);
}

template <typename T>
fsi_status launch_fused(fsi_mesh *m, const void *U, const void *A, const void *f, const void *x,
                        void *R, void *Jx)
{
    if (m->coords64) return launch_geo<T, true, true, true>(m, U, A, f, x, Jx, R);
    return launch_geo<T, true, false, true>(m, U, A, f, x, Jx, R);
}

}  // namespace

// Cost of a schedule in units of one warp's share of an element layer (8
// columns): the warps' work over the SMs plus a quarter of one CTA's own
// duration as the tail, but no less than one CTA alone takes.  `alone` is how much
// longer a layer takes a warp that has an SM to itself than its share of a full
// SM: measured on GB300, 24 us against 6.4 us (FP64, both operators), about
// 10 : 1 in double-float and 16 : 1 in FP32.  A brick of bz layers spends 0.3 of a
// layer more (its lowest plane, the carried parts), and its rim nodes go through
// the node blocks.
// One sweep over the schedules for every type and operator (they share all but
// `alone` and the height): each mesh created runs it.
void default_bricks(const int32_t (*N)[3], int count, int sms, Brick (&best)[3][3])
{
    // of an 8-byte type both operators at once take lower bricks
    // (taller ones leave one CTA per SM); the Jacobian goes by the residual's rule
    constexpr int kRules = 5;
    const struct {
        double alone;
        int max_bz;
    } rule[kRules] = {{4.0, 8}, {16.0, 8}, {10.0, 8}, {4.0, 4}, {10.0, 4}};
    Brick pick[kRules];
    double cost[kRules];
    for (int q = 0; q < kRules; ++q) {
        pick[q] = {8, 4, rule[q].max_bz, 128};
        cost[q] = 1e300;
    }
    // bricks along each axis by brick size
    std::vector<double> along[3], yz(count);
    for (int d = 0; d < 3; ++d) {
        along[d].resize((size_t)16 * count);
        for (int v = 1; v <= 16; ++v)
            for (int i = 0; i < count; ++i) along[d][(size_t)(v - 1) * count + i] = (N[i][d] + v - 1) / v;
    }
    for (int bz = 8; bz >= 1; --bz)
        for (int by = 1; by <= 16; ++by) {
            for (int i = 0; i < count; ++i)
                yz[i] = along[1][(size_t)(by - 1) * count + i] * along[2][(size_t)(bz - 1) * count + i];
            for (int bx = 1; bx * by <= 32 && bx <= 16; ++bx) {
                const Brick b{bx, by, bz, (4 * bx * by + 31) / 32 * 32};
                double ctas = 0.0;
                for (int i = 0; i < count; ++i) ctas += along[0][(size_t)(bx - 1) * count + i] * yz[i];
                const double layer = bz + 0.3;
                const double rim = 1.0 + 0.06 * ((bx + 1.0) * (by + 1.0) / (bx * by) - 1.0);
                const double work = ctas / sms * (b.threads / 32) * layer * rim;
                for (int q = 0; q < kRules; ++q) {
                    if (bz > rule[q].max_bz) continue;
                    const double alone = rule[q].alone * layer,
                                 c = std::max(work + 0.25 * rule[q].alone * layer, alone) + 0.01 * work;
                    if (c < cost[q] * (1.0 - 1e-9)) {
                        cost[q] = c;
                        pick[q] = b;
                    }
                }
            }
        }
    for (int op = 0; op < 3; ++op) {
        best[op][FSI_F64] = pick[op == 2 ? 3 : 0];
        best[op][FSI_F32] = pick[1];
        best[op][FSI_DF64] = pick[op == 2 ? 4 : 2];
    }
}

namespace {

// Candidate schedules of the single-mesh autotuner beside the one the mesh has: the
// first of these, as fit_brick makes them, that differ from it and from each other, up
// to kMeshCandidates in all
constexpr int kMeshCandidates = 10;
const Brick kMeshBricks[] = {
    {8, 8, 4, 128}, {8, 4, 4, 128}, {8, 8, 2, 128}, {4, 4, 4, 64}, {4, 4, 8, 64},
    {16, 4, 4, 128}, {8, 4, 2, 128}, {4, 4, 2, 64}, {8, 2, 4, 64}, {4, 2, 4, 32},
};

template <typename S> __global__ void fill_state_kernel(int64_t n, vec4<S> *U, vec4<S> *A, vec4<S> *x)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        U[i] = {S(0.5), S(-0.25), S(0.125), S(1)};
        A[i] = {S(0), S(0), S(0), S(1)};  // s = 1
        x[i] = {S(1), S(1), S(1), S(1)};
    }
}

// seconds per launch of one operator with the mesh's current brick: one
// warm-up launch, then reps launches between CUDA events
template <typename T>
fsi_status time_op(fsi_mesh *m, int op, int reps, const void *U, const void *A, const void *x,
                   void *out, void *R, cudaEvent_t e0, cudaEvent_t e1, double *seconds)
{
    auto run = [&]() {
        if (op == 2) return launch_fused<T>(m, U, A, nullptr, x, R, out);
        return op ? launch<T, true>(m, U, A, nullptr, x, out)
                  : launch<T, false>(m, U, A, nullptr, nullptr, out);
    };
    FSI_TRY(run());
    FSI_CUDA(cudaEventRecord(e0, m->stream), "event");
    for (int r = 0; r < reps; ++r) FSI_TRY(run());
    FSI_CUDA(cudaEventRecord(e1, m->stream), "event");
    FSI_CUDA(cudaEventSynchronize(e1), "event sync");
    float ms = 0.0f;
    FSI_CUDA(cudaEventElapsedTime(&ms, e0, e1), "elapsed");
    *seconds = 1e-3 * ms / reps;
    return FSI_OK;
}

static_assert(kMeshCandidates <= FSI_TUNE_MAX_CANDIDATES, "the report holds every candidate");
template <typename T> fsi_status autotune(fsi_mesh *m, int op, int reps, fsi_tune_report *rep)
{
    using S = typename StorageOf<T>::type;
    const int slot = prec_slot<T>();
    const Brick start = m->brick[op][slot];
    const size_t bytes = (size_t)m->n_nodes * sizeof(vec4<S>);
    void *buf[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    fsi_status st = FSI_OK;
    for (void *&b : buf)
        if (cudaMalloc(&b, bytes) != cudaSuccess) {
            cudaGetLastError();
            st = set_error(FSI_ERR_OOM, "fsi_mesh_autotune: cudaMalloc failed");
        }
    if (st == FSI_OK &&
        (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess))
        st = set_error(FSI_ERR_CUDA, "fsi_mesh_autotune: cudaEventCreate failed");
    // the present schedule is the first candidate and the one to beat
    const bool jac = op > 0, fused = op == 2;
    std::vector<Brick> cands(1, fit_brick(start, (int)sizeof(T), jac, fused));
    for (const Brick &b : kMeshBricks) {
        const Brick c = fit_brick(b, (int)sizeof(T), jac, fused);
        bool seen = false;
        for (const Brick &o : cands)
            seen = seen || (o.bx == c.bx && o.by == c.by && o.bz == c.bz && o.threads == c.threads);
        if (!seen && (int)cands.size() < kMeshCandidates) cands.push_back(c);
    }
    double best = 1e30;
    Brick best_brick = start;
    int tried = 0;
    auto time_brick = [&](const Brick &b, double *t) {
        m->brick[op][slot] = b;
        return time_op<T>(m, op, reps, buf[0], buf[1], buf[2], buf[3], buf[4], e0, e1, t);
    };
    if (st == FSI_OK) {
        fill_state_kernel<S><<<sm_count() * 4, 256, 0, m->stream>>>(m->n_nodes, (vec4<S> *)buf[0],
                                                             (vec4<S> *)buf[1], (vec4<S> *)buf[2]);
        st = check_launch("autotune fill");
    }
    double t = 0.0;
    if (st == FSI_OK) st = time_brick(start, &t);  // not counted: the clocks come up
    for (const Brick &cand : cands) {
        if (st != FSI_OK) break;
        st = time_brick(cand, &t);
        if (st != FSI_OK) break;
        rep->cand_bx[tried] = cand.bx;
        rep->cand_by[tried] = cand.by;
        rep->cand_bz[tried] = cand.bz;
        rep->cand_ctas[tried] = cand.threads;
        rep->cand_seconds[tried] = t;
        ++tried;
        if (t < best) {
            best = t;
            best_brick = cand;
        }
    }
    m->brick[op][slot] = st == FSI_OK ? best_brick : start;
    cudaStreamSynchronize(m->stream);
    for (void *b : buf) cudaFree(b);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (st != FSI_OK) return st;
    rep->n_candidates = tried;
    rep->bx = best_brick.bx;
    rep->by = best_brick.by;
    rep->bz = best_brick.bz;
    rep->threads = best_brick.threads;
    rep->ctas_per_sm = 0;
    rep->seconds = best;
    return FSI_OK;
}

}  // namespace

fsi_status vms_residual(fsi_mesh *m, fsi_prec prec, const void *U, const void *A,
                        const void *f, void *R)
{
    if (m->tet) return fsi_tet_residual(m->tet, prec, U, A, f, R);
    if (prec == FSI_F64) return launch<double, false>(m, U, A, f, nullptr, R);
    if (prec == FSI_DF64) return launch<df64, false>(m, U, A, f, nullptr, R);
    return launch<float, false>(m, U, A, f, nullptr, R);
}

fsi_status vms_residual_jacobian(fsi_mesh *m, fsi_prec prec, const void *U, const void *A,
                                 const void *f, const void *x, void *R, void *Jx)
{
    if (m->tet) {
        FSI_TRY(fsi_tet_residual(m->tet, prec, U, A, f, R));
        return fsi_tet_jacobian_apply(m->tet, prec, U, A, f, x, Jx);
    }
    if (prec == FSI_F64) return launch_fused<double>(m, U, A, f, x, R, Jx);
    if (prec == FSI_DF64) return launch_fused<df64>(m, U, A, f, x, R, Jx);
    return launch_fused<float>(m, U, A, f, x, R, Jx);
}

fsi_status vms_jacobian(fsi_mesh *m, fsi_prec prec, const void *U, const void *A,
                        const void *f, const void *x, void *Jx)
{
    if (m->tet) return fsi_tet_jacobian_apply(m->tet, prec, U, A, f, x, Jx);
    if (prec == FSI_F64) return launch<double, true>(m, U, A, f, x, Jx);
    if (prec == FSI_DF64) return launch<df64, true>(m, U, A, f, x, Jx);
    return launch<float, true>(m, U, A, f, x, Jx);
}

}  // namespace fsi

using namespace fsi;

extern "C" fsi_status fsi_mesh_autotune(fsi_mesh *mesh, int op, fsi_prec prec, int reps,
                                        fsi_tune_report *report)
{
    FSI_TRY(validate_mesh(mesh));
    FSI_TRY(require_structured(mesh, "fsi_mesh_autotune"));
    if (op < 0 || op > 2 || reps < 1 || !report ||
        (prec != FSI_F64 && prec != FSI_F32 && prec != FSI_DF64))
        return set_error(FSI_ERR_ARG, "fsi_mesh_autotune: bad arguments");
    FSI_DEVICE(mesh->device);
    std::memset(report, 0, sizeof *report);
    if (prec == FSI_F64) return autotune<double>(mesh, op, reps, report);
    if (prec == FSI_DF64) return autotune<df64>(mesh, op, reps, report);
    return autotune<float>(mesh, op, reps, report);
}

