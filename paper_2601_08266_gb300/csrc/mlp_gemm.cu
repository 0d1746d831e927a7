// mlp_gemm.cu -- the training GEMM of the initial-guess network on the
// 5th-generation tensor cores (tcgen05, TMEM accumulators): an extension, the
// paper has no counterpart.
//
// C[M x N] = epi(op(A)[M x K] op(B)[K x N]) with FP32 operands in global
// memory, rounded to BF16 when they are staged into shared memory (the
// rounding points of the network's BF16 arithmetic), FP32 accumulation in
// TMEM.  One CTA (256 threads) computes a 128 x BN tile, BN = N rounded up to
// a multiple of 16 and at most 64, and walks K in chunks of 64 through two
// shared-memory stages:
//
//   all threads    hold the next chunk's A rows and B columns in registers
//                  (all of its loads in flight at once, issued before the
//                  previous chunk's MMAs are waited for), round them to BF16
//                  and store them in the K-major canonical layout of the UMMA
//                  descriptors (8-row x 16-byte core matrices);
//   thread 0       issues 4 tcgen05.mma (M = 128, N = BN, K = 16) and commits
//                  them to the stage's mbarrier, while the other threads go on
//                  with the next chunk;
//   epilogue       warp w reads TMEM lanes 32 (w % 4) .. (its tile rows) and
//                  every other group of 8 columns (w / 4 picks which), adds
//                  the bias, applies ReLU (keeping the pre-activation) or the
//                  ReLU mask of the backward pass, and stores FP32.
//
// The network's GEMMs are small (4096 x 256 x 256 at the training batch: 0.3 us
// at the tensor rate), so what bounds them is the latency of staging and how many
// SMs take part.  64-column tiles make 128 CTAs of a 4096 x 256 output (256-column
// tiles made 32, one fifth of the chip), and with a whole chunk's loads in flight a
// chunk costs one memory latency (eight scalar loads at a time cost twelve).  With
// the grouped weight gradients below, a training step of 4,096 rows (loss, gradient
// and Adam) went from 458 to 133 us, bit for bit the same.
//
// Weight gradients (K = batch, M and N <= 256) split K over up to 32 slices;
// each writes its partial tile to a workspace whose slices are then summed in a
// fixed order, so results are deterministic.  The three weight gradients of a
// training step go as one launch (tc_gemm_group) and one launch sums them.  Every
// mbarrier wait is bounded: one that runs out raises the error flag, the CTA waits
// (bounded) for its own MMAs and frees its TMEM.
#include <algorithm>
#include <cstdint>

#include "fsi_internal.cuh"
#include "tc_common.cuh"

namespace fsi {
namespace {

using namespace tc;

constexpr int TM = 128;       // tile rows (MMA M)
constexpr int BK = 64;        // K per stage (4 MMAs of K = 16)
constexpr int KCH = BK / 8;   // 16-byte chunks along K in a stage
constexpr int kThreads = 256;
constexpr uint32_t SZ_A = TM * BK * 2;      // 16 KB
constexpr int kMaxBN = kGemmMaxBN;
constexpr uint32_t SZ_B = kMaxBN * BK * 2;  // 8 KB
constexpr uint32_t SZ_STAGE = SZ_A + SZ_B;
constexpr uint32_t SMEM_BYTES = 2 * SZ_STAGE;  // 48 KB
constexpr int kTaskA = TM * KCH / kThreads;      // 16-byte chunks of A per thread
constexpr int kTaskB = kMaxBN * KCH / kThreads;  // ... of B
constexpr int kMaxSplit = 32;

// up to three GEMMs of one launch: CTAs [start[q], start[q + 1]) take GEMM q
struct Group {
    int n, start[4];
    TcGemm g[3];
};

// One operand's chunk: N_T tasks of (row, 8 consecutive k) per thread.  KC: k is
// contiguous in memory (lane -> row lane % 8, so that a warp's 16-byte stores fall
// on different banks and each row's 32-byte pieces are whole sectors); otherwise
// rows are contiguous (consecutive lanes take consecutive rows).
template <int N_T, bool KC>
__device__ __forceinline__ void task_place(int tid, int t, int rows, int &r, int &q)
{
    const int id = tid + t * kThreads;
    if (KC) {
        const int lane = id & 31, w = id >> 5;  // warp task: 8 rows x 4 chunks
        r = (w >> 1) * 8 + (lane & 7);
        q = (w & 1) * 4 + (lane >> 3);
    } else {
        r = id % rows;
        q = id / rows;
    }
}
template <int N_T, bool KC>
__device__ __forceinline__ void load_tasks(const float *__restrict__ p, int64_t ld, int rows, int tid,
                                           int row0, int nrow, int k0, int K, bool vec,
                                           float (&v)[N_T][8])
{
#pragma unroll
    for (int t = 0; t < N_T; ++t) {
        int r, q;
        task_place<N_T, KC>(tid, t, rows, r, q);
        const int gr = row0 + r, gk = k0 + 8 * q;
        const bool in = r < rows && q < KCH && gr < nrow;
        if (KC && vec) {
            // 16-byte aligned rows, K a multiple of 4
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
                if (in && gk + 4 * h < K)
                    f = *reinterpret_cast<const float4 *>(p + (int64_t)gr * ld + gk + 4 * h);
                v[t][4 * h] = f.x;
                v[t][4 * h + 1] = f.y;
                v[t][4 * h + 2] = f.z;
                v[t][4 * h + 3] = f.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                v[t][j] = 0.f;
                if (in && gk + j < K)
                    v[t][j] = KC ? p[(int64_t)gr * ld + gk + j] : p[(int64_t)(gk + j) * ld + gr];
            }
        }
    }
}
template <int N_T, bool KC>
__device__ __forceinline__ void store_tasks(uint8_t *s, int rows, int tid, const float (&v)[N_T][8])
{
#pragma unroll
    for (int t = 0; t < N_T; ++t) {
        int r, q;
        task_place<N_T, KC>(tid, t, rows, r, q);
        if (r < rows && q < KCH)
            *reinterpret_cast<uint4 *>(s + kmaj(r, 8 * q, KCH)) =
                make_uint4(pack_bf16(v[t][0], v[t][1]), pack_bf16(v[t][2], v[t][3]),
                           pack_bf16(v[t][4], v[t][5]), pack_bf16(v[t][6], v[t][7]));
    }
}

// AK / BKc: k contiguous in A / in B's columns
template <bool AK, bool BKc>
__device__ __forceinline__ void gemm_body(const TcGemm &g, int cta, int *err, uint8_t *sm,
                                          uint64_t *bars, uint32_t *tmem_holder, int *abort_sh)
{
    volatile int &abort_flag = *abort_sh;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int nt = (g.N + g.BN - 1) / g.BN, mt = (g.M + TM - 1) / TM;
    const int z = cta / (nt * mt), tile = cta - z * (nt * mt);
    const int m0 = (tile / nt) * TM, n0 = (tile % nt) * g.BN;
    const uint32_t s0 = smem_u32(sm);
    const uint32_t bar[2] = {smem_u32(&bars[0]), smem_u32(&bars[1])};
    // K range of this CTA (slice z of g.splits slices of whole chunks)
    const int nchunks_all = (g.K + BK - 1) / BK;
    const int per = (nchunks_all + g.splits - 1) / g.splits;
    const int c_begin = z * per;
    const int c_end = min(nchunks_all, c_begin + per);
    const int nch = max(0, c_end - c_begin);
    // TMEM columns: a power of two >= 32 holding BN FP32 columns
    const uint32_t cols = g.BN <= 32 ? 32 : 64;

    float va[kTaskA][8], vb[kTaskB][8];
    auto load = [&](int c) {
        const int k0 = (c_begin + c) * BK;
        load_tasks<kTaskA, AK>(g.A, g.lda, TM, tid, m0, g.M, k0, g.K, g.vec & 1, va);
        load_tasks<kTaskB, BKc>(g.B, g.ldb, g.BN, tid, n0, g.N, k0, g.K, g.vec & 2, vb);
    };
    if (nch > 0) load(0);
    if (tid == 0) {
        abort_flag = 0;
        mbar_init(bar[0], 1);
        mbar_init(bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    if (warp == 0) tmem_alloc(smem_u32(tmem_holder), cols);
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_holder;
    const uint32_t idesc = idesc_bf16(TM, g.BN);
    // parity of the commit issued on each stage and not yet observed (-1: none)
    int pending[2] = {-1, -1};

    for (int c = 0; c < nch; ++c) {
        const int st = c & 1;
        uint8_t *sa = sm + st * SZ_STAGE;
        uint8_t *sb = sa + SZ_A;
        // the MMAs of chunk c - 2 read this stage: wait for them
        if (c >= 2) {
            const bool ok = mbar_wait(bar[st], ((c - 2) >> 1) & 1);
            if (ok) pending[st] = -1;
            else atomicExch(abort_sh, 1);
            __syncthreads();
            if (abort_flag) break;
        }
        store_tasks<kTaskA, AK>(sa, TM, tid, va);
        store_tasks<kTaskB, BKc>(sb, g.BN, tid, vb);
        if (c + 1 < nch) load(c + 1);
        fence_async_smem();
        fence_before();
        __syncthreads();
        if (tid == 0) {
            fence_after();
            const uint32_t a0 = s0 + st * SZ_STAGE, b0 = a0 + SZ_A;
#pragma unroll
            for (uint32_t ks = 0; ks < BK / 16; ++ks)
                mma_bf16(tmem, sdesc(a0 + ks * 256, 128, KCH * 128),
                         sdesc(b0 + ks * 256, 128, KCH * 128), idesc, (c > 0 || ks > 0) ? 1u : 0u);
            mma_commit(bar[st]);
        }
        pending[st] = (c >> 1) & 1;
    }
    // all MMAs done: the last commit covers every earlier one
    if (nch > 0 && !abort_flag) {
        const int last = nch - 1;
        const bool ok = mbar_wait(bar[last & 1], (last >> 1) & 1);
        if (ok) pending[0] = pending[1] = -1;
        else atomicExch(abort_sh, 1);
    }
    __syncthreads();
    fence_after();
    if (!abort_flag) {
        // epilogue: rows 32 (warp % 4) + lane, column groups of 8 split by warp / 4
        const int row = 32 * (warp & 3) + (tid & 31);
        const int gi = m0 + row;
        const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
        for (int c8 = warp >> 2; c8 * 8 < g.BN; c8 += 2) {
            float v[8];
            if (nch > 0) tmem_ld8(tmem + lane_base + 8 * c8, v);
            else
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = 0.f;
            if (gi >= g.M) continue;
            const int gj0 = n0 + 8 * c8, nc = gemm_piece_columns(gj0, g.N);
            if (nc == 0) continue;
            if (g.splits > 1) {  // partial sum of a K slice
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (j < nc) g.work[((int64_t)z * g.M + gi) * g.N + gj0 + j] = v[j];
                continue;
            }
            const int64_t o = (int64_t)gi * g.ldc + gj0;
            // bias, pre-activation, ReLU or mask
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (j >= nc) break;
                if (g.epi == TC_EPI_BIAS || g.epi == TC_EPI_BIAS_RELU) v[j] += g.bias[gj0 + j];
                if (g.epi == TC_EPI_MASK) v[j] = g.mask[o + j] > 0.f ? v[j] : 0.f;
            }
            if ((g.vec & 4) && nc == 8) {  // whole 16-byte pieces, see tc_gemm_group
                if (g.epi == TC_EPI_BIAS_RELU) {
                    if (g.Cpre) {
                        *reinterpret_cast<float4 *>(g.Cpre + o) = make_float4(v[0], v[1], v[2], v[3]);
                        *reinterpret_cast<float4 *>(g.Cpre + o + 4) = make_float4(v[4], v[5], v[6], v[7]);
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = v[j] > 0.f ? v[j] : 0.f;
                }
                *reinterpret_cast<float4 *>(g.C + o) = make_float4(v[0], v[1], v[2], v[3]);
                *reinterpret_cast<float4 *>(g.C + o + 4) = make_float4(v[4], v[5], v[6], v[7]);
                continue;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (j >= nc) break;
                if (g.epi == TC_EPI_BIAS_RELU) {
                    if (g.Cpre) g.Cpre[o + j] = v[j];
                    v[j] = v[j] > 0.f ? v[j] : 0.f;
                }
                g.C[o + j] = v[j];
            }
        }
    }
    if (abort_flag) {
        if (tid == 0) atomicExch(err, 1);
        // nothing may still be in flight when the TMEM is freed
        for (int q = 0; q < 2; ++q)
            if (pending[q] >= 0) mbar_wait(bar[q], (uint32_t)pending[q]);
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        fence_after();
        tmem_free(tmem, cols);
    }
}

__global__ void __launch_bounds__(kThreads) tc_gemm_kernel(const Group G, int *err)
{
    extern __shared__ __align__(128) uint8_t sm[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ uint32_t tmem_holder;
    __shared__ int abort_flag;
    int q = 0;
    while (q + 1 < G.n && (int)blockIdx.x >= G.start[q + 1]) ++q;
    TcGemm g = G.g[q];
    chain_wait(g.A, g.B, g.bias, g.mask, g.work, g.C, g.Cpre);
    chain_trigger();
    const int cta = blockIdx.x - G.start[q];
    if (g.transA) {
        if (g.transB) gemm_body<false, true>(g, cta, err, sm, bars, &tmem_holder, &abort_flag);
        else gemm_body<false, false>(g, cta, err, sm, bars, &tmem_holder, &abort_flag);
    } else {
        if (g.transB) gemm_body<true, true>(g, cta, err, sm, bars, &tmem_holder, &abort_flag);
        else gemm_body<true, false>(g, cta, err, sm, bars, &tmem_holder, &abort_flag);
    }
}

// C = sum over the K slices of the partial tiles, in slice order, of every GEMM
// of the group that was split
__global__ void tc_gemm_reduce_kernel(const Group G)
{
    chain_wait();
    chain_trigger();
    for (int q = 0; q < G.n; ++q) {
        TcGemm g = G.g[q];
        chain_pin(g.work);
        if (g.splits < 2) continue;
        const int64_t total = (int64_t)g.M * g.N;
        for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
             e += (int64_t)gridDim.x * blockDim.x) {
            float s = 0.f;
#pragma unroll 8
            for (int z = 0; z < g.splits; ++z) s += g.work[(int64_t)z * total + e];
            g.C[(e / g.N) * g.ldc + e % g.N] = s;
        }
    }
}

}  // namespace

size_t tc_gemm_work_floats() { return (size_t)kMaxSplit * 256 * (256 + 256 + 16); }

fsi_status tc_gemm_group(cudaStream_t s, const TcGemm *gs, int n, float *work, int *err)
{
    if (n < 1 || n > 3) return set_error(FSI_ERR_ARG, "tensor-core GEMM: bad group");
    Group G;
    G.n = n;
    G.start[0] = 0;
    int64_t reduce = 0;
    size_t used = 0;
    for (int q = 0; q < n; ++q) {
        TcGemm &g = G.g[q];
        g = gs[q];
        if (g.M <= 0 || g.N <= 0 || g.K <= 0 || g.N > 256)
            return set_error(FSI_ERR_ARG, "tensor-core GEMM: bad shape %d x %d x %d", g.M, g.N, g.K);
        g.BN = gemm_tile_columns(g.N);
        const int mt = (g.M + TM - 1) / TM, nt = (g.N + g.BN - 1) / g.BN;
        const int nchunks = (g.K + BK - 1) / BK;
        // split K when 256-column tiles alone would leave most SMs idle and K is
        // long: 4 chunks a slice (the slices, and so the sums, do not depend on BN)
        int splits = 1;
        if (g.epi == TC_EPI_STORE && work && mt < sm_count() / 2 && nchunks >= 8) {
            splits = nchunks / 4;
            if (splits > kMaxSplit) splits = kMaxSplit;
            if (used + (size_t)splits * g.M * g.N > tc_gemm_work_floats()) splits = 1;
            // every slice gets whole chunks, and none is empty
            const int per = (nchunks + splits - 1) / splits;
            splits = (nchunks + per - 1) / per;
        }
        g.splits = splits;
        g.work = work + used;
        if (splits > 1) {
            used += (size_t)splits * g.M * g.N;
            reduce = std::max(reduce, (int64_t)g.M * g.N);
        }
        auto al = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
        g.vec = (!g.transA && al(g.A) && g.lda % 4 == 0 && g.K % 4 == 0 ? 1 : 0) |
                (g.transB && al(g.B) && g.ldb % 4 == 0 && g.K % 4 == 0 ? 2 : 0) |
                (al(g.C) && al(g.Cpre) && g.ldc % 4 == 0 && g.N % 8 == 0 ? 4 : 0);
        G.start[q + 1] = G.start[q] + mt * nt * splits;
    }
    FSI_TRY(set_smem_limit((const void *)tc_gemm_kernel, SMEM_BYTES));
    launch_chain(tc_gemm_kernel, G.start[n], kThreads, SMEM_BYTES, s, G, err);
    FSI_TRY(check_launch("tensor-core gemm"));
    if (reduce > 0) {
        const int blocks = (int)std::min<int64_t>((reduce + 255) / 256, sm_count() * 8);
        launch_chain(tc_gemm_reduce_kernel, blocks, 256, 0, s, G);
        FSI_TRY(check_launch("tensor-core gemm reduce"));
    }
    return FSI_OK;
}

fsi_status tc_gemm(cudaStream_t s, const TcGemm &g, float *work, int *err)
{
    return tc_gemm_group(s, &g, 1, work, err);
}

}  // namespace fsi
