// Coarse solve and correction of the two-level preconditioner on the tensor
// cores, fused into one kernel: one launch per PCG iteration serves up to
// kCoarseJobs meshes.
//
// u = zb + P e,  e = A_c^{-1} r_c  for every two-level problem of one mesh: the
// product is the one dense contraction of the solve (the preconditioner's
// reduced space; the method itself has none, paper §5) and it is bound by
// streaming A_c^{-1}, stored once per mesh in BF16.
//
//   * A cluster of kFuSplit CTAs owns a row block of kFuAggsBlk aggregates
//     (their 6 kFuAggsBlk rows of A_c^{-1}, padded to the MMA's M = 128); CTA q
//     of the cluster streams the q-th part of the K range: per chunk of kTcKC
//     columns one 32 KB block of A (packed at set-up in the MMA's 128-byte-swizzled
//     K-major layout) and the matching 12 KB chunk of the B
//     operand, by 1-D bulk copies (the TMA engine) into a ring of kFuStages
//     shared-memory stages; one thread issues the MMAs (M = 128, N = 48,
//     K = 16), FP32 accumulation in tensor memory.
//   * The cluster adds its kFuSplit partial products through distributed
//     shared memory in rank order (deterministic), CTA q keeping the rows of
//     its kFuAggsCta aggregates; then every thread of the CTA applies the
//     correction to those aggregates' vertex rows: u_i = zb_i + Q_a (e_t +
//     e_w x (X_i - c_a)), written to the neighbour record the next SpMV
//     gathers.  No slice partials, no separate correction kernel.
//   * B: each problem's r_c split exactly into three BF16 parts (r = hi + mid +
//     lo: 3 x 8 significand bits hold the FP32 value), N = 48 columns for 16
//     request slots; the restriction writes it in the operand layout (see
//     coarse_b_store).  The epilogue adds the three FP32 partial products, so
//     the preconditioner stays the fixed linear map block-Jacobi + P Ahat P^T
//     with Ahat = bf16(A_c^{-1}) (symmetric: rounding is entrywise), which
//     keeps PCG's theory intact at any tolerance.
//
// Every wait on a copy or an MMA is bounded (mbar_wait); a wait that
// runs out sets a bit of the mesh's error word (read by the host after the
// solve), waits (bounded) for the copies it issued and frees its tensor memory.
// The cluster barriers are reached by every CTA of a cluster on every path.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.h"
#include "tc_dev.cuh"

namespace mfem {

namespace {

// Shared-memory ring of A + B chunks: four stages, one CTA an SM; two stages and
// two CTAs an SM where a launch of several meshes has more CTAs than the device
// has SMs, so that none waits for a second wave (12 + 12 streams of the 200k and
// 50k figures 80.0 -> 78.9 us an iteration, the 10k/50k/200k requests 18.75 -> 17.7
// ms; one mesh alone is slower with two: 72.0 -> 74.8 us, 16 poses of the 200k figure).
constexpr int kFuStages = 4, kFuStagesMulti = 2;
constexpr int kFuThreads = 320;                   // 10 warps: one per 32 vertex rows of 5 x 64
constexpr int kTcProbs = kCoarseGroupSlots;       // request slots per CTA group
constexpr int kTcN = kCoarseBRows;                // MMA N: three BF16 parts per slot
constexpr int kFuStepB = kTcN * 16 * 2;           // bytes of B per K step (1.5 KB)
constexpr int kFuChunkB = kFuStepB * kTcSteps;    // 12 KB
constexpr int kFuStage = kFuChunkA + kFuChunkB;   // 44 KB
constexpr int fu_smem(int stages) { return stages * kFuStage + 128; }
constexpr int kTcTmemCols = 64;                   // >= kTcN, a power of two >= 32

static_assert(6 * kFuAggsBlk <= kTcM, "a row block's coarse rows fit the MMA's M");
static_assert(kFuChunkB == kCoarseBChunk * 2, "B chunk layout shared with the restriction");
constexpr int kSms = 152;                         // SMs of a GB300
static_assert(kTcM * kTcN * 4 <= kFuStage, "the partial product fits one stage for the cluster sum");
static_assert(kFuChunkA % 16 == 0 && kFuChunkB % 16 == 0 && kFuStage % 1024 == 0, "bulk copies: 16-byte units");
static_assert(kFuThreads >= 128, "warps 0-3 read the 128 TMEM lanes");

// Set-up: FP32 A_c^{-1} (rows of ld floats) -> per row block and chunk, BF16.
__global__ void k_coarse_pack_bf16(const float* __restrict__ Ainv, int N, int ld, int nkc,
                                   __nv_bfloat16* __restrict__ out) {
    const int kk = threadIdx.x;                        // column within the chunk
    const int r = blockIdx.y % kTcM, rb = blockIdx.y / kTcM;
    const int ch = blockIdx.z;
    const int row = rb * 6 * kFuAggsBlk + r, k = ch * kTcKC + kk;
    const float v = (r < 6 * kFuAggsBlk && row < N && k < N) ? Ainv[(size_t)row * ld + k] : 0.f;
    out[((size_t)rb * nkc + ch) * (kFuChunkA / 2) + a_piece(r, kk >> 3) / 2 + (kk & 7)] = __float2bfloat16_rn(v);
}

// mfem_coarse_apply: r_c of B problems (rows of ldr floats) -> their B operand.
__global__ void k_coarse_split(const float* __restrict__ rc, int N, int ldr, int nkc, uint16_t* __restrict__ bs) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.y;
    if (k >= N) return;
    coarse_b_store(bs + (size_t)(b / kCoarseGroupSlots) * nkc * kCoarseBChunk, b % kCoarseGroupSlots, k,
                   rc[(size_t)b * ldr + k]);
}

__device__ __forceinline__ void stv(float* p, const float (&v)[3]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], 0.f);
}
__device__ __forceinline__ void stv(double* p, const double (&v)[3]) {
    reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(v[2], 0.0);
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    cluster_arrive();
    cluster_wait();
}
// FP32 at the same shared-memory offset in CTA `rank` of the cluster
__device__ __forceinline__ float ld_cluster_f32(const float* local, uint32_t rank) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(local)), "r"(rank));
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(remote) : "memory");
    return v;
}

// The jobs (meshes) of one launch: job j's clusters are c0[j] .. c0[j + 1] - 1.
// One launch for all of them: a small mesh's product takes as long as a large
// one's (its chain of latencies) on a few SMs, so several run side by side.
struct TcJobs {
    struct Job {
        const __nv_bfloat16* Abf;
        const uint16_t* Bs;
        unsigned* err;
        int N, d0, nd;
    } job[kCoarseJobs];
    int c0[kCoarseJobs + 1];
    int n;
};

// Cluster (rb, pg) of a job: row block rb (aggregates kFuAggsBlk rb ..), request slots
// 16 pg .. 16 pg + 15 of the context; CTA q = cluster rank takes chunks
// [q c_per, (q + 1) c_per) of the K range and corrects aggregates
// kFuAggsBlk rb + kFuAggsCta q ...  The problems are found in the descriptor
// table d0 .. d0+nd-1 by slot; a slot without a two-level problem inside PCG
// contributes nothing (its B columns give outputs never read).
// e_out (mfem_coarse_apply): write e[slot][row] instead of the correction.
template <typename T, int ST>
__global__ void __launch_bounds__(kFuThreads, ST == kFuStagesMulti ? 2 : 1)
    k_coarse_fused(const __grid_constant__ TcJobs J, const PcgDesc<T>* __restrict__ D, float* __restrict__ e_out) {
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + ST * kFuStage);   // chunk landed
    uint64_t* empty = full + ST;                                           // its MMAs done
    uint64_t* done = empty + ST;                                           // every MMA done
    uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
    float* red = reinterpret_cast<float*>(smem);   // after the K loop: the partial product [kTcN][kTcM]
    __shared__ const PcgDesc<T>* dp[kTcProbs];
    __shared__ float es[6 * kFuAggsCta][kTcProbs + 1];
    __shared__ float qs[kFuAggsCta][kTcProbs][9];
    __shared__ int any, s_ok;
    constexpr bool kEarly = ST != kFuStagesMulti;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const uint32_t q = cluster_rank();
    const int cid = blockIdx.x / kFuSplit;   // cluster
    int ji = 0;
#pragma unroll
    for (int i = 1; i < kCoarseJobs; ++i) ji += i < J.n && cid >= J.c0[i];
    const __nv_bfloat16* __restrict__ Abf = J.job[ji].Abf;
    const uint16_t* __restrict__ Bs = J.job[ji].Bs;
    unsigned* __restrict__ err = J.job[ji].err;
    const int N = J.job[ji].N, d0 = J.job[ji].d0, nd = J.job[ji].nd;
    const int nkc = coarse_chunks(N);
    const int rb = (cid - J.c0[ji]) % row_blocks(N), pg = (cid - J.c0[ji]) / row_blocks(N);
    const int c_per = coarse_part_chunks(N);
    const int c_lo = min(nkc, (int)q * c_per), nch = min(nkc, c_lo + c_per) - c_lo;   // this CTA's chunks
    const int nst = nch < ST ? nch : ST;
    const unsigned char* gA =
        reinterpret_cast<const unsigned char*>(Abf) + ((size_t)rb * nkc + c_lo) * kFuChunkA;
    const unsigned char* gB =
        reinterpret_cast<const unsigned char*>(Bs) + ((size_t)pg * nkc + c_lo) * kFuChunkB;
    const int a_cta = kFuAggsBlk * rb + kFuAggsCta * (int)q;   // first aggregate this CTA corrects
    // set-up: barriers, the first chunks of A_c^{-1} (their barriers also expect
    // the B chunk, copied after the wait), tensor memory for the 128 x 48 FP32
    // accumulator
    if (t == 0) {
        any = 0;
        s_ok = 1;
        for (int c = 0; c < 2 * ST + 1; ++c) mbar_init(&full[c], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int c = 0; c < nst; ++c) {
            mbar_expect_tx(&full[c], kFuStage);
            bulk_g2s(smem + c * kFuStage, gA + (size_t)c * kFuChunkA, kFuChunkA, &full[c]);
        }
    }
    if (t < kTcProbs) dp[t] = nullptr;
    if (warp == kFuThreads / 32 - 1) tmem_alloc(tslot, kTcTmemCols);
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    if (t == 0)   // B chunks of the first stages: written by the previous kernel
        for (int c = 0; c < nst; ++c)
            bulk_g2s(smem + c * kFuStage + kFuChunkA, gB + (size_t)c * kFuChunkB, kFuChunkB, &full[c]);
    // the group's problems by slot, meanwhile: a thread per descriptor
    if (warp == 1)
        for (int i = lane; i < nd; i += 32) {
            const PcgDesc<T>* d = &D[d0 + i];
            const int p = d->bslot - pg * kTcProbs;
            if (d->coarse && d->sc->state == kActive && p >= 0 && p < kTcProbs) {
                dp[p] = d;
                any = 1;
            }
        }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    // the same for every CTA of the cluster (same slots, states final after the wait)
    if (!any) {   // nothing to compute; let the copies land before the memory is released
        if (t == 0)
            for (int c = 0; c < nst; ++c)
                if (!mbar_wait(&full[c], 0)) atomicOr(err, 4u);
        if (warp == 0) tmem_free(tmem, kTcTmemCols);
        return;
    }

    if (t == 0) {   // one thread issues every MMA and keeps the ring full
        constexpr uint32_t idesc = umma_idesc_bf16(kTcM, kTcN);
        const uint32_t base = smem_u32(smem);
        bool ok = true;
        int issued = nst;   // chunks whose copies were issued
        for (int c = 0; c < nch && ok; ++c) {
            const int s = c % ST;
            ok = mbar_wait(&full[s], (uint32_t)(c / ST) & 1u);
            if (!ok) break;
            tc_fence_after();
            const uint32_t a0 = base + s * kFuStage, b0 = a0 + kFuChunkA;
            for (int k = 0; k < kTcSteps; ++k)
                umma_bf16(tmem, umma_desc_sw128(a0 + a_step(k)), umma_desc(b0 + k * kFuStepB, 128, 256), idesc,
                          (c > 0 || k > 0) ? 1u : 0u);
            umma_commit(&empty[s]);
            // refill the stage of the previous chunk (its MMAs were issued one
            // chunk ago) with the chunk ST after it
            const int cp = c - 1, cn = cp + ST;
            if (cp >= 0 && cn < nch) {
                const int sp = cp % ST;
                ok = mbar_wait(&empty[sp], (uint32_t)(cp / ST) & 1u);
                if (!ok) break;
                mbar_expect_tx(&full[sp], kFuStage);
                bulk_g2s(smem + sp * kFuStage, gA + (size_t)cn * kFuChunkA, kFuChunkA, &full[sp]);
                bulk_g2s(smem + sp * kFuStage + kFuChunkA, gB + (size_t)cn * kFuChunkB, kFuChunkB, &full[sp]);
                issued = cn + 1;
            }
        }
        // arrives once every MMA issued above has completed (at once if none was)
        umma_commit(done);
        if (!ok) {
            s_ok = 0;
            atomicOr(err, 1u);
            // the copies in flight: the last use of each stage that was issued, bounded
            for (int c = issued - nst; c < issued; ++c)
                if (c >= 0) mbar_wait(&full[c % ST], (uint32_t)(c / ST) & 1u);
        }
    }
    // the other warps meanwhile: the aggregates' rotations, and zb and the rest
    // offset of the thread's first vertex row (every load that the correction
    // needs but the product; the two-CTA variant has no registers for them)
    const PcgDesc<T>* d0p = nullptr;
    for (int p = 0; p < kTcProbs && !d0p; ++p) d0p = dp[p];
    const int shift = d0p->agg_shift, n = d0p->n_rows, n_agg = N / 6;
    const int row0 = a_cta << shift;
    const int row1 = e_out ? row0 : min(n, min(n_agg, a_cta + kFuAggsCta) << shift);
    const float4* crel = d0p->crel;
    const size_t np = npad32(n);
    float4 off0 = make_float4(0.f, 0.f, 0.f, 0.f);
    T z0[kTcProbs][3];
    if (kEarly && row0 + t < row1) {
        off0 = crel[row0 + t];
#pragma unroll
        for (int p = 0; p < kTcProbs; ++p)
            if (dp[p]) ld3((const T*)dp[p]->rec, np, kRecZB, row0 + t, z0[p]);
    }
    if (t >= 32)
        for (int i = t - 32; i < kFuAggsCta * kTcProbs * 9; i += kFuThreads - 32) {
            const int ai = i / (kTcProbs * 9), p = (i / 9) % kTcProbs, e = i % 9;
            const PcgDesc<T>* d = dp[p];
            const int a = a_cta + ai;
            qs[ai][p][e] = (d && d->aggq && a < N / 6) ? d->aggq[9 * a + e] : 0.f;
        }
    const bool fin = mbar_wait(done, 0);
    tc_fence_after();
    const int all_done = __syncthreads_and(fin ? 1 : 0);
    if (!all_done && t == 0) {
        atomicOr(err, 2u);
        mbar_wait(done, 0);   // once more, bounded, before the memory is reused
    }
    // this CTA's partial product -> shared memory, column-major [kTcN][kTcM]
    // (no MMA ran for a CTA without chunks: its part is zero)
    if (warp < kTcM / 32) {
        const int row = warp * 32 + lane;
        if (nch > 0 && all_done && s_ok) {
            const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
            float v[16];
#pragma unroll
            for (int part = 0; part < 3; ++part) {
                tmem_ld(lane_addr + part * kTcProbs, v);
#pragma unroll
                for (int p = 0; p < kTcProbs; ++p) red[(part * kTcProbs + p) * kTcM + row] = v[p];
            }
        } else {
#pragma unroll
            for (int c = 0; c < kTcN; ++c) red[c * kTcM + row] = 0.f;
        }
    }
    tc_fence_before();
    cluster_sync();   // every CTA's part visible to the cluster
    // the rows of this CTA's aggregates: the cluster's parts added in rank order
    for (int i = t; i < 6 * kFuAggsCta * kTcProbs; i += kFuThreads) {
        const int r = i % (6 * kFuAggsCta), p = i / (6 * kFuAggsCta);
        const int row = 6 * kFuAggsCta * (int)q + r;
        float e = 0.f;
#pragma unroll
        for (uint32_t j = 0; j < (uint32_t)kFuSplit; ++j) {
            const float hi = ld_cluster_f32(red + p * kTcM + row, j);
            const float mid = ld_cluster_f32(red + (kTcProbs + p) * kTcM + row, j);
            const float lo = ld_cluster_f32(red + (2 * kTcProbs + p) * kTcM + row, j);
            e += (hi + mid) + lo;
        }
        es[r][p] = e;
    }
    cluster_sync();   // no CTA leaves or reuses its part while another reads it
    if (warp == 0) tmem_free(tmem, kTcTmemCols);
    if (e_out) {   // the product alone
        for (int i = t; i < 6 * kFuAggsCta * kTcProbs; i += kFuThreads) {
            const int r = i % (6 * kFuAggsCta), p = i / (6 * kFuAggsCta), row = 6 * a_cta + r;
            if (dp[p] && row < N) e_out[(size_t)(pg * kTcProbs + p) * N + row] = es[r][p];
        }
        return;
    }
    // correction of the aggregates' vertex rows for every problem of the group
    for (int row = row0 + t; row < row1; row += kFuThreads) {
        const bool early = kEarly && row == row0 + t;
        const float4 off = early ? off0 : crel[row];
        const int ai = (row >> shift) - a_cta;
        if (!early)
#pragma unroll
            for (int p = 0; p < kTcProbs; ++p)
                if (dp[p]) ld3((const T*)dp[p]->rec, np, kRecZB, row, z0[p]);
#pragma unroll
        for (int p = 0; p < kTcProbs; ++p) {
            const PcgDesc<T>* d = dp[p];
            if (!d) continue;
            T z[3] = {z0[p][0], z0[p][1], z0[p][2]};
            if (off.w != 0.f) {
                const float e0 = es[6 * ai][p], e1 = es[6 * ai + 1][p], e2 = es[6 * ai + 2][p];
                const float e3 = es[6 * ai + 3][p], e4 = es[6 * ai + 4][p], e5 = es[6 * ai + 5][p];
                const float l0 = e0 + (e4 * off.z - e5 * off.y);
                const float l1 = e1 + (e5 * off.x - e3 * off.z);
                const float l2 = e2 + (e3 * off.y - e4 * off.x);
                const float* Q = qs[ai][p];
#pragma unroll
                for (int i = 0; i < 3; ++i) z[i] += (T)(Q[3 * i] * l0 + Q[3 * i + 1] * l1 + Q[3 * i + 2] * l2);
            }
            stv(d->nb + 4 * (size_t)row, z);
        }
    }
}

}  // namespace

size_t coarse_tc_bytes(int N) { return (size_t)row_blocks(N) * coarse_chunks(N) * (size_t)kFuChunkA; }

size_t coarse_b_bytes(int N, int slots) {
    const size_t groups = ((size_t)slots + kCoarseGroupSlots - 1) / kCoarseGroupSlots;
    return groups * coarse_chunks(N) * (size_t)kFuChunkB;
}

cudaError_t coarse_tc_pack(const float* Ainv, int N, void* Abf, cudaStream_t s) {
    k_coarse_pack_bf16<<<dim3(1, row_blocks(N) * kTcM, coarse_chunks(N)), kTcKC, 0, s>>>(
        Ainv, N, coarse_ld(N), coarse_chunks(N), static_cast<__nv_bfloat16*>(Abf));
    return cudaGetLastError();
}

cudaError_t coarse_split(const float* rc, int N, int ldr, int B, void* Bs, cudaStream_t s) {
    k_coarse_split<<<dim3((N + 255) / 256, B), 256, 0, s>>>(rc, N, ldr, coarse_chunks(N), static_cast<uint16_t*>(Bs));
    return cudaGetLastError();
}

template <typename T, int ST>
static cudaError_t fu_attr() {
    return cudaFuncSetAttribute(k_coarse_fused<T, ST>, cudaFuncAttributeMaxDynamicSharedMemorySize, fu_smem(ST));
}
cudaError_t coarse_tc_init() {
    cudaError_t e = fu_attr<float, kFuStages>();
    if (e == cudaSuccess) e = fu_attr<double, kFuStages>();
    if (e == cudaSuccess) e = fu_attr<float, kFuStagesMulti>();
    if (e == cudaSuccess) e = fu_attr<double, kFuStagesMulti>();
    return e;
}

template <typename T>
cudaError_t launch_coarse_fused(const cudaLaunchConfig_t& base, const CoarseJob* jobs, int n_jobs,
                                const PcgDesc<T>* descs, float* e_out) {
    TcJobs J{};
    int nc = 0;
    for (int i = 0; i < n_jobs; ++i) {   // at most kCoarseJobs
        const CoarseJob& j = jobs[i];
        J.job[i] = TcJobs::Job{static_cast<const __nv_bfloat16*>(j.Abf), static_cast<const uint16_t*>(j.Bs), j.err,
                               j.N, j.d0, j.nd};
        J.c0[i] = nc;
        nc += row_blocks(j.N) * ((j.slots + kCoarseGroupSlots - 1) / kCoarseGroupSlots);
    }
    J.n = n_jobs;
    J.c0[n_jobs] = nc;
    cudaLaunchConfig_t cfg = base;
    cudaLaunchAttribute attr[2];
    int na = 0;
    for (unsigned i = 0; i < base.numAttrs && na < 1; ++i) attr[na++] = base.attrs[i];   // programmatic launch
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = kFuSplit;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
    cfg.attrs = attr;
    cfg.numAttrs = na;
    cfg.gridDim = dim3(kFuSplit * nc);
    cfg.blockDim = dim3(kFuThreads);
    if (n_jobs > 1 && kFuSplit * nc > kSms) {
        cfg.dynamicSmemBytes = fu_smem(kFuStagesMulti);
        return cudaLaunchKernelEx(&cfg, k_coarse_fused<T, kFuStagesMulti>, J, descs, e_out);
    }
    cfg.dynamicSmemBytes = fu_smem(kFuStages);
    return cudaLaunchKernelEx(&cfg, k_coarse_fused<T, kFuStages>, J, descs, e_out);
}

template cudaError_t launch_coarse_fused<float>(const cudaLaunchConfig_t&, const CoarseJob*, int,
                                                const PcgDesc<float>*, float*);
template cudaError_t launch_coarse_fused<double>(const cudaLaunchConfig_t&, const CoarseJob*, int,
                                                 const PcgDesc<double>*, float*);

}  // namespace mfem
