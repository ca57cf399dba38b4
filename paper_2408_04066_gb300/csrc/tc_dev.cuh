// Inline-PTX helpers of the kernels that use the TMA engine, mbarriers and the
// tensor cores (k_coarse_tc.cu, k_pcg_resident.cu), and the layout of the packed
// BF16 rows of A_c^{-1} they both stream.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "dev.cuh"

namespace mfem {

constexpr int kFuSplit = 4;                       // parts of the K range (CTAs per cluster in k_coarse_fused)
constexpr int kFuAggsCta = 5;                     // aggregates each part's CTA corrects
constexpr int kFuAggsBlk = kFuSplit * kFuAggsCta; // aggregates per row block
constexpr int kTcM = 128;                         // MMA M: rows of A_c^{-1} per row block (6 x 20, padded)
constexpr int kTcSteps = kTcKC / 16;              // MMAs per chunk (K = 16 each)
constexpr int kFuStepA = kTcM * 16 * 2;           // bytes of A per K step (4 KB)
constexpr int kFuChunkA = kFuStepA * kTcSteps;    // 32 KB
constexpr uint64_t kTcWaitNs = 200ull * 1000ull * 1000ull;   // 0.2 s per bounded wait ...
constexpr uint32_t kTcWaitPolls = 1u << 12;                  // ... and this many polls of it (under 1 ms of waiting)

// Row blocks of an N x N inverse (runs of the mesh's aggregates)
__host__ __device__ __forceinline__ int row_blocks(int N) { return (N / 6 + kFuAggsBlk - 1) / kFuAggsBlk; }
// Chunks of the K range that one of the kFuSplit parts takes
__host__ __device__ __forceinline__ int coarse_part_chunks(int N) {
    return (coarse_chunks(N) + kFuSplit - 1) / kFuSplit;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for phase `parity` of the barrier to complete; false if it has not after
// kTcWaitNs and kTcWaitPolls polls.  The clock runs on while another process has the
// GPU, the polls do not: a pause alone does not end a wait.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    const uint64_t t0 = global_ns();
    for (uint32_t n = 0; !mbar_try_wait(bar, parity); ++n)
        if (n >= kTcWaitPolls && global_ns() - t0 > kTcWaitNs) return mbar_try_wait(bar, parity);
    return true;
}

// 1-D bulk copy global -> shared through the TMA engine; completes `bytes` of
// transaction count on the barrier.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor of a no-swizzle K-major operand: start
// address, byte offset between K-adjacent core matrices (leading) and between
// 8-row groups (stride), descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lead, uint32_t stride) {
    uint64_t d = (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lead >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((stride >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// Descriptor of a 128-byte-swizzled K-major operand (rows of 128 bytes, 1024-byte
// aligned 8-row atoms 1024 bytes apart; within a row the 16-byte pieces are permuted
// by piece ^ (row mod 8)): A_c^{-1}.  A K step of 16 columns is 32 bytes further.
// An MMA (M = 128, N = 16 or 48) whose A is not swizzled waits for its A operand:
// 165 cycles an instruction.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// Byte offset of K step k (16 columns) of a chunk's A
__host__ __device__ __forceinline__ uint32_t a_step(int k) { return (uint32_t)(k >> 2) * (kTcM * 128) + (k & 3) * 32; }
// Byte offset of 16-byte piece j (columns 8 j .. 8 j + 7) of row `row` of a chunk's A
__host__ __device__ __forceinline__ uint32_t a_piece(int row, int j) {
    return (uint32_t)(j >> 3) * (kTcM * 128) + row * 128 + (((j & 7) ^ (row & 7)) << 4);
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N and M as given.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

// Warp-wide (.aligned) instructions: undefined unless the warp's 32 threads execute them
// together, which neither an `if` on one thread nor a per-thread wait before them, nor
// a block barrier, ensures -- so each starts with its own __syncwarp().

// Tensor memory: `cols` columns (a power of two >= 32) into *slot; their release
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
    __syncwarp();
    asm volatile(
        "tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n\t"
        "tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::"r"(smem_u32(slot)),
        "r"(cols)
        : "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t tmem, uint32_t cols) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}

// 4 or 16 consecutive FP32 columns of this thread's TMEM lane, loaded when it returns
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[4]) {
    uint32_t r[4];
    __syncwarp();
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    __syncwarp();
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// Eight 32-bit columns of this thread's TMEM lane, and the wait for the warp's stores
__device__ __forceinline__ void tmem_st(uint32_t taddr, uint4 a, uint4 b) {
    __syncwarp();
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(a.x),
                 "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
}
__device__ __forceinline__ void tmem_st_wait() {
    __syncwarp();
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Cluster barrier: every write before arrive() is visible to the cluster after wait()
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace mfem
