// PCG of problems that fit the chip: one kernel runs every iteration.
//
// Same recurrences, same preconditioner and the same arithmetic per row as the
// streamed kernels (k_pcg.cu, k_coarse_tc.cu); what differs is where things
// live.  A problem is given a group of CTAs, one per SM; a CTA owns up to
// kResUnits units of 64 rows, a thread owns one row and keeps its r, p, s, dx,
// zb and D^{-1} in registers, and the CTA's slices of the matrix sit in shared
// memory as far as they fit (the rest is read from L2).  Only u, the coarse
// residual, the coarse partial products and the inner-product partials are
// exchanged, between four group barriers an iteration:
//
//   coarse product (tcgen05, the K-range parts of k_coarse_fused as units of
//   work)  |  u = zb + P e  |  w = K u, dots  |  alpha, beta; p, s, dx, r, zb,
//   restriction  |
//
// A group of at most 16 CTAs is a thread-block cluster: it uses the cluster
// barrier, and u, r_c and the inner-product partials go through distributed shared
// memory instead of L2.  A larger one is part of a cooperative launch (every CTA resident) and
// counts arrivals in global memory.  Groups do not wait for one another: each
// problem ends when it converges.
//
// What bounds it: the latency of the barriers and of the L2 round trips between
// them, not bytes -- these problems are the ones whose streamed iteration is
// three dependent launches that each leave most of the chip idle.  An iteration,
// streamed and here: 11k tets, one pose, 18.9 -> 9.7 us; 10k tets, 5 poses, 23.4
// -> 9.5; 50k tets, 3 poses, 26.1 -> 13.5; 200k tets, one pose, 41.0 -> 16.3 (streamed:
// before the later changes of those kernels).
//
// The chunks of A_c^{-1} a CTA multiplies stay in tensor memory (seven of its
// units' 32 KB chunks; the eighth and later ones in shared memory): streaming
// them from L2 every iteration took 19000 of its 58000 cycles on the 200k figure,
// and an MMA whose A comes from tensor memory issues in 59 cycles instead of 165.
//
// Every wait is bounded, in global memory by a number of polls, on an mbarrier by
// the global timer and a number of polls; one that runs out marks the problem
// (ProbScal::fault) and the CTA leaves after its copies in flight have landed and its
// tensor memory is freed.  The host then leaves x where it was and solves that step
// again with the streamed kernels: a CTA needs a whole SM, so another stream's long
// kernel can keep a group's last CTAs from starting for longer than its first ones wait.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.h"
#include "pcg_dev.cuh"
#include "tc_dev.cuh"

namespace mfem {

namespace {

constexpr int kResStepB = 16 * 16 * 2;              // bytes of B per K step: 16 columns (hi, mid, lo, zeros)
constexpr int kResChunkB = kResStepB * kTcSteps;    // 4 KB
constexpr int kResTmemD = 32;                       // tensor-memory columns before the chunks of A: the accumulator
constexpr int kResTmemChunk = kTcKC / 2;            // columns a chunk takes (two BF16 a word)
constexpr int kResTmemChunks = 7;                   // chunks tensor memory holds (512 columns)
static_assert(kResTmemD + kResTmemChunks * kResTmemChunk <= 512, "tensor memory");
constexpr int kResMaxStages = 8;
constexpr int kResPolls = 1 << 18;                  // polls of a group barrier before it gives up (over 0.1 s of running time)
constexpr int kResStatic = 2048;                    // bound of the static shared memory below
constexpr int kResMaxThreads = kCoarseRows * kResUnits;   // one thread per row

// Scalars of one problem's recurrences; every CTA of the group keeps a copy,
// formed from the same totals.
struct ResState {
    double rho, alpha, beta, rr0, rr, tol2;
    int first, iter, maxit, state;
    double inv_rho, inv_alpha;   // FP32 path: 1 / rho and 1 / alpha, formed while the others update their rows
};

template <typename T>
struct ResShared {
    uint64_t full[kResMaxStages], empty[kResMaxStages], done, vals;
    uint32_t tmem;
    int fail;                       // a wait of this CTA ran out
    int gfail[2];                   // cluster: one of some CTA's did, in the set-up and in an iteration (tell_fail)
    int voff[kResUnits];            // byte offset of a unit's values in the value area, -1: read from global memory
    int slots[kResUnits];
    double wsum[kResMaxThreads / 32][3];
    ResState st;
    float ws[kResMaxThreads / 32][6];
    float qs[kResUnits][9];
};
static_assert(sizeof(ResShared<double>) <= kResStatic, "static shared memory");

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release(unsigned* p) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

// Exchange area of a cluster's CTA, at the same offset in each: the other CTAs
// write its copies of the inner-product partials and of r_c, and read its u.
constexpr int kExPart = 0;                                          // [256][3] doubles, by warp of 32 rows
constexpr int kExRc = kExPart + 256 * 3 * 8;                        // [16 kResUnits][6] floats
constexpr int kExU = kExRc + 16 * kResUnits * 6 * 4;                // [rows of the CTA][4]
template <typename T>
constexpr int kExW = kExU + kResMaxThreads * 4 * (int)sizeof(T);     // FP64: [3][64] products by component
template <typename T>
constexpr int kExBytes = kExW<T> + (sizeof(T) == 8 ? 2048 : 0);
static_assert(kExBytes<float> % 1024 == 0 && kExBytes<double> % 1024 == 0, "the A ring after it is aligned");

__device__ __forceinline__ uint32_t mapa(uint32_t addr, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void ld_cluster(uint32_t a, float (&q)[3]) {
    asm volatile("{\n\t.reg .f32 w;\n\tld.shared::cluster.v4.f32 {%0, %1, %2, w}, [%3];\n\t}\n"
                 : "=f"(q[0]), "=f"(q[1]), "=f"(q[2])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void ld_cluster(uint32_t a, double (&q)[3]) {
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(q[0]), "=d"(q[1]) : "r"(a) : "memory");
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(q[2]) : "r"(a + 16) : "memory");
}

// MMA with A in tensor memory
__device__ __forceinline__ void umma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The neighbour records of up to NB slots of a row (kNone: none): column ids into nb,
// or, in a cluster, shared-memory addresses (any but kNone, which is not aligned) of the
// owning CTA's u
constexpr int kNone = -1;
template <typename T, int NB, bool CLUSTER>
__device__ __forceinline__ void gather(const T* nb, const int (&c)[NB], T (&q)[NB][3]) {
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        q[i][0] = q[i][1] = q[i][2] = (T)0;
        if (c[i] == kNone) continue;
        if (CLUSTER) ld_cluster((uint32_t)c[i], q[i]);
        else ld4(nb + 4 * (size_t)c[i], q[i]);
    }
}
template <int NB>
__device__ __forceinline__ void load_cols(const int* cp, int k, int w, int (&c)[NB]) {
#pragma unroll
    for (int i = 0; i < NB; ++i) c[i] = k + i < w ? cp[32 * (k + i)] : kNone;
}
// w_i += those slots' products, in slot order
template <typename T, int NB>
__device__ __forceinline__ void products(const T* vp, const int (&c)[NB], const T (&q)[NB][3], T& a0, T& a1, T& a2) {
#pragma unroll
    for (int i = 0; i < NB; ++i)
        if (c[i] != kNone) {
            const T* vv = vp + 288 * i;
            a0 += vv[0] * q[i][0] + vv[32] * q[i][1] + vv[64] * q[i][2];
            a1 += vv[96] * q[i][0] + vv[128] * q[i][1] + vv[160] * q[i][2];
            a2 += vv[192] * q[i][0] + vv[224] * q[i][1] + vv[256] * q[i][2];
        }
}

// U: most units a CTA of this launch owns (registers: 255, 168 or 128 a thread
// for U = 4, 6, 8)
template <typename T, bool CLUSTER, int U>
__global__ void __launch_bounds__(kCoarseRows * U, 1)
    k_pcg_resident(const PcgDesc<T>* __restrict__ D, const ResJob* __restrict__ J, int n_probs, ResShape sh) {
    constexpr int kThreads = kCoarseRows * U;
    // neighbour records in flight a thread: a whole row's where the registers allow
    constexpr int NB = sizeof(T) == 4 ? (U <= 6 ? 16 : 8) : (U <= 4 ? 8 : 4);
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ ResShared<T> S;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int p = 0;
    {
        int hi = n_probs - 1;
        while (p < hi) {
            const int mid = (p + hi + 1) >> 1;
            if (J[mid].cta0 <= (int)blockIdx.x) p = mid;
            else hi = mid - 1;
        }
    }
    const PcgDesc<T>& d = D[p];
    const ResJob job = J[p];
    const int rank = (int)blockIdx.x - job.cta0, G = job.ncta;
    ProbScal* sc = d.sc;
    if (sc->state != kActive) return;   // the same for the whole group: its state is written only after every CTA's last barrier
    const bool coarse = d.coarse != 0;
    const int n = d.n_rows, N = d.coarse_n;
    const int ashift = coarse ? d.agg_shift - 6 : 0;   // units per aggregate (log2)
    const size_t np = npad32(n);

    // this CTA's units u0 .. u0 + nu - 1; the last CTAs, which have no coarse unit
    // when there are fewer of those than CTAs, take the remainder
    const int n_units = (n + kCoarseRows - 1) / kCoarseRows;
    const int u_rem = G - n_units % G;
    const int u0 = (n_units / G) * rank + max(0, rank - u_rem), nu = n_units / G + (rank >= u_rem ? 1 : 0);
    const int ul = t / kCoarseRows, row = (u0 + ul) * kCoarseRows + (t & (kCoarseRows - 1));
    const bool valid = ul < nu && row < n;

    // coarse units: part q of the K range of row block rb
    const int nkc = coarse ? coarse_chunks(N) : 0, c_per = coarse ? coarse_part_chunks(N) : 1;
    const int nq = coarse ? (nkc + c_per - 1) / c_per : 0, n_cu = coarse ? row_blocks(N) * nq : 0;
    const int ld_e = coarse_ld(N);
    constexpr int kEx = CLUSTER ? kExBytes<T> : 0;
    unsigned char* ring = smem + kEx;
    unsigned char* bmem = ring + (size_t)sh.stages * kFuChunkA;
    const bool has_cu = rank < n_cu;
    unsigned char* vmem = has_cu ? bmem + (size_t)sh.b_chunks * kResChunkB : ring;
    const int v_bytes = has_cu ? sh.v_bytes : sh.smem - kEx;

    // ---- set-up: barriers, the unit values that fit, the first chunks of A
    if (t == 0) {
        for (int i = 0; i < kResMaxStages; ++i) {
            mbar_init(&S.full[i], 1);
            mbar_init(&S.empty[i], 1);
        }
        mbar_init(&S.done, 1);
        mbar_init(&S.vals, 1);
        S.fail = 0;
        S.gfail[0] = S.gfail[1] = 0;
        S.st = ResState{sc->rho, sc->alpha, sc->beta, sc->rr0, sc->rr, sc->tol2, sc->first, sc->iter, sc->maxit,
                        sc->state, 0.0, 0.0};
        if (!S.st.first) {
            S.st.inv_rho = 1.0 / S.st.rho;
            S.st.inv_alpha = 1.0 / S.st.alpha;
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (t < kResUnits) {
        int s = 0;
        if (t < nu) {
            const int n_slices = (n + 31) >> 5, s0 = 2 * (u0 + t);
            s = d.slice_ptr[min(n_slices, s0 + 2)] - d.slice_ptr[s0];
        }
        S.slots[t] = s;
    }
    for (int i = t; i < kResUnits * 9; i += kThreads) {
        const int a = (u0 + i / 9) >> ashift;
        S.qs[i / 9][i % 9] = coarse && i / 9 < nu ? d.aggq[9 * a + i % 9] : 0.f;
    }
    if (has_cu)
        for (int i = t; i < sh.b_chunks * kResChunkB / 16; i += kThreads)
            reinterpret_cast<uint4*>(bmem)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    // chunks of A of this CTA's units, in order: the first kResTmemChunks stay in
    // tensor memory, the others go through the shared-memory ring (and stay there
    // if it holds them all)
    auto chunks_of = [&](int cu) {
        const int c_lo = (cu % nq) * c_per;
        return min(nkc, c_lo + c_per) - c_lo;
    };
    auto chunk_ptr = [&](int cu, int c) {
        return reinterpret_cast<const unsigned char*>(job.Abf) +
               ((size_t)(cu / nq) * nkc + (cu % nq) * c_per + c) * kFuChunkA;
    };
    int n_a = 0;
    for (int cu = rank; cu < n_cu; cu += G) n_a += chunks_of(cu);
    const int n_tm = min(n_a, kResTmemChunks), n_ring = n_a - n_tm;
    const bool keep = n_ring <= sh.stages;
    const uint32_t tm_need = kResTmemD + n_tm * kResTmemChunk;
    const uint32_t tm_cols = tm_need <= 32 ? 32 : (tm_need <= 128 ? 128 : (tm_need <= 256 ? 256 : 512));
    int l_cu = rank, l_c = 0;            // the ring's next chunk (thread 0)
    long long loaded = 0, used = 0;
    auto ring_start = [&]() {            // first chunk past the ones in tensor memory
        l_cu = rank;
        l_c = n_tm;
        while (l_cu < n_cu && l_c >= chunks_of(l_cu)) {
            l_c -= chunks_of(l_cu);
            l_cu += G;
        }
    };
    auto load_next = [&]() {   // one more chunk into its stage (free by now)
        const int s = (int)(loaded % sh.stages);
        mbar_expect_tx(&S.full[s], kFuChunkA);
        bulk_g2s(ring + (size_t)s * kFuChunkA, chunk_ptr(l_cu, l_c), kFuChunkA, &S.full[s]);
        ++loaded;
        if (++l_c >= chunks_of(l_cu)) {
            l_c = 0;
            l_cu += G;
            if (l_cu >= n_cu) ring_start();
        }
    };
    if (t == 0) {
        int off = 0;
        uint32_t bytes = 0;
        for (int i = 0; i < kResUnits; ++i) {
            const int need = S.slots[i] * (9 * (int)sizeof(T) + 4);
            const bool fits = i < nu && off + need <= v_bytes;
            S.voff[i] = fits ? off : -1;
            if (fits) {
                off += need;
                bytes += need;
            }
        }
        if (bytes) {
            mbar_expect_tx(&S.vals, bytes);
            for (int i = 0; i < nu; ++i) {
                if (S.voff[i] < 0 || !S.slots[i]) continue;
                const size_t base = d.slice_ptr[2 * (u0 + i)];
                const uint32_t vb = S.slots[i] * 9 * (uint32_t)sizeof(T);
                bulk_g2s(vmem + S.voff[i], d.val + base * 9, vb, &S.vals);
                bulk_g2s(vmem + S.voff[i] + vb, d.col + base, S.slots[i] * 4u, &S.vals);
            }
        } else {
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&S.vals)) : "memory");
        }
        ring_start();
        for (int i = 0; i < n_ring && i < sh.stages; ++i) load_next();
    }
    if (has_cu && warp == 0) tmem_alloc(&S.tmem, tm_cols);

    // ---- the row's state
    T r[3] = {0, 0, 0}, pp[3] = {0, 0, 0}, ss[3] = {0, 0, 0}, dx[3] = {0, 0, 0}, zb[3] = {0, 0, 0}, di[kDinv];
    float4 off = make_float4(0.f, 0.f, 0.f, 0.f);
    int base = 0, w = 0;
#pragma unroll
    for (int e = 0; e < kDinv; ++e) di[e] = 0;
    if (valid) {
        ld3(d.rec, np, kRecR, row, r);
        ld3(d.rec, np, kRecP, row, pp);
        ld3(d.rec, np, kRecS, row, ss);
        ld3(d.rec, np, kRecDX, row, dx);
        ld3(d.rec, np, kRecZB, row, zb);
#pragma unroll
        for (int e = 0; e < kDinv; ++e) di[e] = d.dinv[e * np + row];
        if (coarse) off = d.crel[row];
        const int s = row >> 5;
        base = __ldg(d.slice_ptr + s);
        w = (__ldg(d.slice_ptr + s + 1) - base) >> 5;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = has_cu ? S.tmem : 0u;
    // chunks of A into tensor memory: lane = row, two consecutive columns of A a
    // word; a warp reaches the 32 lanes of its number mod 4
    if (has_cu) {
        const uint32_t lane0 = (uint32_t)((warp & 3) * 32) << 16;
        const int arow = (warp & 3) * 32 + lane;
        int i = 0;
        for (int cu = rank; cu < n_cu; cu += G)
            for (int c = 0, nch = chunks_of(cu); c < nch && i < n_tm; ++c, ++i) {
                const unsigned char* src = chunk_ptr(cu, c);
#pragma unroll 4
                for (int k = warp >> 2; k < kTcSteps; k += kThreads / 128) {
                    const uint4 x = __ldg(reinterpret_cast<const uint4*>(src + a_piece(arow, 2 * k)));
                    const uint4 y = __ldg(reinterpret_cast<const uint4*>(src + a_piece(arow, 2 * k + 1)));
                    tmem_st(tmem + lane0 + kResTmemD + i * kResTmemChunk + 8 * k, x, y);
                }
            }
        tmem_st_wait();
        tc_fence_before();
    }
    const int voff = ul < kResUnits ? S.voff[ul] : -1;
    // the row's first slot in the value area (bytes), if its unit is there
    const bool in_smem = valid && voff >= 0;
    int v_at = 0, c_at = 0;
    if (in_smem) {
        const int rel = base - __ldg(d.slice_ptr + 2 * (u0 + ul));   // slots of the unit before the row's slice
        v_at = voff + (rel * 9 + lane) * (int)sizeof(T);
        c_at = voff + S.slots[ul] * 9 * (int)sizeof(T) + (rel + lane) * 4;
    }
    const T* vg = d.val + (size_t)base * 9 + lane;
    const int* cg = d.col + base + lane;
    if (!mbar_wait(&S.vals, 0)) S.fail = 1;
    const bool landed = !__syncthreads_or(S.fail);

    double* xpart = reinterpret_cast<double*>(smem + kExPart);   // cluster: every warp's inner products
    float* xrc = reinterpret_cast<float*>(smem + kExRc);         // cluster: r_c by unit
    T* xu = reinterpret_cast<T*>(smem + kExU);                   // cluster: u of this CTA's rows
    // cluster: shared-memory address of a row's u in its CTA
    const int q_units = n_units / G;
    auto u_address = [&](int c) {
        const int unit = c >> 6;
        const int rk = unit < q_units * u_rem ? unit / max(1, q_units) : u_rem + (unit - q_units * u_rem) / (q_units + 1);
        const int local = (unit - q_units * rk - max(0, rk - u_rem)) * kCoarseRows + (c & (kCoarseRows - 1));
        return (int)mapa(smem_u32(xu) + local * 4 * (int)sizeof(T), rk);
    };
    if (CLUSTER) {
        if (landed && in_smem)   // column ids -> addresses, once
            for (int k = 0; k < w; ++k) {
                int* cp = reinterpret_cast<int*>(vmem + c_at) + 32 * k;
                if (*cp != kNone) *cp = u_address(*cp);
            }
        // the other CTAs' copies start from this launch's residual
        if (coarse && has_cu)
            for (int i = t; i < 6 * n_units; i += kThreads) xrc[i] = d.rcp[i];
        __syncthreads();
    }
    int c0[NB];   // the first slots' column ids
    load_cols(in_smem ? reinterpret_cast<const int*>(vmem + c_at) : cg, 0, landed ? w : 0, c0);
    if (CLUSTER && !in_smem)
#pragma unroll
        for (int i = 0; i < NB; ++i)
            if (c0[i] != kNone) c0[i] = u_address(c0[i]);
    // A failed wait of a cluster's CTA is told to all of them before a barrier and looked
    // at after that barrier only, so that all leave together and none reads the memory
    // of one that has left.  The word of the set-up is written before the set-up's last
    // barrier alone; that of the iterations before the coarse product's barrier, with two
    // barriers more between a look at it and the next write.  (A look after any other
    // barrier could meet the next iteration's write in some threads and not in others.)
    // S.fail is written by its own CTA alone, between block barriers.
    auto tell_fail = [&](int k) {
        if (CLUSTER && t == 0 && S.fail)
            for (int rk = 0; rk < G; ++rk)
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(mapa(smem_u32(&S.gfail[k]), rk)), "r"(1) : "memory");
    };
    if (CLUSTER) {   // every CTA of the cluster runs before the first remote access
        cluster_arrive();
        cluster_wait();
        tell_fail(0);
        cluster_arrive();
        cluster_wait();
    }
    const bool go = CLUSTER ? !S.gfail[0] : landed;
    // FP64, one unit a CTA: an FP64 instruction holds a scheduler for 64 cycles and
    // the unit's two warps would use two of the four, so six warps form the product,
    // a component of w each (bar of 1536 tets: an iteration 19.8 -> 16.4 us)
    const bool by_comp = sizeof(T) == 8 && CLUSTER && nu == 1 && S.voff[0] >= 0;
    int hw = 0, hv = 0, hc = 0;   // the helped row's slots, first value and column id
    if (by_comp && t < 3 * kCoarseRows && u0 * kCoarseRows + (t & 63) < n) {
        const int s = 2 * u0 + ((t >> 5) & 1), b0 = __ldg(d.slice_ptr + 2 * u0), b = __ldg(d.slice_ptr + s);
        hw = (__ldg(d.slice_ptr + s + 1) - b) >> 5;
        hv = S.voff[0] + ((b - b0) * 9 + lane) * (int)sizeof(T);
        hc = S.voff[0] + S.slots[0] * 9 * (int)sizeof(T) + (b - b0 + lane) * 4;
    }

    unsigned bar_n = 0;
    uint32_t done_ph = 0;
    // every write of the group's CTAs before arrive() is visible to their reads after wait()
    auto arrive = [&]() {
        if (CLUSTER) {
            cluster_arrive();
            return;
        }
        __syncthreads();
        ++bar_n;
        if (t == 0) red_release(job.bar);
    };
    auto wait = [&]() {
        if (CLUSTER) {
            cluster_wait();
            return;
        }
        if (t == 0) {
            const unsigned target = bar_n * (unsigned)G;
            for (int i = 0; ld_acquire(job.bar) < target; ++i)
                if (i >= kResPolls) {
                    S.fail = 1;
                    break;
                }
        }
        __syncthreads();
    };

    bool active = true;
    for (int it = 0; go && it < sh.iters; ++it) {
        T u[3] = {zb[0], zb[1], zb[2]};
        if (it == sh.expire) {   // tests
            __syncthreads();
            if (t == 0 && rank == G - 1) S.fail = 1;
            __syncthreads();
        }
        if (coarse) {
            // ---- coarse product: this CTA's units
            int a_at = 0;   // chunks issued this iteration (thread 0)
            for (int cu = rank; cu < n_cu; cu += G) {
                const int rb = cu / nq, q = cu % nq, c_lo = q * c_per, nch = chunks_of(cu);
                // B: r_c of the part's columns as three BF16 rows, eight columns (one core-matrix row) a thread
                for (int g = t; g < nch * (kTcKC / 8); g += kThreads) {
                    const int k = c_lo * kTcKC + 8 * g;
                    float v[8];
                    const float* rc = CLUSTER ? xrc : d.rcp;
                    if (ashift == 0) {
                        if (k + 7 < N) {
                            const float4 x = *reinterpret_cast<const float4*>(rc + k);
                            const float4 y = *reinterpret_cast<const float4*>(rc + k + 4);
                            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
                            v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
                        } else {
#pragma unroll
                            for (int e = 0; e < 8; ++e) v[e] = k + e < N ? rc[k + e] : 0.f;
                        }
                    } else {
                        for (int e = 0; e < 8; ++e) {
                            float s = 0.f;
                            if (k + e < N) {
                                const int a = (k + e) / 6, comp = (k + e) - 6 * a, e1 = min(n_units, (a + 1) << ashift);
                                for (int x = a << ashift; x < e1; ++x) s += rc[6 * (size_t)x + comp];
                            }
                            v[e] = s;
                        }
                    }
                    uint32_t h[4], m[4], l[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        uint32_t hh[2], mm[2], ll[2];
#pragma unroll
                        for (int f = 0; f < 2; ++f) {
                            const float x = v[2 * e + f];
                            const __nv_bfloat16 b0 = __float2bfloat16_rn(x);
                            const float r1 = x - __bfloat162float(b0);
                            const __nv_bfloat16 b1 = __float2bfloat16_rn(r1);
                            const __nv_bfloat16 b2 = __float2bfloat16_rn(r1 - __bfloat162float(b1));
                            hh[f] = __bfloat16_as_ushort(b0);
                            mm[f] = __bfloat16_as_ushort(b1);
                            ll[f] = __bfloat16_as_ushort(b2);
                        }
                        h[e] = hh[0] | (hh[1] << 16);
                        m[e] = mm[0] | (mm[1] << 16);
                        l[e] = ll[0] | (ll[1] << 16);
                    }
                    unsigned char* o = bmem + (g >> 4) * kResChunkB + ((g & 15) >> 1) * kResStepB + (g & 1) * 128;
                    *reinterpret_cast<uint4*>(o) = make_uint4(h[0], h[1], h[2], h[3]);
                    *reinterpret_cast<uint4*>(o + 16) = make_uint4(m[0], m[1], m[2], m[3]);
                    *reinterpret_cast<uint4*>(o + 32) = make_uint4(l[0], l[1], l[2], l[3]);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncthreads();
                if (t == 0) {
                    constexpr uint32_t idesc = umma_idesc_bf16(kTcM, 16);
                    const uint32_t a_base = smem_u32(ring), b_base = smem_u32(bmem);
                    tc_fence_after();
                    for (int c = 0; c < nch; ++c, ++a_at) {
                        const uint32_t b0 = b_base + c * kResChunkB;
                        if (a_at < n_tm) {
                            const uint32_t ta = tmem + kResTmemD + a_at * kResTmemChunk;
#pragma unroll
                            for (int k = 0; k < kTcSteps; ++k)
                                umma_bf16_ta(tmem, ta + 8 * k, umma_desc(b0 + k * kResStepB, 128, 256), idesc,
                                             (c > 0 || k > 0) ? 1u : 0u);
                            continue;
                        }
                        const int s = (int)((keep ? a_at - n_tm : used) % sh.stages);
                        if (!mbar_wait(&S.full[s], keep ? 0u : (uint32_t)(used / sh.stages) & 1u)) {
                            S.fail = 1;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t a0 = a_base + s * kFuChunkA;
#pragma unroll
                        for (int k = 0; k < kTcSteps; ++k)
                            umma_bf16(tmem, umma_desc_sw128(a0 + a_step(k)),
                                      umma_desc(b0 + k * kResStepB, 128, 256), idesc, (c > 0 || k > 0) ? 1u : 0u);
                        if (keep) continue;
                        umma_commit(&S.empty[s]);
                        // refill the stage before this one, whose products were issued a chunk ago
                        if (loaded < used + sh.stages) {
                            const long long prev = loaded - sh.stages;
                            if (!mbar_wait(&S.empty[prev % sh.stages], (uint32_t)(prev / sh.stages) & 1u)) {
                                S.fail = 1;
                                break;
                            }
                            load_next();
                        }
                        ++used;
                    }
                    umma_commit(&S.done);
                }
                if (!mbar_wait(&S.done, done_ph)) S.fail = 1;
                done_ph ^= 1u;
                tc_fence_after();
                if (warp < kTcM / 32) {
                    float v[4];
                    tmem_ld(tmem + ((uint32_t)(warp * 32) << 16), v);
                    const int lr = warp * 32 + lane, er = 6 * kFuAggsBlk * rb + lr;
                    if (lr < 6 * kFuAggsBlk && er < N) job.epart[(size_t)q * ld_e + er] = (v[0] + v[1]) + v[2];
                }
                tc_fence_before();
                if (__syncthreads_or(S.fail)) break;
            }
            // the last chunk's stage, for the next iteration
            if (t == 0 && !keep && !S.fail)
                while (loaded < used + sh.stages) {
                    const long long prev = loaded - sh.stages;
                    if (!mbar_wait(&S.empty[prev % sh.stages], (uint32_t)(prev / sh.stages) & 1u)) {
                        S.fail = 1;
                        break;
                    }
                    load_next();
                }
            tell_fail(1);
            arrive();
            wait();
            if (CLUSTER ? S.gfail[1] : S.fail) break;
            // ---- u = zb + Q_a P_i e_a, the parts of e_a added in part order
            float ev = 0.f;
            if (lane < 6 && ul < nu) {
                const int a = (u0 + ul) >> ashift;
                const float* ep = job.epart + 6 * a + lane;
                float x[kFuSplit];
#pragma unroll
                for (int q = 0; q < kFuSplit; ++q) x[q] = q < nq ? ep[(size_t)q * ld_e] : 0.f;
#pragma unroll
                for (int q = 0; q < kFuSplit; ++q) ev += x[q];
            }
            const float e0 = __shfl_sync(0xffffffffu, ev, 0), e1 = __shfl_sync(0xffffffffu, ev, 1);
            const float e2 = __shfl_sync(0xffffffffu, ev, 2), e3 = __shfl_sync(0xffffffffu, ev, 3);
            const float e4 = __shfl_sync(0xffffffffu, ev, 4), e5 = __shfl_sync(0xffffffffu, ev, 5);
            if (off.w != 0.f) {
                const float l0 = e0 + (e4 * off.z - e5 * off.y);
                const float l1 = e1 + (e5 * off.x - e3 * off.z);
                const float l2 = e2 + (e3 * off.y - e4 * off.x);
                const float* Q = S.qs[ul];
#pragma unroll
                for (int i = 0; i < 3; ++i) u[i] += (T)(Q[3 * i] * l0 + Q[3 * i + 1] * l1 + Q[3 * i + 2] * l2);
            }
        }
        if (valid) st4(CLUSTER ? xu + 4 * t : d.nb + 4 * (size_t)row, u[0], u[1], u[2]);
        arrive();
        if (!valid) u[0] = u[1] = u[2] = 0;
        const Partial<T> d0 = dot3_partial(r[0], r[1], r[2], u[0], u[1], u[2]);
        const Partial<T> d2 = dot3_partial(r[0], r[1], r[2], r[0], r[1], r[2]);
        wait();
        if (!CLUSTER && S.fail) break;
        // ---- w = K u
        T a0 = 0, a1 = 0, a2 = 0;
        if (by_comp) {
            T* xw = reinterpret_cast<T*>(smem + kExW<T>);
            if (t < 3 * kCoarseRows) {
                const int comp = t / kCoarseRows;
                const T* vp = reinterpret_cast<const T*>(vmem + hv) + 96 * comp;
                T a = 0;
                for (int k = 0; k < hw; k += 4) {
                    int c[4];
                    T q[4][3];
                    load_cols(reinterpret_cast<const int*>(vmem + hc), k, hw, c);
                    gather<T, 4, CLUSTER>(d.nb, c, q);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (c[i] != kNone) {
                            const T* vv = vp + 288 * (k + i);
                            a += vv[0] * q[i][0] + vv[32] * q[i][1] + vv[64] * q[i][2];
                        }
                }
                xw[t] = a;
            }
            __syncthreads();
            if (valid) {
                a0 = xw[t];
                a1 = xw[kCoarseRows + t];
                a2 = xw[2 * kCoarseRows + t];
            }
        } else {
            T q[NB][3];
            gather<T, NB, CLUSTER>(d.nb, c0, q);
            if (in_smem) {
                products<T, NB>(reinterpret_cast<const T*>(vmem + v_at), c0, q, a0, a1, a2);
                for (int k = NB; k < w; k += NB) {
                    int c[NB];
                    load_cols(reinterpret_cast<const int*>(vmem + c_at), k, w, c);
                    gather<T, NB, CLUSTER>(d.nb, c, q);
                    products<T, NB>(reinterpret_cast<const T*>(vmem + v_at) + 288 * k, c, q, a0, a1, a2);
                }
            } else {
                products<T, NB>(vg, c0, q, a0, a1, a2);
                for (int k = NB; k < w; k += NB) {
                    int c[NB];
                    load_cols(cg, k, w, c);
                    if (CLUSTER)
#pragma unroll
                        for (int i = 0; i < NB; ++i)
                            if (c[i] != kNone) c[i] = u_address(c[i]);
                    gather<T, NB, CLUSTER>(d.nb, c, q);
                    products<T, NB>(vg + 288 * (size_t)k, c, q, a0, a1, a2);
                }
            }
        }
        {
            const double v = warp_sums3(d0, dot3_wu(a0, a1, a2, u[0], u[1], u[2]), d2);
            if (lane < 3) S.wsum[warp][lane] = v;
        }
        __syncthreads();
        // partials: FP64 one per warp (32 rows), which the totals add in the
        // streamed kernel's order; FP32 one per warp in a cluster and one per CTA of a larger group (FP64 sums of float-float
        // warp sums: their order shows in the last bits of alpha and beta only,
        // which are rounded to FP32).  An FP64 instruction takes a scheduler 64
        // cycles, so few warps do few of them, a value each.
        if (CLUSTER) {   // to every CTA of the cluster
            for (int i = t; i < 6 * nu * G; i += kThreads) {
                const int k = i % (6 * nu), w0 = 2 * u0 + k / 3;
                if (32 * w0 < n) st_cluster(mapa(smem_u32(xpart + 3 * w0 + k % 3), i / (6 * nu)), S.wsum[k / 3][k % 3]);
            }
        } else if (sizeof(T) == 8) {
            if (t < 6 * nu && 32 * (2 * u0 + t / 3) < n) d.part[4 * (size_t)(2 * u0 + t / 3) + t % 3] = S.wsum[t / 3][t % 3];
        } else if (warp < 3) {
            double x = lane < 2 * U ? S.wsum[lane & 15][warp] : 0.0;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (lane == 0) d.part[4 * (size_t)rank + warp] = x;
        }
        arrive();
        wait();
        if (!CLUSTER && S.fail) break;
        double tot[3] = {0.0, 0.0, 0.0};   // valid in thread 0
        if (sizeof(T) == 8) {
            const int nw = sh.rtile / 32, n_tiles = (n + sh.rtile - 1) / sh.rtile, n_warps = (n + 31) / 32;
            for (int x = t; t < sh.rtile && x < n_tiles; x += sh.rtile)
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    double v[8];
#pragma unroll
                    for (int y = 0; y < 8; ++y)
                        v[y] = y >= nw || x * nw + y >= n_warps ? 0.0
                               : CLUSTER                        ? xpart[3 * (x * nw + y) + i]
                                                                : d.part[4 * (size_t)(x * nw + y) + i];
                    tot[i] += ((v[0] + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));
                }
            if (warp < nw) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int i = 0; i < 3; ++i) tot[i] += __shfl_xor_sync(0xffffffffu, tot[i], o);
                if (lane == 0)
#pragma unroll
                    for (int i = 0; i < 3; ++i) S.wsum[warp][i] = tot[i];
            }
            __syncthreads();
            if (warp == 0) {
#pragma unroll
                for (int i = 0; i < 3; ++i) tot[i] = lane < nw ? S.wsum[lane & 7][i] : 0.0;
#pragma unroll
                for (int o = 4; o > 0; o >>= 1)
#pragma unroll
                    for (int i = 0; i < 3; ++i) tot[i] += __shfl_xor_sync(0xffffffffu, tot[i], o);
            }
        } else {
            if (warp < 3) {   // warp i sums value i
                const int n_part = CLUSTER ? (n + 31) / 32 : G;   // at most 256
                double x[8], s = 0.0;
#pragma unroll
                for (int j = 0; j < 8; ++j)   // every load first
                    x[j] = lane + 32 * j >= n_part ? 0.0
                           : CLUSTER                ? xpart[3 * (lane + 32 * j) + warp]
                                                    : d.part[4 * (size_t)(lane + 32 * j) + warp];
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (32 * j < n_part) s += x[j];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) S.wsum[0][warp] = s;
            }
            __syncthreads();
            if (t == 0)
#pragma unroll
                for (int i = 0; i < 3; ++i) tot[i] = S.wsum[0][i];
        }
        if (t == 0) {
            ResState& q = S.st;
            const double gamma = tot[0], delta = tot[1];
            q.rr = tot[2];
            if (!(tot[2] > q.tol2 * q.rr0)) {
                q.state = kConverged;
            } else if (q.iter >= q.maxit) {
                q.state = kMaxIter;
            } else {
                double beta = 0.0, den = delta;
                if (!q.first) {
                    if (sizeof(T) == 8) {
                        beta = gamma / q.rho;
                        den = delta - beta * gamma / q.alpha;
                    } else {
                        beta = gamma * q.inv_rho;
                        den = delta - beta * gamma * q.inv_alpha;
                    }
                }
                if (gamma > 0.0 && den > 0.0 && isfinite(gamma) && isfinite(den)) {
                    q.alpha = gamma / den;
                    q.beta = beta;
                    q.rho = gamma;
                    q.first = 0;
                    q.iter = q.iter + 1;
                } else {
                    q.alpha = 0.0;
                    q.beta = 0.0;
                    q.state = kConverged;
                }
            }
        }
        __syncthreads();
        if (S.st.state != kActive) {
            active = false;
            break;
        }
        // ---- the update and the restriction of the new residual
        const T alpha = (T)S.st.alpha, beta = (T)S.st.beta;
        const T ww[3] = {a0, a1, a2};
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            pp[i] = fma(beta, pp[i], u[i]);
            ss[i] = fma(beta, ss[i], ww[i]);
            dx[i] = fma(alpha, pp[i], dx[i]);
            r[i] = fma(-alpha, ss[i], r[i]);
        }
        sym_product(di, r, zb);
        if (coarse) {
            float y[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            if (off.w != 0.f) {
                const float r32[3] = {(float)r[0], (float)r[1], (float)r[2]};
                const float* Qt = S.qs[ul];
                const float q0 = Qt[0] * r32[0] + Qt[3] * r32[1] + Qt[6] * r32[2];
                const float q1 = Qt[1] * r32[0] + Qt[4] * r32[1] + Qt[7] * r32[2];
                const float q2 = Qt[2] * r32[0] + Qt[5] * r32[1] + Qt[8] * r32[2];
                y[0] = q0;
                y[1] = q1;
                y[2] = q2;
                y[3] = off.y * q2 - off.z * q1;
                y[4] = off.z * q0 - off.x * q2;
                y[5] = off.x * q1 - off.y * q0;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int c = 0; c < 6; ++c) y[c] += __shfl_xor_sync(0xffffffffu, y[c], o);
            if (lane == 0)
#pragma unroll
                for (int c = 0; c < 6; ++c) S.ws[warp][c] = y[c];
            __syncthreads();
            if (t < 6 * nu) {
                const int x = t / 6, c = t - 6 * x;
                const float v = S.ws[2 * x][c] + S.ws[2 * x + 1][c];
                d.rcp[6 * (size_t)(u0 + x) + c] = v;
                if (CLUSTER)   // to the CTAs that multiply it
                    for (int rk = 0; rk < min(G, n_cu); ++rk) st_cluster(mapa(smem_u32(xrc + 6 * (u0 + x) + c), rk), v);
            }
            arrive();
        }
        if (sizeof(T) == 4 && t == kThreads - 32) {
            S.st.inv_rho = 1.0 / S.st.rho;
            S.st.inv_alpha = 1.0 / S.st.alpha;
        }
        if (coarse) {
            wait();
            if (!CLUSTER && S.fail) break;
        }
    }

    __syncthreads();   // the reciprocals of the last coefficients
    // ---- write back: the increment; the other vectors only if the solve goes on
    if (valid) {
        st3(d.rec, np, kRecDX, row, dx[0], dx[1], dx[2]);
        if (active) {
            st3(d.rec, np, kRecR, row, r[0], r[1], r[2]);
            st3(d.rec, np, kRecP, row, pp[0], pp[1], pp[2]);
            st3(d.rec, np, kRecS, row, ss[0], ss[1], ss[2]);
            st3(d.rec, np, kRecZB, row, zb[0], zb[1], zb[2]);
            // a served solve may go on in the streamed kernels: what their update leaves
            if (!coarse) st4(d.nb + 4 * (size_t)row, zb[0], zb[1], zb[2]);
        }
    }
    if (active && d.bunit && t < 6 * nu) {   // ... the residual's B operand among it
        const int k = 6 * u0 + t;
        if (k < N) coarse_b_store(d.bunit, d.bslot % kCoarseGroupSlots, k, d.rcp[k]);
    }
    if (t == 0) {
        // a word of its own: one block may fail and another of its group not
        if (S.fail || S.gfail[0] || S.gfail[1]) {
            sc->fault = 1u;
        } else if (rank == 0) {
            sc->rho = S.st.rho;
            sc->alpha = S.st.alpha;
            sc->beta = S.st.beta;
            if (sizeof(T) == 4) {
                sc->inv_rho = S.st.inv_rho;
                sc->inv_alpha = S.st.inv_alpha;
            }
            sc->alpha_f = (float)S.st.alpha;
            sc->beta_f = (float)S.st.beta;
            sc->rr = S.st.rr;
            sc->first = S.st.first;
            sc->iter = S.st.iter;
            sc->state = S.st.state;
        }
        // copies in flight land, and after a failed wait the matrix values and the products
        // issued last as well, before the memory is released (each bounded again)
        if (S.fail) {
            mbar_wait(&S.vals, 0);
            mbar_wait(&S.done, done_ph ^ 1u);
        }
        if (keep) {
            for (int i = 0; i < n_ring; ++i) mbar_wait(&S.full[i], 0);
        } else {
            for (long long i = used; i < loaded; ++i)
                mbar_wait(&S.full[i % sh.stages], (uint32_t)(i / sh.stages) & 1u);
        }
    }
    __syncthreads();
    if (has_cu && warp == 0) tmem_free(tmem, tm_cols);
}

template <typename T, bool CLUSTER, int U>
cudaError_t res_attr() {
    cudaError_t e =
        cudaFuncSetAttribute(k_pcg_resident<T, CLUSTER, U>, cudaFuncAttributeMaxDynamicSharedMemorySize, res_smem_max());
    if (e == cudaSuccess && CLUSTER)
        e = cudaFuncSetAttribute(k_pcg_resident<T, CLUSTER, U>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

void res_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, const ResShape& sh, cudaStream_t s) {
    cfg = cudaLaunchConfig_t{};
    if (sh.cluster > 0) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = sh.cluster;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
    } else {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    }
    cfg.gridDim = dim3(sh.grid);
    cfg.blockDim = dim3(kCoarseRows * sh.units);
    cfg.dynamicSmemBytes = sh.smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

}  // namespace

int res_tmem_chunks() { return kResTmemChunks; }
int res_smem_exchange(bool fp64) { return fp64 ? kExBytes<double> : kExBytes<float>; }
int res_smem_max() { return 227 * 1024 - kResStatic; }
int res_smem_coarse(int stages, int b_chunks) { return stages * kFuChunkA + b_chunks * kResChunkB; }
int res_part_chunks(int N) { return coarse_part_chunks(N); }
int res_coarse_units(int N) {
    const int nkc = coarse_chunks(N), c_per = coarse_part_chunks(N);
    return row_blocks(N) * ((nkc + c_per - 1) / c_per);
}

cudaError_t res_init(ResLimits& lim) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&lim.sms, cudaDevAttrMultiProcessorCount, dev);
#define MFEM_RES_ATTR(T, U)                                   \
    if (e == cudaSuccess) e = res_attr<T, true, U>();         \
    if (e == cudaSuccess) e = res_attr<T, false, U>();
    MFEM_RES_ATTR(float, 4)
    MFEM_RES_ATTR(float, 6)
    MFEM_RES_ATTR(float, 8)
    MFEM_RES_ATTR(double, 4)
    MFEM_RES_ATTR(double, 6)
    MFEM_RES_ATTR(double, 8)
#undef MFEM_RES_ATTR
    if (e != cudaSuccess) return e;
    for (int i = 0, c = 1; i < kResClusterSizes; ++i, c *= 2) {   // clusters of 1, 2, 4, 8, 16 CTAs resident at once
        ResShape sh{};
        sh.grid = c;
        sh.cluster = c;
        sh.units = kResUnits;
        sh.smem = res_smem_max();
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[1];
        res_config(cfg, attr, sh, nullptr);
        int nc = 0;   // one CTA an SM in every variant (shared memory)
        if (cudaOccupancyMaxActiveClusters(&nc, k_pcg_resident<double, true, kResUnits>, &cfg) != cudaSuccess) nc = 0;
        cudaGetLastError();
        lim.clusters[i] = nc;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_pcg_resident(const PcgDesc<T>* descs, const ResJob* jobs, int n_probs, const ResShape& sh,
                                cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    res_config(cfg, attr, sh, s);
#define MFEM_RES_CASE(UN)                                                                                           \
    if (sh.units == UN)                                                                                             \
        return sh.cluster > 0 ? cudaLaunchKernelEx(&cfg, k_pcg_resident<T, true, UN>, descs, jobs, n_probs, sh)     \
                              : cudaLaunchKernelEx(&cfg, k_pcg_resident<T, false, UN>, descs, jobs, n_probs, sh);
    MFEM_RES_CASE(4)
    MFEM_RES_CASE(6)
    MFEM_RES_CASE(8)
#undef MFEM_RES_CASE
    return cudaErrorInvalidValue;
}

template cudaError_t launch_pcg_resident<float>(const PcgDesc<float>*, const ResJob*, int, const ResShape&, cudaStream_t);
template cudaError_t launch_pcg_resident<double>(const PcgDesc<double>*, const ResJob*, int, const ResShape&,
                                                 cudaStream_t);

}  // namespace mfem
