// Device helpers shared by the PCG kernels (k_pcg.cu, k_pcg_resident.cu): vector
// access, inner-product partials, step coefficients and the block-Jacobi product.
#pragma once

#include <cuda_runtime.h>

#include "dev.cuh"

namespace mfem {

// ---- vector access ------------------------------------------------------------
// 3-vectors stored as aligned 4-element groups (x, y, z, 0)
__device__ __forceinline__ void ld4(const float* p, float (&v)[3]) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
}

__device__ __forceinline__ void ld4(const double* p, double (&v)[3]) {
    const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
    v[0] = a.x;
    v[1] = a.y;
    v[2] = b.x;
}

__device__ __forceinline__ void st4(float* p, float a, float b, float c) {
    *reinterpret_cast<float4*>(p) = make_float4(a, b, c, 0.f);
}

__device__ __forceinline__ void st4(double* p, double a, double b, double c) {
    reinterpret_cast<double2*>(p)[0] = make_double2(a, b);
    reinterpret_cast<double2*>(p)[1] = make_double2(c, 0.0);
}

// Per-row contribution to an inner product and its warp sum: float-float in
// the FP32 path (no FP64 instructions until one conversion per warp), plain
// FP64 in the FP64 path.
template <typename T>
struct Partial;

template <>
struct Partial<float> {
    FF v;
    static __device__ __forceinline__ Partial zero() { return Partial{FF{0.f, 0.f}}; }
};

template <>
struct Partial<double> {
    double v;
    static __device__ __forceinline__ Partial zero() { return Partial{0.0}; }
};

__device__ __forceinline__ Partial<float> dot3_partial(float a0, float a1, float a2, float b0, float b1, float b2) {
    const float a[3] = {a0, a1, a2}, b[3] = {b0, b1, b2};
    return Partial<float>{ff_dot3(a, b)};
}

// FP64: the products' rounding order is written out, so that every kernel forms
// the same bits (a compiler contracts the same sum differently in different
// places): a2 b2 + (a1 b1 + a0 b0), the inner sum rounded once after a0 b0, and
// for (w, u) once after a1 b1.
__device__ __forceinline__ Partial<double> dot3_partial(double a0, double a1, double a2, double b0, double b1,
                                                        double b2) {
    return Partial<double>{fma(a2, b2, fma(a1, b1, a0 * b0))};
}
__device__ __forceinline__ Partial<double> dot3_wu(double a0, double a1, double a2, double b0, double b1, double b2) {
    return Partial<double>{fma(a2, b2, fma(a0, b0, a1 * b1))};
}
__device__ __forceinline__ Partial<float> dot3_wu(float a0, float a1, float a2, float b0, float b1, float b2) {
    return dot3_partial(a0, a1, a2, b0, b1, b2);
}

// The warp sums of three partials (fixed xor tree), value i in lane i (0
// elsewhere).  GB300 issues an FP64 instruction of a warp every 64 cycles, the
// FP32 <-> FP64 conversions among them, so the three float-float sums are
// widened by one instruction sequence, a value per lane, instead of three.
__device__ __forceinline__ double warp_sums3(Partial<float> a, Partial<float> b, Partial<float> c) {
    FF x = a.v, y = b.v, z = c.v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x = ff_add(x, FF{__shfl_xor_sync(0xffffffffu, x.hi, o), __shfl_xor_sync(0xffffffffu, x.lo, o)});
        y = ff_add(y, FF{__shfl_xor_sync(0xffffffffu, y.hi, o), __shfl_xor_sync(0xffffffffu, y.lo, o)});
        z = ff_add(z, FF{__shfl_xor_sync(0xffffffffu, z.hi, o), __shfl_xor_sync(0xffffffffu, z.lo, o)});
    }
    const int lane = threadIdx.x & 31;   // every lane holds the three sums
    const FF s = lane == 0 ? x : (lane == 1 ? y : z);
    return lane < 3 ? (double)s.hi + (double)s.lo : 0.0;
}
__device__ __forceinline__ double warp_sums3(Partial<double> a, Partial<double> b, Partial<double> c) {
    double x = a.v, y = b.v, z = c.v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
        z += __shfl_xor_sync(0xffffffffu, z, o);
    }
    const int lane = threadIdx.x & 31;
    return lane == 0 ? x : (lane == 1 ? y : (lane == 2 ? z : 0.0));
}

// Sum of NW (2, 4, 8 or 16) warps' values of one kind, v[w * 3]: the order of a
// shuffle tree over the warps.
template <int NW>
__device__ __forceinline__ double warps_sum(const double* v) {
    double x[NW];
#pragma unroll
    for (int w = 0; w < NW; ++w) x[w] = v[3 * w];
#pragma unroll
    for (int o = NW / 2; o > 0; o >>= 1)
#pragma unroll
        for (int w = 0; w < o; ++w) x[w] += x[w + o];
    return x[0];
}

// step coefficients in the kernel's precision
__device__ __forceinline__ void coeffs(const ProbScal* sc, float& a, float& b) {
    a = sc->alpha_f;
    b = sc->beta_f;
}
__device__ __forceinline__ void coeffs(const ProbScal* sc, double& a, double& b) {
    a = sc->alpha;
    b = sc->beta;
}

// z = M r, M symmetric with entries 00, 11, 22, 12, 02, 01
template <typename T>
__device__ __forceinline__ void sym_product(const T (&s)[kDinv], const T (&r)[3], T (&z)[3]) {
    const T m[9] = {s[0], s[5], s[4], s[5], s[1], s[3], s[4], s[3], s[2]};
#pragma unroll
    for (int i = 0; i < 3; ++i) z[i] = m[3 * i] * r[0] + m[3 * i + 1] * r[1] + m[3 * i + 2] * r[2];
}
// z_bj = D^{-1} r for one row: entry e of D^{-1} of every row stored contiguously
// (at di[e * np + row], np = npad32(n)), so a warp's load of one entry is one
// contiguous 32-row run
template <typename T>
__device__ __forceinline__ void apply_dinv(const T* __restrict__ di, size_t np, int row, const T (&r)[3], T (&z)[3]) {
    T m[kDinv];
#pragma unroll
    for (int e = 0; e < kDinv; ++e) m[e] = di[e * np + row];
    sym_product(m, r, z);
}

}  // namespace mfem
