// ews_arith.cuh -- the per-cell arithmetic of the scheme with every rounding
// written out (no operation is left to the compiler to contract), so that
// kernels that visit the cells in different orders -- the z-marching passes
// at every tile shape, and the resident time loop -- store the same bits.
#pragma once
#include "ews_internal.cuh"

namespace ews {
namespace ar {

// Eq. 4 difference of the four samples a..d (the inner pair is b, c).
__device__ __forceinline__ float d4(float c1, float c2, float a, float b, float c, float d) {
    return __fmaf_rn(c2, __fsub_rn(d, a), __fmul_rn(c1, __fsub_rn(c, b)));
}
__device__ __forceinline__ float sum3(float a, float b, float c) {
    return __fadd_rn(__fadd_rn(a, b), c);
}
// psi = b psi + a d; d += psi (one C-PML term).
__device__ __forceinline__ void pml(float& p, float a, float b, float& d) {
    p = __fmaf_rn(b, p, __fmul_rn(a, d));
    d = __fadd_rn(d, p);
}
// v + (dt b) (d1 + d2 + d3), Eq. 1.
__device__ __forceinline__ float vnew(float v, float dto, float b, float d1, float d2, float d3) {
    return __fmaf_rn(__fmul_rn(dto, b), sum3(d1, d2, d3), v);
}
// Normal stress s + dt ((lambda + 2 mu) e0 + lambda (e1 + e2)), Eq. 2/3.
__device__ __forceinline__ float snormal(float s, float dto, float l2m, float lam, float e0, float e1,
                                         float e2) {
    return __fmaf_rn(dto, __fmaf_rn(l2m, e0, __fmul_rn(lam, __fadd_rn(e1, e2))), s);
}
// Shear stress s + (dt mu) (d1 + d2).
__device__ __forceinline__ float sshear(float s, float dto, float mu, float d1, float d2) {
    return __fmaf_rn(__fmul_rn(dto, mu), __fadd_rn(d1, d2), s);
}
__device__ __forceinline__ float l2m(float lam, float mu) { return __fmaf_rn(2.0f, mu, lam); }
// Mean of four cells (shear points), and 2 / (r0 + r1) (buoyancy).
__device__ __forceinline__ float mean4(float a, float b, float c, float d) {
    return __fmul_rn(0.25f, __fadd_rn(__fadd_rn(__fadd_rn(a, b), c), d));
}
__device__ __forceinline__ float harm4(float a, float b, float c, float d) {
    return 4.0f / (__fadd_rn(__fadd_rn(__fadd_rn(1.0f / a, 1.0f / b), 1.0f / c), 1.0f / d));
}
__device__ __forceinline__ float buoyancy(float r0, float r1) {
    return __fdividef(2.0f, __fadd_rn(r0, r1));
}
// Sponge gain of a cell from its axis profiles.
__device__ __forceinline__ float gain(float gx, float gy, float gz) {
    return __fmul_rn(__fmul_rn(gx, gz), gy);
}

}  // namespace ar
}  // namespace ews
