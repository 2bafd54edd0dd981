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
    return __fmaf_rn(c1, __fsub_rn(c, b), __fmul_rn(c2, __fsub_rn(d, a)));
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
// 1 / x by rcp.approx.ftz (at most 1 ulp by the PTX manual; __fdividef is given
// to 2 ulp): a density is a normal number.
__device__ __forceinline__ float rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// Mean of four cells (shear points), and 2 / (r0 + r1) (buoyancy).
__device__ __forceinline__ float mean4(float a, float b, float c, float d) {
    return __fmul_rn(0.25f, __fadd_rn(__fadd_rn(__fadd_rn(a, b), c), d));
}
__device__ __forceinline__ float harm4(float a, float b, float c, float d) {
    return 4.0f / (__fadd_rn(__fadd_rn(__fadd_rn(1.0f / a, 1.0f / b), 1.0f / c), 1.0f / d));
}
__device__ __forceinline__ float buoyancy(float r0, float r1) {
    return __fmul_rn(2.0f, rcp(__fadd_rn(r0, r1)));
}
// Sponge gain of a cell from its axis profiles.
__device__ __forceinline__ float gain(float gx, float gy, float gz) {
    return __fmul_rn(__fmul_rn(gx, gz), gy);
}

// The arithmetic of a pass with wavefields of type T: as above for FP32; for
// 16-bit storage, which no other route serves, the plain expressions.
template <bool WIDE>
struct Form {
    __device__ static float d4(float c1, float c2, float a, float b, float c, float d) {
        if constexpr (WIDE) return ar::d4(c1, c2, a, b, c, d);
        return c1 * (c - b) + c2 * (d - a);
    }
    __device__ static void pml(float& p, float a, float b, float& d) {
        if constexpr (WIDE) {
            ar::pml(p, a, b, d);
        } else {
            p = b * p + a * d;
            d += p;
        }
    }
    __device__ static float vnew(float v, float dto, float b, float d1, float d2, float d3) {
        if constexpr (WIDE) return ar::vnew(v, dto, b, d1, d2, d3);
        return v + dto * b * (d1 + d2 + d3);
    }
    __device__ static float snormal(float s, float dto, float l2m, float lam, float e0, float e1, float e2) {
        if constexpr (WIDE) return ar::snormal(s, dto, l2m, lam, e0, e1, e2);
        return s + dto * (l2m * e0 + lam * (e1 + e2));
    }
    __device__ static float sshear(float s, float dto, float mu, float d1, float d2) {
        if constexpr (WIDE) return ar::sshear(s, dto, mu, d1, d2);
        return s + dto * mu * (d1 + d2);
    }
    __device__ static float l2m(float lam, float mu) {
        if constexpr (WIDE) return ar::l2m(lam, mu);
        return lam + 2.0f * mu;
    }
    __device__ static float mean4(float a, float b, float c, float d) {
        if constexpr (WIDE) return ar::mean4(a, b, c, d);
        return 0.25f * (a + b + c + d);
    }
    __device__ static float harm4(float a, float b, float c, float d) {
        if constexpr (WIDE) return ar::harm4(a, b, c, d);
        return 4.0f / (1.0f / a + 1.0f / b + 1.0f / c + 1.0f / d);
    }
    __device__ static float buoyancy(float r0, float r1) {
        if constexpr (WIDE) return ar::buoyancy(r0, r1);
        return __fdividef(2.0f, r0 + r1);
    }
};

}  // namespace ar
}  // namespace ews
