// Real cube roots cbrt(z / beta) of the DOCH update (Eq. FPE), refined by Newton's
// method on beta y^3 = z from a base-2 logarithm / exponential start.
//
// Start: l = log2|z| / 3 + c3 with c3 = -log2(beta) / 3, y0 = 2^l (the hardware's
// FP32 approximations; relative error below 1e-6, cbrt_log of cbrt.cuh).
// A Newton step y - (beta y^3 - z) / (3 beta y^2) squares the error.
#pragma once

#include <cmath>

namespace doch {

template <typename T> struct RootOf;
struct RootF32 {
    float inv_beta, c3;
};
struct RootF64 {
    double beta;
    float c3, m3;  // m3 = 3 c3 - log2 3: log2 of 1 / (3 beta)
};

template <> struct RootOf<float> { using type = RootF32; };
template <> struct RootOf<double> { using type = RootF64; };

inline RootF32 root_f32(double inv_beta) {
    return {static_cast<float>(inv_beta), static_cast<float>(std::log2(inv_beta) / 3.0)};
}
inline RootF64 root_f64(double beta) {
    const double l = std::log2(beta);
    return {beta, static_cast<float>(-l / 3.0), static_cast<float>(-l - 1.5849625007211561)};
}

__device__ __forceinline__ float lg2_fast(float v) {
    float l;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(v));
    return l;
}
__device__ __forceinline__ float ex2_fast(float v) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(v));
    return y;
}

// the same from a beta in device memory (the start's offset from the hardware logarithm; the Newton
// steps remove its error; a beta outside the FP32 range sends FP64 roots to cbrt)
template <typename T>
__device__ __forceinline__ typename RootOf<T>::type make_root(double beta) {
    const float l = lg2_fast(static_cast<float>(beta));
    if constexpr (sizeof(T) == 4) return {static_cast<float>(1.0 / beta), l * (-1.0f / 3.0f)};
    else return {beta, l * (-1.0f / 3.0f), -l - 1.5849625007211561f};
}

// FP32: one Newton step, the reciprocal 1 / (3 y^2) also from an exponential (2^(-2 l - log2 3)).
// The residual a - y^3 with a = z / beta carries one rounding of a and one of y^2, each divided
// by three: the result is within about 0.6 ulp of cbrt of the rounded z / beta (CUDA's cbrtf: 1).
// This holds for y in (2^-kNear, 2^kNear). `far` collects the largest |log2 y|: where it reaches kNear (zeros and
// subnormal z among them, as -infinity) root_near's result is not to be used. NaN passes through.
constexpr float kNear = 40.f;
__device__ __forceinline__ float root_near(float z, RootF32 p, float &far) {
    const float l = fmaf(lg2_fast(fabsf(z)), 1.0f / 3.0f, p.c3);
    const float y = copysignf(ex2_fast(l), z);
    const float w = ex2_fast(fmaf(l, -2.0f, -1.5849625007211561f));
    const float e = fmaf(-(y * y), y, z * p.inv_beta);
    far = fmaxf(far, fabsf(l));
    return fmaf(e, w, y);
}
// the same for any z: CUDA's cbrtf outside that range
static __device__ __noinline__ float root_far(float z, float inv_beta) { return cbrtf(z * inv_beta); }
__device__ __forceinline__ float root_newton(float z, RootF32 p) {
    float far = 0.f;
    const float y = root_near(z, p, far);
    return far < kNear ? y : root_far(z, p.inv_beta);
}

// 2^-126 <= |f| < 2^128 as a double, by moving the exponent and mantissa fields (conversions and
// FP64 arithmetic run at 2 lanes per clock and SM here, integer operations at 64)
__device__ __forceinline__ double widen_normal(float f) {
    const unsigned u = __float_as_uint(f);
    return __hiloint2double(
        static_cast<int>((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), static_cast<int>(u << 29));
}

// FP64: two Newton steps from the FP32 start (1e-6 -> 1e-12 -> rounding), nine FP64 operations
// against about forty for a division and CUDA's cbrt. The last step adds a correction of relative
// size 1e-12, so the error is that of one rounding plus a third of the residual's (about 0.9 ulp;
// the division and cbrt together: up to 1.2). Zero, infinities, NaN and arguments whose FP32 start
// or weight 1 / (3 beta y^2) leaves its range take cbrt(z / beta).
static __device__ __noinline__ double root_far(double z, double beta) { return cbrt(z / beta); }
__device__ __forceinline__ double root_newton(double z, const RootF64 &p) {
    const float l = fmaf(lg2_fast(fabsf(static_cast<float>(z))), 1.0f / 3.0f, p.c3);
    const float m = fmaf(l, -2.0f, p.m3);
    if (!(fabsf(l) < 100.f && fabsf(m) < 100.f)) return root_far(z, p.beta);
    double y = widen_normal(ex2_fast(l));
    y = __hiloint2double(__double2hiint(y) | (__double2hiint(z) & static_cast<int>(0x80000000u)), __double2loint(y));
    const double w = widen_normal(ex2_fast(m));
    y = fma(fma(-(y * y), p.beta * y, z), w, y);
    return fma(fma(-(y * y), p.beta * y, z), w, y);
}

// The adjoint's weight w = g / (3 x^2), 0 where x = 0: the fast division (within 2 ulp) for a normal
// denominator below 2^126, the IEEE division for the rest
__device__ __forceinline__ float dcbrt_weight(float g, float x) {
    const float d = 3.0f * x * x;
    if (d >= 0x1p-126f && d < 0x1p126f) return __fdividef(g, d);
    return x == 0.0f ? 0.0f : g / d;
}

}  // namespace doch
