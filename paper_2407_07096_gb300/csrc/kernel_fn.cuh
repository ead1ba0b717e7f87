// The kernel functions of Sec. 3 in the log2-shifted form the plain kernels evaluate:
// with negc = -a log2(e) and a per-row integer shift s, one term is k(r) 2^-s, where
//   Gaussian     k = exp(-a r^2)                      -> 2^(negc d2 - s)
//   exponential  k = exp(-a r)                        -> 2^(negc r - s)
//   logistic     k = 4 / (2 + e^{ar} + e^{-ar})       -> 4 t' / (1 + t)^2,
//                t = 2^(negc r) <= 1, t' = 2^(negc r - s)
// (the logistic form in the bounded variable t equals the definition and cannot
// overflow). d2 is the squared distance, r = sqrt(d2).
#pragma once
#include "f32x2.cuh"
#include "stag_kde.h"

namespace stagkde {
namespace kfn {

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// sqrt with the hardware approximation (relative error ~2^-23, 0 at 0): r enters the
// exponent, where this adds ~a r 2^-23 to a term's relative error, below the squared
// distance's own rounding error for d >= 4 and within the plain form's bound for all d.
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// v 2^de for de in [-4000, 0] on the integer pipe (ldexp's FP64 multiplications hold the
// FP64 pipe, two lanes per SM and clock, for 16 clocks each). Results below 2^-1022 are 0.
__device__ __forceinline__ double scale_down(double v, int de) {
    const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff;
    if (e == 0x7ff) return v;
    return e + de > 0 ? __hiloint2double(hi + (de << 20), __double2loint(v)) : 0.0;
}

template <int KERN>
__device__ __forceinline__ float term(float negc, float d2, float shift) {
    if constexpr (KERN == STAG_KDE_KERNEL_GAUSSIAN) {
        return ex2_approx(fmaf(negc, d2, -shift));
    } else {
        const float x = negc * sqrt_approx(d2);  // log2 of exp(-a r)
        const float ts = ex2_approx(x - shift);
        if constexpr (KERN == STAG_KDE_KERNEL_EXPONENTIAL) {
            return ts;
        } else {
            const float t = ex2_approx(x);
            const float den = (1.f + t) * (1.f + t);
            return __fdividef(4.f * ts, den);
        }
    }
}

// term for a packed pair of squared distances (the Gaussian's multiply-add is packed too;
// each half's result is that of term).
template <int KERN>
__device__ __forceinline__ void term2(float negc, uint64_t negc2, uint64_t d2, float shift, float &e0, float &e1) {
    if constexpr (KERN == STAG_KDE_KERNEL_GAUSSIAN) {
        float a0, a1;
        f2::unpack(f2::fma(negc2, d2, f2::pack(-shift, -shift)), a0, a1);
        e0 = ex2_approx(a0);
        e1 = ex2_approx(a1);
    } else {
        float a0, a1;
        f2::unpack(d2, a0, a1);
        e0 = term<KERN>(negc, a0, shift);
        e1 = term<KERN>(negc, a1, shift);
    }
}

// Upper bound (log2) of a term before the shift, used to choose a new shift.
template <int KERN>
__device__ __forceinline__ float term_log2(float negc, float d2) {
    if constexpr (KERN == STAG_KDE_KERNEL_GAUSSIAN)
        return negc * d2;
    else
        return negc * sqrt_approx(d2);  // the logistic factor 4 / (1 + t)^2 is at most 4
}

}  // namespace kfn
}  // namespace stagkde
