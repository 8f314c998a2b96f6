// Complex products and phases evaluated from float32 costs and eigenvalues, shared
// by every kernel on complex64 states.
#pragma once

#include "common.cuh"

namespace qg {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a * conj(b)
__device__ __forceinline__ float2 cmul_conj(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}

constexpr float kTwoPiF = 6.2831853071795864769f;

// e^{-i 2 pi t} for a turn count t = th + tl, a float pair: its integer part is
// removed exactly and the remaining turn f in [-1/2, 1/2] fed to the hardware
// sine/cosine at 2 pi f in [-pi, pi].  Their pair is off unit length by 7e-8 on
// average, alike for every amplitude of every round, so it is scaled to it (one
// Newton step for the inverse root, exact to float32 rounding this close to 1):
// without, <C> drifts by 1.5e-7 a round.  SK and weighted MaxCut, n = 6..23, p = 8,
// <C> against 64 bits, median (largest): 1.2e-6 (1.8e-6) without, 1.7e-7 (8e-7)
// with; sines and cosines by polynomials of 9 terms measured the same and took 4%
// of a gradient at n = 28, this 1%.
__device__ __forceinline__ float2 phase_of_turns(float th, float tl) {
    const float f = (th - rintf(th)) + tl;
    float s, c;
    __sincosf(kTwoPiF * f, &s, &c);
    const float k = fmaf(-0.5f, fmaf(c, c, s * s), 1.5f);
    return make_float2(c * k, -s * k);
}

// e^{-i gamma C} for a float32 cost, gamma/(2 pi) = g_hi + g_lo (exact head
// product by FMA).
__device__ __forceinline__ float2 phase_f32(float C, float ghi, float glo) {
    const float th = ghi * C;
    return phase_of_turns(th, fmaf(glo, C, fmaf(ghi, C, -th)));
}
// e^{-i 2 pi (g_hi + g_lo) (x_hi + x_lo)} (eigenvalues as float pairs).
__device__ __forceinline__ float2 turn_phase(float ghi, float glo, float xhi, float xlo) {
    const float th = ghi * xhi;
    return phase_of_turns(th, fmaf(ghi, xlo, fmaf(glo, xhi, fmaf(ghi, xhi, -th))));
}

}  // namespace qg
