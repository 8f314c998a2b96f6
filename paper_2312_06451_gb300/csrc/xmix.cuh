// Device helpers of the transverse-field (X) mixer kernels: phase tables, round
// coefficients, packed rotations and warp sums, shared by the pass kernels
// (xpass.cuh), the kernels for all rounds in one launch (kernels_onchip.cu,
// kernels_grid.cu) and the coefficient and small-state kernels (kernels_xmix.cu).
#pragma once

#include "common.cuh"
#include "bulk.cuh"
#include "phase.cuh"

#include <math.h>

#include <algorithm>

namespace qg {
namespace {

// Tile of the pass and grid kernels: 2^12 amplitudes, 16 in each of 256 threads.
constexpr int kT = kPassTileBits;
constexpr int kTile = 1 << kT;
constexpr int kNT = 256;
constexpr int kNW = kNT / 32;

// (sin, cos) of 2 pi t for a float64 turn count t, without float64
// transcendentals (slow on this part): t = q/4 + r with the nearest quarter
// turn q/4 removed in float64, |r| <= 1/8 to the float32 sincospi, then the
// quarter turns applied exactly.  Values near zero keep their relative accuracy.
__device__ __forceinline__ void sincos_turns(double t, float *s, float *c) {
    const double q = rint(4.0 * t);
    const float r = (float)(t - 0.25 * q);
    float sr, cr;
    sincospif(2.f * r, &sr, &cr);
    switch ((int)((long long)q & 3)) {
    case 0: *s = sr; *c = cr; break;
    case 1: *s = cr; *c = -sr; break;
    case 2: *s = -sr; *c = -cr; break;
    default: *s = -cr; *c = sr; break;
    }
}

// gamma / (2 pi) for whole costs without its own whole turns, which change no
// phase: what is left fits a float pair to 2^-49 of a turn however large gamma is.
__device__ __forceinline__ double whole_cost_turns(double g) {
    return ((uint32_t)__double2hiint(g) & 0x7fffffffu) >= 0x3fe00000u ? g - rint(g) : g;  // |g| >= 1/2
}

// e^{-i gamma c} for a small whole cost c, gamma/(2 pi) = g_hi + g_lo (see
// whole_cost_turns): the quarter turns of the head product removed exactly in float32, the tail (the
// head's rounding and g_lo c) added to the remainder, so the phase is as
// accurate as from a float64 turn count, without float64 arithmetic (16 cycles
// a warp instruction on this part).
__device__ __forceinline__ float2 phase_turns(float ghi, float glo, float c) {
    const float th = ghi * c;
    const float tail = fmaf(glo, c, fmaf(ghi, c, -th));
    const float q = rintf(4.f * th);
    const float r = fmaf(-0.25f, q, th) + tail;
    float sr, cr;
    sincospif(2.f * r, &sr, &cr);
    // quarter turns: q mod 4 from the float (exact: q is whole)
    const int m = (int)(q - 4.f * floorf(0.25f * q));
    const float sn = m == 0 ? sr : m == 1 ? cr : m == 2 ? -sr : -cr;
    const float cs = m == 0 ? cr : m == 1 ? -sr : m == 2 ? -cr : sr;
    return make_float2(cs, -sn);
}

constexpr double kInvTwoPi = 0.15915494309189533577;  // 1 / (2 pi)

// Product of two float pairs (value x + y, |y| at most half an ulp of x).
__device__ __forceinline__ float2 pair_mul(float2 a, float2 b) {
    const float p = a.x * b.x;
    const float e = fmaf(a.x, b.x, -p) + fmaf(a.x, b.y, a.y * b.x);
    const float t = p + e;
    return make_float2(t, e - (t - p));
}

// Round coefficients from one beta (rotation) and the round's gamma (whole:
// for phases of whole costs only).
__device__ __forceinline__ RoundCoef make_coef(double be, double ga, bool whole = false) {
    const double bb = be * kInvTwoPi;
    float sb, cb;
    sincos_turns(bb, &sb, &cb);
    RoundCoef c;
    c.cb = cb;
    c.sb = sb;
    // tan form unless cos b is so small that the running 1/cos factors or
    // the pair-term scale would leave float32 range (then: direct form)
    if (fabsf(cb) >= 2.44140625e-4f) {
        c.bmode = 0;
        c.bt = sb / cb;
    } else {
        c.bmode = 2;
        c.bt = 0.f;
    }
    c.rescale = fabsf(cb) < 0.25f ? 1 : 0;
    const double g = whole ? whole_cost_turns(ga * kInvTwoPi) : ga * kInvTwoPi;
    c.g_hi = (float)g;
    c.g_lo = (float)(g - (double)c.g_hi);
    c.b_hi = (float)bb;
    c.b_lo = (float)(bb - (double)c.b_hi);
    // cos b as the rounded tan b has it, so that the rotations keep the norm
    // whatever t was rounded to, and its powers rounded once each
    double ce = (double)cb;
    if (c.bmode == 0) {  // 1 / sqrt(1 + t^2): a float32 start and two Newton steps
        const double x = fma((double)c.bt, (double)c.bt, 1.0);
        double y = (double)rsqrtf((float)x);
        y = y * fma(-0.5 * x * y, y, 1.5);
        y = y * fma(-0.5 * x * y, y, 1.5);
        ce = cb < 0.f ? -y : y;
    }
    const double c2 = ce * ce, c4 = c2 * c2, c8 = c4 * c4;
    const double pw[13] = {1.0, ce, c2, c2 * ce, c4, c4 * ce, c4 * c2, c4 * c2 * ce, c8, c8 * ce, c8 * c2,
                           c8 * c2 * ce, c8 * c4};
#pragma unroll
    for (int k = 0; k <= kPassTileBits; k++) c.pw[k] = (float)pw[k];
    c.c_lo = (float)(ce - (double)c.pw[1]);
    c.pad = 0.f;
    return c;
}

// ----------------------------------------------------------------------------
// Packed (f32x2) rotations in the twisted basis s_x = (-i)^{|x|} psi_x, where
// e^{-i b X} on a qubit is the real matrix [[c, s], [-s, c]] applied to the
// (re, im) pair of both amplitudes alike.  Register pairs (i, i | 1<<RB).
struct Rot {
    float2 tt, ntt;  // (t, t), (-t, -t), t = tan b   (bmode 0)
    float c, s;      // cos b, sin b                  (bmode 2)
    float psc;       // pair-term scale per rotation: c^2 (bmode 0) or 1
    int mode;
};

template <int RB, int MODE>
__device__ __forceinline__ void rot_pairs(float2 (&a)[16], const Rot &R) {
    if (MODE == 0) {
#pragma unroll
        for (int i = 0; i < 16; i++) {
            if (i & (1 << RB)) continue;
            const int j = i | (1 << RB);
            const float2 x = a[i], y = a[j];
            a[i] = __ffma2_rn(R.tt, y, x);   // s0 + t s1
            a[j] = __ffma2_rn(R.ntt, x, y);  // s1 - t s0
        }
    } else {
        const float2 cc = make_float2(R.c, R.c), ss = make_float2(R.s, R.s), nss = make_float2(-R.s, -R.s);
#pragma unroll
        for (int i = 0; i < 16; i++) {
            if (i & (1 << RB)) continue;
            const int j = i | (1 << RB);
            const float2 x = a[i], y = a[j];
            a[i] = __ffma2_rn(ss, y, __fmul2_rn(cc, x));   // c s0 + s s1
            a[j] = __ffma2_rn(nss, x, __fmul2_rn(cc, y));  // c s1 - s s0
        }
    }
}

// This thread's share of Im <lambda| X_q |psi> in the twisted basis, where
// X_q becomes [[0, i], [-i, 0]]: sum over pairs of l0.p1 - l1.p0 (real dot
// products of (re, im) pairs), with four independent packed accumulators.
template <int RB>
__device__ __forceinline__ float pair_dot(const float2 (&l)[16], const float2 (&p)[16]) {
    float2 ap[4], am[4];
#pragma unroll
    for (int k = 0; k < 4; k++) ap[k] = am[k] = make_float2(0.f, 0.f);
    int k = 0;
#pragma unroll
    for (int i = 0; i < 16; i++) {
        if (i & (1 << RB)) continue;
        const int j = i | (1 << RB);
        ap[k & 3] = __ffma2_rn(l[i], p[j], ap[k & 3]);
        am[k & 3] = __ffma2_rn(l[j], p[i], am[k & 3]);
        k++;
    }
    const float2 sp = __fadd2_rn(__fadd2_rn(ap[0], ap[1]), __fadd2_rn(ap[2], ap[3]));
    const float2 sm = __fadd2_rn(__fadd2_rn(am[0], am[1]), __fadd2_rn(am[2], am[3]));
    return (sp.x + sp.y) - (sm.x + sm.y);
}

// The rotations of one register layout ("stage"): on bit k = register bit k
// carries an active qubit.  The adjoint first takes the pair terms
// <lambda|X_q|psi> of all the stage's qubits at the stage's starting point --
// any point of the round where both vectors have had the same rotations
// gives the same value, because all X_q commute -- and then rotates lambda,
// and psi only when rot_psi is set (its later values are not always needed).
template <int BWD, int MODE>
__device__ __forceinline__ void stage_rot(float2 (&a)[16], float2 (&l)[16], uint32_t on, const Rot &R,
                                          float &pscale, float &bacc, bool rot_psi, bool pairs = true) {
    if (BWD) {
        if (pairs) {
            float s = 0.f;
            if (on & 1u) s += pair_dot<0>(l, a);
            if (on & 2u) s += pair_dot<1>(l, a);
            if (on & 4u) s += pair_dot<2>(l, a);
            if (on & 8u) s += pair_dot<3>(l, a);
            bacc = fmaf(s, pscale, bacc);
        }
        for (uint32_t m = on; m; m &= m - 1u) pscale *= R.psc;
        if (on & 1u) rot_pairs<0, MODE>(l, R);
        if (on & 2u) rot_pairs<1, MODE>(l, R);
        if (on & 4u) rot_pairs<2, MODE>(l, R);
        if (on & 8u) rot_pairs<3, MODE>(l, R);
    }
    if (!BWD || rot_psi) {
        if (on & 1u) rot_pairs<0, MODE>(a, R);
        if (on & 2u) rot_pairs<1, MODE>(a, R);
        if (on & 4u) rot_pairs<2, MODE>(a, R);
        if (on & 8u) rot_pairs<3, MODE>(a, R);
    }
}

// Multi-angle rotations (one angle per qubit): register bit j of the stage
// carries local bit Lj, with rot[Lj] = (cos b, +-sin b, +-tan b, cos^2 b).
// MODE 0 is the tan form (the cosines are applied per stage or per pass like
// the single-angle path, pscale tracks them for the pair terms), MODE 2 the
// direct form.  The adjoint's pair terms go to one accumulator per local bit.
template <int BWD, int MODE, int L0, int L1, int L2, int L3, int NQ>
__device__ __forceinline__ void stage_rot_ma(float2 (&a)[16], float2 (&l)[16], uint32_t on, const float4 *rot,
                                             float (&bq)[NQ], float &pscale, bool rot_psi) {
    Rot R[4];
    const int Ls[4] = {L0, L1, L2, L3};
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const float4 q = rot[Ls[j]];
        R[j].c = q.x;
        R[j].s = q.y;
        R[j].tt = make_float2(q.z, q.z);
        R[j].ntt = make_float2(-q.z, -q.z);
    }
    if (BWD) {
        if (on & 1u) bq[L0] = fmaf(pair_dot<0>(l, a), pscale, bq[L0]);
        if (on & 2u) bq[L1] = fmaf(pair_dot<1>(l, a), pscale, bq[L1]);
        if (on & 4u) bq[L2] = fmaf(pair_dot<2>(l, a), pscale, bq[L2]);
        if (on & 8u) bq[L3] = fmaf(pair_dot<3>(l, a), pscale, bq[L3]);
        if (MODE == 0) {
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (on & (1u << j)) pscale *= rot[Ls[j]].w;
        }
        if (on & 1u) rot_pairs<0, MODE>(l, R[0]);
        if (on & 2u) rot_pairs<1, MODE>(l, R[1]);
        if (on & 4u) rot_pairs<2, MODE>(l, R[2]);
        if (on & 8u) rot_pairs<3, MODE>(l, R[3]);
    }
    if (!BWD || rot_psi) {
        if (on & 1u) rot_pairs<0, MODE>(a, R[0]);
        if (on & 2u) rot_pairs<1, MODE>(a, R[1]);
        if (on & 4u) rot_pairs<2, MODE>(a, R[2]);
        if (on & 8u) rot_pairs<3, MODE>(a, R[3]);
    }
}

template <int BWD>
__device__ __forceinline__ void scale_all(float2 (&a)[16], float2 (&l)[16], float f) {
    const float2 ff = make_float2(f, f);
#pragma unroll
    for (int i = 0; i < 16; i++) {
        a[i] = __fmul2_rn(ff, a[i]);
        if (BWD) l[i] = __fmul2_rn(ff, l[i]);
    }
}

// (-i)^k * v
__device__ __forceinline__ float2 twist(float2 v, int k) {
    switch (k & 3) {
    case 0: return v;
    case 1: return make_float2(v.y, -v.x);
    case 2: return make_float2(-v.x, -v.y);
    default: return make_float2(-v.y, v.x);
    }
}

// Float64 arithmetic runs at a small fraction of the float32 rate on this
// part, so the per-tile partial sums below are summed across a warp in
// float32 (a fixed shuffle tree, so still bitwise reproducible) and only the
// warp totals are widened to float64 for the sums over tiles and warps.
// Each thread's share is itself a float32 sum of a few hundred terms, so the
// warp step adds an error of the same order (~1e-7 of the sum of magnitudes).

// Warp sum of one float per lane; every lane gets the total.
__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Warp sums of two floats per lane in one tree: the total of x lands in
// lanes 0..15, the total of y in lanes 16..31.
__device__ __forceinline__ float warp_sum2_f(float x, float y) {
    const bool hi = (threadIdx.x & 16u) != 0;
    float v = (hi ? y : x) + __shfl_xor_sync(0xffffffffu, hi ? x : y, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Warp sums of 16 floats per lane as a reduce-scatter: each step halves the
// values a lane keeps and trades the other half with its partner, so value
// j's total lands in lanes 2j and 2j + 1 after 16 shuffles (not 80).
__device__ __forceinline__ float warp_sum16_f(const float (&v)[16]) {
    const uint32_t lane = threadIdx.x & 31u;
    float w8[8], w4[4], w2[2];
    const bool h4 = lane & 16u, h3 = lane & 8u, h2 = lane & 4u, h1 = lane & 2u;
#pragma unroll
    for (int k = 0; k < 8; k++)
        w8[k] = (h4 ? v[k + 8] : v[k]) + __shfl_xor_sync(0xffffffffu, h4 ? v[k] : v[k + 8], 16);
#pragma unroll
    for (int k = 0; k < 4; k++)
        w4[k] = (h3 ? w8[k + 4] : w8[k]) + __shfl_xor_sync(0xffffffffu, h3 ? w8[k] : w8[k + 4], 8);
#pragma unroll
    for (int k = 0; k < 2; k++)
        w2[k] = (h2 ? w4[k + 2] : w4[k]) + __shfl_xor_sync(0xffffffffu, h2 ? w4[k] : w4[k + 2], 4);
    float w = (h1 ? w2[1] : w2[0]) + __shfl_xor_sync(0xffffffffu, h1 ? w2[0] : w2[1], 2);
    return w + __shfl_xor_sync(0xffffffffu, w, 1);
}

// Deterministic block sum of one float per thread: float32 within each
// warp, float64 across warps; the result is valid in thread 0.
template <int NW>
__device__ __forceinline__ double block_sum(float v, double *red) {
    double d = (double)warp_sum_f(v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) red[warp] = d;
    __syncthreads();
    double tot = 0.0;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 0; w < NW; w++) tot += red[w];
    }
    __syncthreads();
    return tot;
}


}  // namespace
}  // namespace qg
