// Register layouts and rounds of the on-chip X-mixer kernels (kernels_onchip.cu,
// kernels_grid.cu): 2^NB amplitudes, 16 in each of 2^(NB-4) threads.
#pragma once

#include "xmix.cuh"

namespace qg {
namespace {

constexpr int kChunk = 32;  // rounds whose coefficients are in shared memory

struct RoundC {
    Rot R;
    int rescale;
    float fq, fr, fp, fe;  // cos factors of the layouts' rotations and of all of them
    float hq, hp, he;      // the same for the rotations after an exchange (kernels_grid.cu)
    float ghi, glo;
};

template <int NB>
struct Chip {
    static constexpr int NT = 1 << (NB - 4);
    static constexpr int NW = NT / 32;
    static constexpr int kP = NB - 4;  // lowest amplitude bit of layout P
    static constexpr int N = 1 << NB;
};

__device__ __forceinline__ uint32_t sw(uint32_t l) { return l ^ (((l >> 4) & 7u) << 1); }

template <int NB>
struct Pos {  // swizzled slots of amplitude 0 in the layouts, and local indexes
    uint32_t lp, lq, sp, sr;
    __device__ __forceinline__ Pos() {
        const uint32_t t = threadIdx.x;
        lp = t;
        lq = (t & 15u) | ((t >> 4) << 8);
        sp = sw(lp);
        sr = sw(t << 4);
    }
};

// One vector moved between layouts through its slots.
template <int NB>
__device__ __forceinline__ void put_p(const float2 (&v)[16], float2 *s, const Pos<NB> &T) {
#pragma unroll
    for (int i = 0; i < 16; i++) s[T.sp ^ sw((uint32_t)i << Chip<NB>::kP)] = v[i];
}
template <int NB>
__device__ __forceinline__ void get_p(float2 (&v)[16], const float2 *s, const Pos<NB> &T) {
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = s[T.sp ^ sw((uint32_t)i << Chip<NB>::kP)];
}
template <int NB>
__device__ __forceinline__ void put_q(const float2 (&v)[16], float2 *s, const Pos<NB> &T) {
#pragma unroll
    for (int i = 0; i < 16; i++) s[(T.lq ^ ((i & 7) << 1)) + (i << 4)] = v[i];
}
template <int NB>
__device__ __forceinline__ void get_q(float2 (&v)[16], const float2 *s, const Pos<NB> &T) {
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = s[(T.lq ^ ((i & 7) << 1)) + (i << 4)];
}
template <int NB>
__device__ __forceinline__ void put_r(const float2 (&v)[16], float2 *s, const Pos<NB> &T) {
#pragma unroll
    for (int r = 0; r < 8; r++)
        *reinterpret_cast<float4 *>(s + (T.sr ^ (r << 1))) =
            make_float4(v[2 * r].x, v[2 * r].y, v[2 * r + 1].x, v[2 * r + 1].y);
}
template <int NB>
__device__ __forceinline__ void get_r(float2 (&v)[16], const float2 *s, const Pos<NB> &T) {
#pragma unroll
    for (int r = 0; r < 8; r++) {
        const float4 w = *reinterpret_cast<const float4 *>(s + (T.sr ^ (r << 1)));
        v[2 * r] = make_float2(w.x, w.y);
        v[2 * r + 1] = make_float2(w.z, w.w);
    }
}

struct Masks {
    uint32_t q, r, p;
};

// Shared constants of a round whose layouts rotate M's bits (and, after an
// exchange, the bits hp of P and hq of Q).
__device__ __forceinline__ RoundC round_consts(const RoundCoef &cf, const Masks &M, uint32_t hp, uint32_t hq) {
    RoundC C;
    const bool tan = cf.bmode == 0;
    C.R.mode = cf.bmode;
    C.R.tt = make_float2(cf.bt, cf.bt);
    C.R.ntt = make_float2(-cf.bt, -cf.bt);
    C.R.c = cf.cb;
    C.R.s = cf.sb;
    C.R.psc = tan ? cf.pw[2] : 1.f;
    C.rescale = tan && cf.rescale ? 1 : 0;
    const int nq = __popc(M.q), nr = __popc(M.r), np = __popc(M.p), xq = __popc(hq), xp = __popc(hp);
    C.fq = tan ? cf.pw[nq] : 1.f;
    C.fr = tan ? cf.pw[nr] : 1.f;
    C.fp = tan ? cf.pw[np] : 1.f;
    C.fe = tan && !C.rescale ? cf.pw[nq + nr + np] : 1.f;
    C.hq = tan ? cf.pw[xq] : 1.f;
    C.hp = tan ? cf.pw[xp] : 1.f;
    C.he = tan && !C.rescale ? cf.pw[xq + xp] : 1.f;
    C.ghi = cf.g_hi;
    C.glo = cf.g_lo;
    return C;
}
// The round's constants, or those that undo it (sgn < 0).
__device__ __forceinline__ RoundC signed_round(RoundC C, float sgn) {
    if (sgn < 0.f) {
        const float2 t = C.R.tt;
        C.R.tt = C.R.ntt;
        C.R.ntt = t;
        C.R.s = -C.R.s;
    }
    return C;
}

// The rotations of one round on a (and l, undone): from layout Q to P (UP) or
// from P to Q.
template <int NB, int BWD, int MODE, int UP>
__device__ __forceinline__ void rotate_round(float2 (&a)[16], float2 (&l)[16], float2 *sa, float2 *sl,
                                             const RoundC &C, const Masks &M, const Pos<NB> &T, float &bacc) {
    float ps = 1.f;
    stage_rot<BWD, MODE>(a, l, UP ? M.q : M.p, C.R, ps, bacc, true);
    if (C.rescale) {
        scale_all<BWD>(a, l, UP ? C.fq : C.fp);
        ps = 1.f;
    }
    if (UP) {
        put_q<NB>(a, sa, T);
        if (BWD) put_q<NB>(l, sl, T);
        __syncwarp();
    } else {
        put_p<NB>(a, sa, T);
        if (BWD) put_p<NB>(l, sl, T);
        __syncthreads();
    }
    get_r<NB>(a, sa, T);
    if (BWD) get_r<NB>(l, sl, T);
    stage_rot<BWD, MODE>(a, l, M.r, C.R, ps, bacc, true);
    if (C.rescale) {
        scale_all<BWD>(a, l, C.fr);
        ps = 1.f;
    }
    put_r<NB>(a, sa, T);
    if (BWD) put_r<NB>(l, sl, T);
    if (UP) {
        __syncthreads();
        get_p<NB>(a, sa, T);
        if (BWD) get_p<NB>(l, sl, T);
    } else {
        __syncwarp();
        get_q<NB>(a, sa, T);
        if (BWD) get_q<NB>(l, sl, T);
    }
    stage_rot<BWD, MODE>(a, l, UP ? M.p : M.q, C.R, ps, bacc, true);
    scale_all<BWD>(a, l, C.rescale ? (UP ? C.fp : C.fq) : C.fe);
}

template <int NB, int BWD, int UP>
__device__ __forceinline__ void rotate_any(float2 (&a)[16], float2 (&l)[16], float2 *sa, float2 *sl, const RoundC &C,
                                           const Masks &M, const Pos<NB> &T, float &bacc) {
    if (C.R.mode == 0) rotate_round<NB, BWD, 0, UP>(a, l, sa, sl, C, M, T, bacc);
    else rotate_round<NB, BWD, 2, UP>(a, l, sa, sl, C, M, T, bacc);
}

}  // namespace
}  // namespace qg
