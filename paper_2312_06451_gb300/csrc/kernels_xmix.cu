// Transverse-field (X) mixer path: phase separator, per-qubit mixer
// rotations, expectation and adjoint (reverse-mode) gradient on complex64
// states.
//
// Method (arXiv 2312.06451): round k applies e^{-i gamma_k C} elementwise and
// then e^{-i beta_k sum_i X_i} (Eq. 1).  Because the X_i commute, the mixer is
// n independent single-qubit rotations (Sec. 2.2; Eq. 2 is the equivalent
// Hadamard-diagonal form), each mixing the amplitude pairs (x, x xor 2^i).
//
// Kernel design (sm_103a, HBM-bound):
//   * A pass streams the state once through the SMs in tiles of 2^T
//     amplitudes and applies every rotation whose qubit is a tile bit, so one
//     round costs ceil(n / T)-ish passes instead of n sweeps.  The first pass
//     of a tile set covers qubits 0..T-1 with fully contiguous tiles; later
//     passes gather 2^c contiguous amplitudes (c >= 4: whole 128-byte lines)
//     times 2^(T-c) strided ones to reach the high qubits.
//   * Each thread holds 16 amplitudes of each vector in registers (a tile of
//     2^12 amplitudes, 256 threads).  A tile goes through as many register
//     layouts as its rotated bits need (four bits each: one to three), with a
//     bank-conflict free shared-memory transpose between two.  Every rotation
//     happens in registers, in the layout where its bit is a register bit.
//   * The phase e^{-i gamma C} is applied as the tile is loaded, the
//     expectation sum |psi|^2 C as it is stored, so neither costs a pass.
//   * The adjoint pass carries lambda and psi together, undoing the rotations
//     of both and accumulating 2 Im <lambda|X_i|psi> for the beta derivative
//     as each qubit comes by (valid at any point of the round because all
//     X_i commute); the gamma derivative 2 Im <mu|C|phi> and the undone phase
//     are fused into the last adjoint pass of the round.
//   * Partial sums are per tile in float32, combined in float64 in a fixed
//     order, so results are bitwise reproducible.
#include "xmix.cuh"

namespace qg {
namespace {

// --------------------------------------------------------------------------
// Whole state in shared memory (n <= kSmallMaxN): all p rounds, the
// expectation and (GRAD) the adjoint sweep in one block per unit.  The adjoint
// undoes each round on psi in place.
constexpr int kSmallMaxN = 12;
constexpr int kSmallThreads = 256;

template <int COST, int GRAD>
__global__ void __launch_bounds__(kSmallThreads)
small_kernel(const SmallDesc *__restrict__ descs, int *err) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ double s_red[kSmallThreads / 32];
    const SmallDesc D = descs[blockIdx.x];
    const int N = 1 << D.n, H = N >> 1, n = D.n, p = D.p;
    float2 *psi = reinterpret_cast<float2 *>(smem_raw);
    float2 *lam = psi + N;
    float2 *tab = psi + 2 * N;
    const int tid = threadIdx.x;
    (void)err;

    auto costv = [&](int x) -> float {
        if (COST == 0) return __ldg(reinterpret_cast<const float *>(D.cost) + x);
        return (float)__ldg(reinterpret_cast<const unsigned char *>(D.cost) + x);
    };
    auto phase = [&](int x, const RoundCoef &cf) -> float2 {
        if (COST == 0) return phase_f32(costv(x), cf.g_hi, cf.g_lo);
        return tab[__ldg(reinterpret_cast<const unsigned char *>(D.cost) + x)];
    };
    auto load_table = [&](int k) {
        if (COST == 1) {
            __syncthreads();
            for (int i = tid; i < kPhaseTable; i += kSmallThreads)
                tab[i] = D.table[k * kPhaseTable + i];
            __syncthreads();
        }
    };
    // e^{-i b X_q} on every pair of qubit q (cb, sb: cos b, sin b)
    auto mix = [&](float2 *v, int q, float cb, float sb) {
        for (int j = tid; j < H; j += kSmallThreads) {
            const int lo = j & ((1 << q) - 1);
            const int x0 = ((j - lo) << 1) | lo, x1 = x0 | (1 << q);
            const float2 u = v[x0], w = v[x1];
            v[x0] = make_float2(fmaf(cb, u.x, sb * w.y), fmaf(cb, u.y, -sb * w.x));
            v[x1] = make_float2(fmaf(cb, w.x, sb * u.y), fmaf(cb, w.y, -sb * u.x));
        }
    };

    // general X mixer (plain basis here): H^n diag(e^{-i b d_|x|}) H^n
    __shared__ float2 s_gph[kSmallMaxN + 1];
    auto hadamard_all = [&](float2 *v) {
        const float r = 0.70710678118654752f;
        for (int q = 0; q < n; q++) {
            __syncthreads();
            for (int j = tid; j < H; j += kSmallThreads) {
                const int lo = j & ((1 << q) - 1);
                const int x0 = ((j - lo) << 1) | lo, x1 = x0 | (1 << q);
                const float2 u = v[x0], w = v[x1];
                v[x0] = make_float2(r * (u.x + w.x), r * (u.y + w.y));
                v[x1] = make_float2(r * (u.x - w.x), r * (u.y - w.y));
            }
        }
        __syncthreads();
    };
    auto weight_phases = [&](double b) {  // s_gph[w] = e^{-i b d_w}
        __syncthreads();
        if (tid <= n) {
            float sn, cs;
            sincos_turns(b * D.wts[tid] * kInvTwoPi, &sn, &cs);
            s_gph[tid] = make_float2(cs, -sn);
        }
        __syncthreads();
    };
    // coefficients of round k: one entry, one per qubit (multi-angle) or two
    // (general X mixer); nb angles per round's mixer
    const int nb = D.nq ? D.nq : 1;
    const int cs = D.nq ? D.nq : (D.wts ? 2 : 1);
    auto qcoef = [&](int k, int q) -> const RoundCoef & { return D.coef[k * cs + (D.nq ? q : 0)]; };

    for (int x = tid; x < N; x += kSmallThreads)
        psi[x] = D.init ? D.init[x] : make_float2(D.amp0, 0.f);
    for (int k = 0; k < p; k++) {
        const RoundCoef cf = D.coef[k * cs];
        __syncthreads();
        load_table(k);
        for (int x = tid; x < N; x += kSmallThreads) psi[x] = cmul(psi[x], phase(x, cf));
        if (D.wts) {
            weight_phases(D.angles_beta[k]);
            hadamard_all(psi);
            for (int x = tid; x < N; x += kSmallThreads) psi[x] = cmul(psi[x], s_gph[__popc(x)]);
            hadamard_all(psi);
            continue;
        }
        for (int q = 0; q < n; q++) {
            __syncthreads();
            mix(psi, q, qcoef(k, q).cb, qcoef(k, q).sb);
        }
    }
    __syncthreads();
    float e = 0.f;
    for (int x = tid; x < N; x += kSmallThreads)
        e = fmaf(costv(x), fmaf(psi[x].x, psi[x].x, psi[x].y * psi[x].y), e);
    const double E = block_sum<kSmallThreads / 32>(e, s_red);
    if (tid == 0) *D.E_out = E;
    if constexpr (GRAD) {
    // the adjoint uses C - <C>: the same gradient, without the common
    // component <C> psi in lambda
    __shared__ float s_c0;
    if (tid == 0) s_c0 = (float)E;
    __syncthreads();
    const float c0 = s_c0;
    for (int x = tid; x < N; x += kSmallThreads) {
        const float c = costv(x) - c0;
        lam[x] = make_float2(c * psi[x].x, c * psi[x].y);
    }
    for (int k = p - 1; k >= 0; k--) {
        const RoundCoef cf = D.coef[k * cs];
        __syncthreads();
        float gb = 0.f;
        if (D.wts) {
            // in the Hadamard frame: beta partial sum_z d_|z| Im(conj(lam) psi),
            // then the diagonal undone and the frame left again
            weight_phases(D.angles_beta[k]);
            hadamard_all(lam);
            hadamard_all(psi);
            for (int x = tid; x < N; x += kSmallThreads) {
                const float2 l = lam[x], a = psi[x];
                gb = fmaf((float)D.wts[__popc(x)], l.x * a.y - l.y * a.x, gb);
                lam[x] = cmul_conj(l, s_gph[__popc(x)]);
                psi[x] = cmul_conj(a, s_gph[__popc(x)]);
            }
            const double GB = block_sum<kSmallThreads / 32>(gb, s_red);
            if (tid == 0) D.grad_out[k] = 2.0 * GB;
            hadamard_all(lam);
            hadamard_all(psi);
        }
        for (int q = 0; q < (D.wts ? 0 : n); q++) {
            float gq = 0.f;
            for (int j = tid; j < H; j += kSmallThreads) {
                const int lo = j & ((1 << q) - 1);
                const int x0 = ((j - lo) << 1) | lo, x1 = x0 | (1 << q);
                const float2 l0 = lam[x0], l1 = lam[x1], a0 = psi[x0], a1 = psi[x1];
                gq += l0.x * a1.y - l0.y * a1.x + l1.x * a0.y - l1.y * a0.x;
            }
            if (D.nq) {  // one partial per qubit
                const double GQ = block_sum<kSmallThreads / 32>(gq, s_red);
                if (tid == 0) D.grad_out[k * n + q] = 2.0 * GQ;
            } else {
                gb += gq;
            }
        }
        if (!D.nq && !D.wts) {
            const double GB = block_sum<kSmallThreads / 32>(gb, s_red);
            if (tid == 0) D.grad_out[k] = 2.0 * GB;
        }
        for (int q = 0; q < (D.wts ? 0 : n); q++) {
            __syncthreads();
            mix(lam, q, qcoef(k, q).cb, -qcoef(k, q).sb);
            mix(psi, q, qcoef(k, q).cb, -qcoef(k, q).sb);
        }
        __syncthreads();
        load_table(k);
        float gg = 0.f;
        for (int x = tid; x < N; x += kSmallThreads) {
            const float2 l = lam[x], a = psi[x];
            gg = fmaf(costv(x) - c0, l.x * a.y - l.y * a.x, gg);
        }
        const double GG = block_sum<kSmallThreads / 32>(gg, s_red);
        if (tid == 0) D.grad_out[p * nb + k] = 2.0 * GG;
        for (int x = tid; x < N; x += kSmallThreads) {
            const float2 ph = phase(x, cf);
            lam[x] = cmul_conj(lam[x], ph);
            psi[x] = cmul_conj(psi[x], ph);
        }
    }
    }  // GRAD
}

// --------------------------------------------------------------------------
// n = 12: the whole state is one tile of the pass kernels (256 threads x 16
// amplitudes), so one CTA per angle set runs every round with the pass
// kernels' three register stages and two swizzled transposes; between rounds
// the state waits in shared memory in natural order, never in global memory.
// Same twisted basis as the pass kernels (every qubit is a tile bit, so the
// stage masks are full).  The adjoint undoes each round on psi as well.
struct Round12 {
    Rot R;
    int rescale;
    float fs, fse;  // cos factors: per stage (4 rotations), per round (12)
    float ghi, glo;
};

__device__ __forceinline__ Round12 round12(const RoundCoef &cf, float sgn) {
    Round12 r;
    r.R.mode = cf.bmode;
    r.R.tt = make_float2(sgn * cf.bt, sgn * cf.bt);
    r.R.ntt = make_float2(-sgn * cf.bt, -sgn * cf.bt);
    r.R.c = cf.cb;
    r.R.s = sgn * cf.sb;
    r.R.psc = cf.bmode == 0 ? cf.pw[2] : 1.f;
    r.rescale = (cf.bmode == 0 && cf.rescale) ? 1 : 0;
    r.fs = cf.bmode == 0 ? cf.pw[4] : 1.f;
    r.fse = r.rescale || cf.bmode != 0 ? 1.f : cf.pw[12];
    r.ghi = cf.g_hi;
    r.glo = cf.g_lo;
    return r;
}

// One round on the state in shared memory (natural order in and out).
// Forward: phase on load (initial state generated or twisted in when first),
// rotations; last: <C> partial, and (GRAD) lambda = C psi written to sl.
// Adjoint: rotations of lambda and psi undone with the pair terms, then the
// gamma partial and the phase undone on both.
template <int BWD, int COST, int MODE>
__device__ void tile12_round(float2 *sp, float2 *sl, const float2 *stab, const void *scost, const SmallDesc &D,
                             const Round12 &rc, bool first, bool last, float c0, float &bacc, float &eacc) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t l1 = ((uint32_t)lane << 1) | ((uint32_t)warp << 6);
    const uint32_t l2 = ((uint32_t)lane & 1u) | ((((uint32_t)lane >> 1) & 7u) << 6) |
                        ((((uint32_t)lane >> 4) & 1u) << 5) | ((uint32_t)warp << 9);
    const uint32_t l3 = (uint32_t)lane | ((uint32_t)warp << 9);
    const uint32_t p1 = swz(l1), p2 = swz(l2), p3 = swz(l3);
    auto costv = [&](uint32_t x) -> float {  // the cost vector, copied to shared memory
        if (COST == 0) return reinterpret_cast<const float *>(scost)[x];
        return (float)reinterpret_cast<const unsigned char *>(scost)[x];
    };
    auto phase = [&](uint32_t x) -> float2 {
        if (COST == 0) return phase_f32(costv(x), rc.ghi, rc.glo);
        return stab[reinterpret_cast<const unsigned char *>(scost)[x]];
    };
    float2 a[16], l[16];
    float pscale = 1.f;
    // ---- stage 1: local bits {0, 9, 10, 11} in registers
    if (!BWD && first && !D.init) {
        const float2 a0 = twist(make_float2(D.amp0, 0.f), __popc(l1));
#pragma unroll
        for (int r = 0; r < 8; r++) {
            a[2 * r] = twist(a0, __popc(r));
            a[2 * r + 1] = twist(a0, __popc(r) + 1);
        }
    } else {
        const float2 *src = (!BWD && first) ? D.init : sp;
#pragma unroll
        for (int r = 0; r < 8; r++) {
            const float4 v = *reinterpret_cast<const float4 *>(src + (l1 | ((uint32_t)r << 9)));
            a[2 * r] = make_float2(v.x, v.y);
            a[2 * r + 1] = make_float2(v.z, v.w);
        }
        if (!BWD && first) {
            const float2 w0 = twist(make_float2(1.f, 0.f), __popc(l1));
#pragma unroll
            for (int r = 0; r < 8; r++) {
                a[2 * r] = cmul(twist(a[2 * r], __popc(r)), w0);
                a[2 * r + 1] = cmul(twist(a[2 * r + 1], __popc(r) + 1), w0);
            }
        }
    }
    if (BWD) {
#pragma unroll
        for (int r = 0; r < 8; r++) {
            const float4 v = *reinterpret_cast<const float4 *>(sl + (l1 | ((uint32_t)r << 9)));
            l[2 * r] = make_float2(v.x, v.y);
            l[2 * r + 1] = make_float2(v.z, v.w);
        }
    } else {
#pragma unroll
        for (int r = 0; r < 8; r++) {
            const uint32_t x = l1 | ((uint32_t)r << 9);
            a[2 * r] = cmul(a[2 * r], phase(x));
            a[2 * r + 1] = cmul(a[2 * r + 1], phase(x | 1u));
        }
    }
    stage_rot<BWD, MODE>(a, l, 0xFu, rc.R, pscale, bacc, true);
    if (rc.rescale) {
        scale_all<BWD>(a, l, rc.fs);
        pscale = 1.f;
    }
    // ---- stage 1 -> 2 (in place, swizzled; crosses warps)
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 8; r++) {
        const uint32_t idx = p1 ^ swz((uint32_t)r << 9);
        *reinterpret_cast<float4 *>(sp + idx) = make_float4(a[2 * r].x, a[2 * r].y, a[2 * r + 1].x, a[2 * r + 1].y);
        if (BWD)
            *reinterpret_cast<float4 *>(sl + idx) = make_float4(l[2 * r].x, l[2 * r].y, l[2 * r + 1].x, l[2 * r + 1].y);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; i++) {
        a[i] = sp[p2 ^ ((uint32_t)i << 1)];
        if (BWD) l[i] = sl[p2 ^ ((uint32_t)i << 1)];
    }
    stage_rot<BWD, MODE>(a, l, 0xFu, rc.R, pscale, bacc, true);
    if (rc.rescale) {
        scale_all<BWD>(a, l, rc.fs);
        pscale = 1.f;
    }
    // ---- stage 2 -> 3 (inside each warp's 512-amplitude block)
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; i++) {
        sp[p2 ^ ((uint32_t)i << 1)] = a[i];
        if (BWD) sl[p2 ^ ((uint32_t)i << 1)] = l[i];
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; i++) {
        const uint32_t idx = p3 ^ swz((uint32_t)i << 5);
        a[i] = sp[idx];
        if (BWD) l[i] = sl[idx];
    }
    stage_rot<BWD, MODE>(a, l, 0xFu, rc.R, pscale, bacc, true);
    scale_all<BWD>(a, l, rc.rescale ? rc.fs : rc.fse);
    // ---- epilogue and natural-order store (still this warp's block)
    if (BWD) {
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const uint32_t x = l3 | ((uint32_t)i << 5);
            const float C = costv(x);
            const float2 ph = phase(x);
            eacc = fmaf(C - c0, fmaf(l[i].x, a[i].y, -l[i].y * a[i].x), eacc);
            l[i] = cmul_conj(l[i], ph);
            a[i] = cmul_conj(a[i], ph);
        }
    } else if (last) {
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const float C = costv(l3 | ((uint32_t)i << 5));
            eacc = fmaf(C, fmaf(a[i].x, a[i].x, a[i].y * a[i].y), eacc);
        }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; i++) {
        sp[l3 | ((uint32_t)i << 5)] = a[i];
        if (BWD) sl[l3 | ((uint32_t)i << 5)] = l[i];
    }
    __syncthreads();
}

template <int COST, int GRAD>
__global__ void __launch_bounds__(kNT) tile12_kernel(const SmallDesc *__restrict__ descs, int *err) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float2 *sp = reinterpret_cast<float2 *>(smem_raw);
    float2 *sl = sp + kTile;
    float2 *stab = sl + kTile;
    unsigned char *scost = reinterpret_cast<unsigned char *>(stab + kPhaseTable);
    __shared__ double s_red[2][kNW];
    const SmallDesc D = descs[blockIdx.x];
    const int p = D.p, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    {  // cost vector to shared memory (16-byte words)
        const int words = kTile * (COST == 0 ? 4 : 1) / 16;
        for (int i = tid; i < words; i += kNT)
            reinterpret_cast<uint4 *>(scost)[i] = __ldg(reinterpret_cast<const uint4 *>(D.cost) + i);
        __syncthreads();
    }
    // coefficients and the uint8 phase table come from the angles here (no
    // separate preparation launch); every thread forms the round's coefficients
    const double *ang = D.angles_beta;
    if (tid < 2 * p && !isfinite(ang[tid])) atomicOr(err, DERR_BAD_ANGLE);
    auto load_table = [&](int k) {  // the previous round ended with a block barrier
        if (COST == 1) {
            for (int i = tid; i < kPhaseTable; i += kNT) {
                float sn, cs;
                sincos_turns(ang[p + k] * kInvTwoPi * (double)i, &sn, &cs);
                stab[i] = make_float2(cs, -sn);
            }
            __syncthreads();
        }
    };
    // fixed-order block sums of two per-thread values: float32 within a
    // warp (x in lanes 0..15, y in 16..31), float64 across warps
    auto block_sum2 = [&](float x, float y, double &X, double &Y) {
        const float t = warp_sum2_f(x, y);
        if (lane == 0) s_red[0][warp] = (double)t;
        if (lane == 16) s_red[1][warp] = (double)t;
        __syncthreads();
        X = 0.0;
        Y = 0.0;
        for (int w = 0; w < kNW; w++) {
            X += s_red[0][w];
            Y += s_red[1][w];
        }
        __syncthreads();
    };
    float bacc = 0.f, eacc = 0.f;
    for (int k = 0; k < p; k++) {
        const Round12 rc = round12(make_coef(ang[k], ang[p + k]), 1.f);
        load_table(k);
        if (rc.R.mode == 0)
            tile12_round<0, COST, 0>(sp, sl, stab, scost, D, rc, k == 0, k == p - 1, 0.f, bacc, eacc);
        else
            tile12_round<0, COST, 2>(sp, sl, stab, scost, D, rc, k == 0, k == p - 1, 0.f, bacc, eacc);
    }
    double E, unused;
    block_sum2(eacc, 0.f, E, unused);
    if (tid == 0) *D.E_out = E;
    if constexpr (GRAD) {
        // lambda_p = (C - <C>) psi_p: the adjoint with the cost shifted by its
        // expectation gives the same gradient without the common component
        // <C> psi in lambda (every thread holds E after block_sum2)
        const float c0 = (float)E;
        for (int x = tid; x < kTile; x += kNT) {
            const float C = COST == 0 ? reinterpret_cast<const float *>(scost)[x]
                                      : (float)reinterpret_cast<const unsigned char *>(scost)[x];
            const float2 v = sp[x];
            sl[x] = make_float2((C - c0) * v.x, (C - c0) * v.y);
        }
        __syncthreads();
        for (int k = p - 1; k >= 0; k--) {
            const Round12 rc = round12(make_coef(ang[k], ang[p + k]), -1.f);
            load_table(k);
            float b = 0.f, g = 0.f;
            if (rc.R.mode == 0)
                tile12_round<1, COST, 0>(sp, sl, stab, scost, D, rc, false, false, c0, b, g);
            else
                tile12_round<1, COST, 2>(sp, sl, stab, scost, D, rc, false, false, c0, b, g);
            double B, Gm;
            block_sum2(b, g, B, Gm);
            if (tid == 0) {
                D.grad_out[k] = 2.0 * B;
                D.grad_out[p + k] = 2.0 * Gm;
            }
        }
    }
}

// --------------------------------------------------------------------------
// Angles -> per-round coefficients and uint8 phase tables (float64 math).

__global__ void __launch_bounds__(256) prep_kernel(const PrepDesc *__restrict__ descs, int *err) {
    const PrepDesc D = descs[blockIdx.x];
    // nb angles per round's mixer (nq qubits for multi-angle, else 1):
    // beta_{k,q} = angles[k nb + q], gamma_k = angles[p nb + k]
    const int nb = D.nq ? D.nq : 1;
    for (int e = threadIdx.x; e < (D.gm_n ? 0 : D.p * nb); e += blockDim.x) {
        const int k = e / nb;
        const double be = D.angles[e], ga = D.angles[D.p * nb + k];
        if (!isfinite(be) || !isfinite(ga)) atomicOr(err, DERR_BAD_ANGLE);
        const RoundCoef c = make_coef(be, ga);
        D.coef[e] = c;
    }
    if (D.gm_n) {
        // general X mixer: its passes keep plain (untwisted) amplitudes, on
        // which the real rotation [[c, s], [-s, c]] is e^{i t Y}; e^{i (pi/4) Y}
        // on every qubit takes X_S to Z_S, so e^{-i b f(X)} is the rotation by
        // t = pi/4 (coefficient 2k, with gamma_k), e^{-i b d_|x|}, and the
        // rotation by t = -pi/4 (coefficient 2k + 1)
        const int n = D.gm_n;
        for (int e = threadIdx.x; e < 2 * D.p; e += blockDim.x) {
            const int k = e >> 1;
            const double ga = D.angles[D.p + k];
            if (!isfinite(D.angles[k]) || !isfinite(ga)) atomicOr(err, DERR_BAD_ANGLE);
            RoundCoef c;
            sincos_turns((e & 1) ? -0.125 : 0.125, &c.sb, &c.cb);  // t = -+pi/4
            c.bmode = 2;
            c.bt = 0.f;
            c.rescale = 0;
            const double g = ga * kInvTwoPi;
            c.g_hi = (float)g;
            c.g_lo = (float)(g - (double)c.g_hi);
            c.b_hi = c.b_lo = c.pad[0] = c.pad[1] = 0.f;
            for (int j = 0; j <= kPassTileBits; j++) c.pw[j] = 1.f;  // direct form: no cosine factors
            D.coef[e] = c;
        }
        for (int e = threadIdx.x; e < D.p * (n + 1); e += blockDim.x) {
            const int k = e / (n + 1), w = e - k * (n + 1);
            const double G = D.wts[w];
            float sn, cs;
            sincos_turns(D.angles[k] * G * kInvTwoPi, &sn, &cs);
            D.wtab[e] = make_float4(cs, -sn, (float)G, 0.f);
        }
    }
    if (D.table) {
        const int tot = D.p * D.tsize;
        for (int e = threadIdx.x; e < tot; e += blockDim.x) {
            const int k = e / D.tsize, cst = e - k * D.tsize;
            // e^{-i gamma c} from the turn count gamma c / (2 pi)
            float s, c;
            sincos_turns(D.angles[D.p * nb + k] * kInvTwoPi * (double)cst, &s, &c);
            D.table[k * kPhaseTable + cst] = make_float2(c, -s);
        }
    }
}

// Fixed-order two-level reduction of the per-(tile, warp) partial sums.
__global__ void __launch_bounds__(256) reduce1_kernel(const RedChunk *__restrict__ chunks, double *level2) {
    __shared__ double red[8];
    const RedChunk C = chunks[blockIdx.x];
    double acc = 0.0;
    for (int i = threadIdx.x; i < C.cnt; i += 256) acc += C.src[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < 8; w++) tot += red[w];
        level2[blockIdx.x] = tot;
    }
}

__global__ void __launch_bounds__(32) reduce2_kernel(const RedOut *__restrict__ outs, const double *level2) {
    const RedOut O = outs[blockIdx.x];
    double acc = 0.0;
    for (int i = threadIdx.x; i < O.n; i += 32) acc += level2[O.first + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (threadIdx.x == 0) *O.out = O.scale * acc;
}

// One thread waits, with the pass kernels' bounded wait, for a barrier phase
// that no thread and no copy ever completes: the wait gives up, the error word
// records it, and the kernel returns.
__global__ void wait_probe_kernel(int *err) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    mbar_init(smem_u32(&bar), 1);
    fence_mbar_init();
    if (!mbar_wait(smem_u32(&bar), 0u)) atomicOr(err, DERR_TIMEOUT);
}

}  // namespace

cudaError_t launch_wait_probe(int *err, cudaStream_t s) {
    wait_probe_kernel<<<1, 32, 0, s>>>(err);
    return cudaGetLastError();
}

int small_max_n() { return kSmallMaxN; }

// xpass_x.cu, xpass_fused.cu, xpass_ma.cu, xpass_gm.cu
cudaError_t launch_xpass_x(int bwd, int cost_dtype, int nbuf, int gather, const PassDesc *d, const uint32_t *tb,
                 int nd, uint32_t tiles, int *err, uint32_t *sched, cudaStream_t s);
cudaError_t launch_xpass_fused(int bwd, int cost_dtype, int nbuf, int gather, const PassDesc *d, const uint32_t *tb,
                 int nd, uint32_t tiles, int *err, uint32_t *sched, cudaStream_t s);
cudaError_t launch_xpass_ma(int bwd, int cost_dtype, int nbuf, int gather, const PassDesc *d, const uint32_t *tb,
                 int nd, uint32_t tiles, int *err, uint32_t *sched, cudaStream_t s);
cudaError_t launch_xpass_gm(int bwd, int cost_dtype, int nbuf, int gather, const PassDesc *d, const uint32_t *tb,
                 int nd, uint32_t tiles, int *err, uint32_t *sched, cudaStream_t s);
cudaError_t launch_xpass(int bwd, int cost_dtype, int nbuf, int var, const PassDesc *d, const uint32_t *tb,
                         int nd, uint32_t tiles, int *err, uint32_t *sched, int gather, int fused, cudaStream_t s) {
    if (tiles == 0) return cudaSuccess;
    if (!sched) return cudaErrorInvalidValue;
    if (fused && var != 0) return cudaErrorInvalidValue;  // round-boundary passes: transverse field only
    if (fused) return launch_xpass_fused(bwd, cost_dtype, nbuf, gather, d, tb, nd, tiles, err, sched, s);
    if (var == 1) return launch_xpass_ma(bwd, cost_dtype, nbuf, gather, d, tb, nd, tiles, err, sched, s);
    if (var == 2) return launch_xpass_gm(bwd, cost_dtype, nbuf, gather, d, tb, nd, tiles, err, sched, s);
    return launch_xpass_x(bwd, cost_dtype, nbuf, gather, d, tb, nd, tiles, err, sched, s);
}

cudaError_t launch_small(const SmallDesc *d, int nd, int cost_dtype, int want_grad, int max_n,
                         int *err, cudaStream_t s) {
    const size_t smem = (size_t)2 * (1u << max_n) * sizeof(float2) + kPhaseTable * sizeof(float2);
    // the opt-in shared-memory size is raised once per kernel to the largest
    // size any call needs (n <= kSmallMaxN)
    const size_t smem_max = (size_t)2 * (1u << kSmallMaxN) * sizeof(float2) + kPhaseTable * sizeof(float2);
    auto go = [&](auto kern, int slot) -> cudaError_t {
        static int attr_done[4][kMaxDevices];
        cudaError_t e = smem_attr_once(kern, (int)smem_max, attr_done[slot]);
        if (e != cudaSuccess) return e;
        kern<<<nd, kSmallThreads, smem, s>>>(d, err);
        return cudaGetLastError();
    };
    if (cost_dtype == 0) return want_grad ? go(small_kernel<0, 1>, 0) : go(small_kernel<0, 0>, 1);
    return want_grad ? go(small_kernel<1, 1>, 2) : go(small_kernel<1, 0>, 3);
}

cudaError_t launch_tile12(const SmallDesc *d, int nd, int cost_dtype, int want_grad, int *err, cudaStream_t s) {
    const size_t smem = (size_t)2 * kTile * sizeof(float2) + kPhaseTable * sizeof(float2) +
                        (size_t)kTile * (cost_dtype == 0 ? 4 : 1);
    auto go = [&](auto kern, int slot) -> cudaError_t {
        static int attr_done[4][kMaxDevices];
        cudaError_t e = smem_attr_once(kern, (int)smem, attr_done[slot]);
        if (e != cudaSuccess) return e;
        kern<<<nd, kNT, smem, s>>>(d, err);
        return cudaGetLastError();
    };
    if (cost_dtype == 0) return want_grad ? go(tile12_kernel<0, 1>, 0) : go(tile12_kernel<0, 0>, 1);
    return want_grad ? go(tile12_kernel<1, 1>, 2) : go(tile12_kernel<1, 0>, 3);
}

cudaError_t launch_prep(const PrepDesc *d, int nd, int *err, cudaStream_t s) {
    prep_kernel<<<nd, 256, 0, s>>>(d, err);
    return cudaGetLastError();
}

cudaError_t launch_reduce(const RedChunk *chunks, int nchunks, double *level2, const RedOut *outs, int nouts,
                          cudaStream_t s) {
    reduce1_kernel<<<nchunks, 256, 0, s>>>(chunks, level2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    reduce2_kernel<<<nouts, 32, 0, s>>>(outs, level2);
    return cudaGetLastError();
}

}  // namespace qg
