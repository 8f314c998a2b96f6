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
// Multi-angle and general X mixers on a whole state in shared memory (n <=
// kSmallMaxN): all p rounds, the expectation and (GRAD) the adjoint sweep in one
// block per unit.  The adjoint undoes each round on psi in place.
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
    // coefficients of round k: one entry per qubit (multi-angle) or two (general X
    // mixer); nb angles per round's mixer
    const int nb = D.wts ? 1 : n, cs = D.wts ? 2 : n;
    // the round's rotations, fetched together (one 96-byte entry per qubit and
    // rotation, in front of each barrier, took 3% of a call)
    __shared__ float2 s_rot[kSmallMaxN];
    auto load_rot = [&](int k) {
        if (!D.wts && tid < n) {
            const RoundCoef &q = D.coef[k * cs + tid];
            s_rot[tid] = make_float2(q.cb, q.sb);
        }
    };

    for (int x = tid; x < N; x += kSmallThreads)
        psi[x] = D.init ? D.init[x] : make_float2(D.amp0, 0.f);
    for (int k = 0; k < p; k++) {
        const RoundCoef cf = D.coef[k * cs];
        __syncthreads();
        load_rot(k);
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
            mix(psi, q, s_rot[q].x, s_rot[q].y);
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
        load_rot(k);
        if (D.wts) {
            float gb = 0.f;
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
            const double GQ = block_sum<kSmallThreads / 32>(gq, s_red);
            if (tid == 0) D.grad_out[k * n + q] = 2.0 * GQ;
        }
        for (int q = 0; q < (D.wts ? 0 : n); q++) {
            __syncthreads();
            mix(lam, q, s_rot[q].x, -s_rot[q].y);
            mix(psi, q, s_rot[q].x, -s_rot[q].y);
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
// Angles -> per-round coefficients and uint8 phase tables (float64 math).

__global__ void __launch_bounds__(256) prep_kernel(const PrepDesc *__restrict__ descs, int *err) {
    const PrepDesc D = descs[blockIdx.x];
    // nb angles per round's mixer (nq qubits for multi-angle, else 1):
    // beta_{k,q} = angles[k nb + q], gamma_k = angles[p nb + k]
    // The coefficients' float64 chain is long: where one warp can form them all at
    // once, it does while the others fill the table, else every thread takes part
    // (always one warp: multi-angle, n = 14, p = 100 114 us, now 54; n = 20, p = 4
    // 13.5, now 8.7).
    const int nb = D.nq ? D.nq : 1;
    const int tid = threadIdx.x, nt = blockDim.x;
    const bool split = D.table && !D.gm_n && D.p * nb <= 32;
    const int tab0 = split ? 32 : 0, nco = split ? 32 : nt;  // table threads from tab0, coefficient threads below nco
    for (int e = tid; !D.gm_n && tid < nco && e < D.p * nb; e += nco) {
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
            // tan form: tan t = +-1 and the even cosine powers are exact, so a half
            // round costs one or two rounded scale factors (the rounded cosine, 2 n
            // times a round, is short of unit length by 1.7e-8 each)
            c.bmode = 0;
            c.bt = (e & 1) ? -1.f : 1.f;
            c.rescale = 0;
            const double g = ga * kInvTwoPi;
            c.g_hi = (float)g;
            c.g_lo = (float)(g - (double)c.g_hi);
            c.b_hi = c.b_lo = c.c_lo = c.pad = 0.f;
            float pw = 1.f;
            for (int j = 0; j <= kPassTileBits; j += 2, pw *= 0.5f) {
                c.pw[j] = pw;
                if (j < kPassTileBits) c.pw[j + 1] = pw * 0.70710678f;
            }
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
    if (D.table && tid >= tab0) {
        // e^{-i gamma c} from the turn count gamma c / (2 pi): a warp takes half a
        // round's table at a time, so gamma's float64 part is formed once for four
        // entries of a lane
        const int lane = tid & 31, step = (nt - tab0) >> 5, half = kPhaseTable / 2;
        for (int w = (tid - tab0) >> 5; w < 2 * D.p; w += step) {
            const int k = w >> 1, c0 = (w & 1) * half;
            const double g = whole_cost_turns(D.angles[D.p * nb + k] * kInvTwoPi);
            const float hi = (float)g, lo = (float)(g - (double)hi);
            for (int c = c0 + lane; c < min(c0 + half, D.tsize); c += 32)
                D.table[k * kPhaseTable + c] = phase_turns(hi, lo, (float)c);
        }
    }
}

// Fixed-order two-level reduction of the per-(tile, warp) partial sums.
__global__ void __launch_bounds__(256) reduce1_kernel(const RedChunk *__restrict__ chunks, double *level2) {
    __shared__ double red[8];
    chain_begin();
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
    chain_begin();
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

cudaError_t launch_prep(const PrepDesc *d, int nd, int *err, cudaStream_t s) {
    prep_kernel<<<nd, 256, 0, s>>>(d, err);
    return cudaGetLastError();
}

cudaError_t launch_reduce(const RedChunk *chunks, int nchunks, double *level2, const RedOut *outs, int nouts,
                          cudaStream_t s) {
    cudaError_t e = launch_chained(reduce1_kernel, nchunks, 256, 0, s, chunks, level2);
    if (e != cudaSuccess) return e;
    return launch_chained(reduce2_kernel, nouts, 32, 0, s, outs, static_cast<const double *>(level2));
}

}  // namespace qg
