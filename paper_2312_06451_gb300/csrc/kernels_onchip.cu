// Transverse-field mixer on at most 12 qubits: one CTA per angle set keeps the
// whole state in registers through all p rounds, <C> and the adjoint sweep
// (which undoes each round on psi as well).
//
// 2^NB amplitudes, 16 in each of 2^(NB-4) threads, NB = 9..12 (n < 9: the
// first 2^n of 512, the missing qubits never rotated).  The pass kernels'
// register layouts (xpass.cuh): Q amplitude bits 4..7, R bits 0..3, P the top
// four, of which bits 8 and up are rotated.  Even rounds run Q, R, P and odd
// rounds P, R, Q, so a round starts in the layout the last one ended in and
// costs two transposes, one block barrier and one warp barrier; the phase is
// applied there, and shared memory holds no state between rounds.  A thread
// rewrites the slots it has read, so the transposes need no other barrier.
//
// Latency bounds it (a 1024-amplitude round is a few hundred instructions in
// two warps), so everything once per round is off the threads' path: the
// float64 part of the coefficients is formed by one warp for 32 rounds at a
// time, uint8 phase tables reach only to the largest cost and come from float
// pairs, and the derivatives of a round are summed across warps one round
// later, behind a barrier that is there anyway.
// 256 gradients at n = 10, p = 8, uint8 costs: 95.5 us (a shared-memory sweep
// and two barriers per qubit and vector) and 11.5 us of coefficient preparation
// before, 30.3 us now.
#include "xmix.cuh"

namespace qg {
namespace {

constexpr int kChunk = 32;  // rounds whose coefficients are in shared memory

struct RoundC {
    Rot R;
    int rescale;
    float fq, fr, fp, fe;  // cos factors of the layouts' rotations and of all of them
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

template <int NB, int COST, int GRAD>
__global__ void __launch_bounds__(Chip<NB>::NT) onchip_kernel(const SmallDesc *__restrict__ descs, int *err) {
    constexpr int NT = Chip<NB>::NT, NW = Chip<NB>::NW, N = Chip<NB>::N;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float2 *sa = reinterpret_cast<float2 *>(smem_raw);
    float2 *sl = sa + (GRAD ? N : 0);
    unsigned char *scost = reinterpret_cast<unsigned char *>(sl + N);
    __shared__ RoundC s_rc[kChunk];
    __shared__ float2 stab[kPhaseTable];
    __shared__ double s_red[2][2][NW];  // [round parity][beta, gamma][warp]
    __shared__ int s_top;               // largest uint8 cost
    const SmallDesc D = descs[blockIdx.x];
    const int p = D.p, n = D.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double *ang = D.angles_beta;
    const Pos<NB> T;
    // rotated amplitude bits (n = NB except for the smallest instances)
    const Masks M = {NB > 9 || n >= 8 ? 0xFu : (n > 4 ? (1u << (n - 4)) - 1u : 0u),
                     NB > 9 || n >= 4 ? 0xFu : (1u << n) - 1u,
                     NB > 9 ? (0xFu << (12 - NB)) & 0xFu : (n == 9 ? 8u : 0u)};

    // cost vector to shared memory (zero beyond 2^n), its largest value
    if (tid == 0) s_top = 0;
    __syncthreads();
    {
        int top = 0;
        const int have = 1 << n;
        for (int x = tid; x < N; x += NT) {
            if (COST == 0) {
                reinterpret_cast<float *>(scost)[x] = x < have ? __ldg(reinterpret_cast<const float *>(D.cost) + x) : 0.f;
            } else {
                const int c = x < have ? (int)__ldg(reinterpret_cast<const unsigned char *>(D.cost) + x) : 0;
                scost[x] = (unsigned char)c;
                top = max(top, c);
            }
        }
        if (COST == 1) {
            top = __reduce_max_sync(0xffffffffu, top);
            if (lane == 0) atomicMax(&s_top, top);
        }
    }
    bool bad = false;
    for (int k = tid; k < 2 * p; k += NT) bad = bad || !isfinite(ang[k]);
    if (bad) atomicOr(err, DERR_BAD_ANGLE);

    // coefficients of the kChunk rounds that hold round k
    int chunk = -1;
    auto load_chunk = [&](int k) {
        if (k / kChunk == chunk) return;
        chunk = k / kChunk;
        __syncthreads();
        const int r = chunk * kChunk + tid;
        if (tid < kChunk && r < p) {
            const RoundCoef cf = make_coef(ang[r], ang[p + r]);
            RoundC C;
            const bool tan = cf.bmode == 0;
            C.R.mode = cf.bmode;
            C.R.tt = make_float2(cf.bt, cf.bt);
            C.R.ntt = make_float2(-cf.bt, -cf.bt);
            C.R.c = cf.cb;
            C.R.s = cf.sb;
            C.R.psc = tan ? cf.pw[2] : 1.f;
            C.rescale = tan && cf.rescale ? 1 : 0;
            const int nq = __popc(M.q), nr = __popc(M.r), np = __popc(M.p);
            C.fq = tan ? cf.pw[nq] : 1.f;
            C.fr = tan ? cf.pw[nr] : 1.f;
            C.fp = tan ? cf.pw[np] : 1.f;
            C.fe = tan && !C.rescale ? cf.pw[nq + nr + np] : 1.f;
            C.ghi = cf.g_hi;
            C.glo = cf.g_lo;
            s_rc[tid] = C;
        }
        __syncthreads();
    };
    auto coef = [&](int k, float sgn) -> RoundC {
        RoundC C = s_rc[k % kChunk];
        if (sgn < 0.f) {  // undoing the round
            const float2 t = C.R.tt;
            C.R.tt = C.R.ntt;
            C.R.ntt = t;
            C.R.s = -C.R.s;
        }
        return C;
    };
    auto load_table = [&](const RoundC &C) {
        if (COST == 1) {  // its last readers passed a barrier since
            for (int i = tid; i <= s_top; i += NT) stab[i] = phase_turns(C.ghi, C.glo, (float)i);
            __syncthreads();
        }
    };
    auto phase_of = [&](uint32_t x, const RoundC &C, float &c) -> float2 {
        if (COST == 0) {
            c = reinterpret_cast<const float *>(scost)[x];
            return phase_f32(c, C.ghi, C.glo);
        }
        const unsigned char u = scost[x];
        c = (float)u;
        return stab[u];
    };
    auto at = [&](bool inp, int i) -> uint32_t {
        return inp ? T.lp + ((uint32_t)i << Chip<NB>::kP) : T.lq + ((uint32_t)i << 4);
    };

    // ---------------- initial state in layout Q, twisted basis
    float2 a[16], l[16];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; i++) {
        const uint32_t x = at(false, i);
        const bool in = NB > 9 || x < (1u << n);
        const float2 v = !in ? make_float2(0.f, 0.f) : (D.init ? D.init[x] : make_float2(D.amp0, 0.f));
        a[i] = twist(v, __popc(x));
    }
    // ---------------- forward
    float eacc = 0.f, unused = 0.f;
    for (int k = 0; k < p; k++) {
        load_chunk(k);
        const RoundC C = coef(k, 1.f);
        load_table(C);
        const bool odd = k & 1;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            float c;
            a[i] = cmul(a[i], phase_of(at(odd, i), C, c));
        }
        if (odd) rotate_any<NB, 0, 0>(a, l, sa, sl, C, M, T, unused);
        else rotate_any<NB, 0, 1>(a, l, sa, sl, C, M, T, unused);
    }
    const bool end_p = p & 1;
    auto cost_at = [&](int i) -> float {
        const uint32_t x = at(end_p, i);
        return COST == 0 ? reinterpret_cast<const float *>(scost)[x] : (float)scost[x];
    };
#pragma unroll
    for (int i = 0; i < 16; i++) eacc = fmaf(cost_at(i), fmaf(a[i].x, a[i].x, a[i].y * a[i].y), eacc);
    // sums over the block: float32 within a warp, float64 across warps in a fixed order
    {
        const float t = warp_sum_f(eacc);
        if (lane == 0) s_red[0][0][warp] = (double)t;
    }
    __syncthreads();
    double E = 0.0;
    for (int w = 0; w < NW; w++) E += s_red[0][0][w];
    if (tid == 0) *D.E_out = E;
    if constexpr (GRAD) {
        // lambda_p = (C - <C>) psi_p: the cost shifted by its expectation gives
        // the same gradient without the common component <C> psi in lambda
        const float c0 = (float)E;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const float d = cost_at(i) - c0;
            l[i] = make_float2(d * a[i].x, d * a[i].y);
        }
        __syncthreads();  // s_red is free
        auto flush = [&](int k) {  // round k's derivatives, once every warp's sums are in
            if (tid < 2) {
                double t = 0.0;
                for (int w = 0; w < NW; w++) t += s_red[k & 1][tid][w];
                D.grad_out[tid * p + k] = 2.0 * t;
            }
        };
        for (int k = p - 1; k >= 0; k--) {
            load_chunk(k);
            const RoundC C = coef(k, -1.f);
            const bool odd = k & 1;
            float bacc = 0.f, gacc = 0.f;
            // (the table's last readers passed rotate_any's barrier of the previous round)
            if (odd) rotate_any<NB, 1, 1>(a, l, sa, sl, C, M, T, bacc);
            else rotate_any<NB, 1, 0>(a, l, sa, sl, C, M, T, bacc);
            if (k < p - 1) flush(k + 1);
            load_table(C);
#pragma unroll
            for (int i = 0; i < 16; i++) {
                float c;
                const float2 ph = phase_of(at(odd, i), C, c);
                gacc = fmaf(c - c0, fmaf(l[i].x, a[i].y, -l[i].y * a[i].x), gacc);
                l[i] = cmul_conj(l[i], ph);
                a[i] = cmul_conj(a[i], ph);
            }
            const float t = warp_sum2_f(bacc, gacc);
            if (lane == 0) s_red[k & 1][0][warp] = (double)t;
            if (lane == 16) s_red[k & 1][1][warp] = (double)t;
        }
        __syncthreads();
        flush(0);
    }
}

template <int NB>
cudaError_t go_onchip(const SmallDesc *d, int nd, int cost_dtype, int want_grad, int *err, cudaStream_t s) {
    const size_t smem = (size_t)Chip<NB>::N * ((want_grad ? 16 : 8) + (cost_dtype == 0 ? 4 : 1));
    auto go = [&](auto kern, int slot) -> cudaError_t {
        static int attr_done[4][kMaxDevices];
        cudaError_t e = smem_attr_once(kern, (int)smem, attr_done[slot]);
        if (e != cudaSuccess) return e;
        kern<<<nd, Chip<NB>::NT, smem, s>>>(d, err);
        return cudaGetLastError();
    };
    if (cost_dtype == 0) return want_grad ? go(onchip_kernel<NB, 0, 1>, 0) : go(onchip_kernel<NB, 0, 0>, 1);
    return want_grad ? go(onchip_kernel<NB, 1, 1>, 2) : go(onchip_kernel<NB, 1, 0>, 3);
}

}  // namespace

int onchip_class(int n) { return n < 1 || n > kPassTileBits ? 0 : (n < 9 ? 9 : n); }

cudaError_t launch_onchip(const SmallDesc *d, int nd, int cls, int cost_dtype, int want_grad, int *err,
                          cudaStream_t s) {
    switch (cls) {
    case 9: return go_onchip<9>(d, nd, cost_dtype, want_grad, err, s);
    case 10: return go_onchip<10>(d, nd, cost_dtype, want_grad, err, s);
    case 11: return go_onchip<11>(d, nd, cost_dtype, want_grad, err, s);
    case 12: return go_onchip<12>(d, nd, cost_dtype, want_grad, err, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace qg
