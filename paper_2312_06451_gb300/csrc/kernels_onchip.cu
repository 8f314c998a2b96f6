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
// before, 30.3 us in these registers.  Costs fetched 16 bytes at a time, with the
// first coefficients formed meanwhile by one warp, took a further 10% (between
// event pairs 37.0 -> 33.3 us; one <C> at n = 12, p = 3: 16.5 -> 13.4).
#include "onchip.cuh"

namespace qg {
namespace {

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
    beside_begin();
    const SmallDesc D = descs[blockIdx.x];
    const int p = D.p, n = D.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double *ang = D.angles_beta;
    const Pos<NB> T;
    // rotated amplitude bits (n = NB except for the smallest instances)
    const Masks M = {NB > 9 || n >= 8 ? 0xFu : (n > 4 ? (1u << (n - 4)) - 1u : 0u),
                     NB > 9 || n >= 4 ? 0xFu : (1u << n) - 1u,
                     NB > 9 ? (0xFu << (12 - NB)) & 0xFu : (n == 9 ? 8u : 0u)};

    // coefficients of the kChunk rounds that hold round k; the first chunk by one
    // warp while the others fetch the costs
    int chunk = 0;
    auto form = [&](int first, int j) {
        if (first + j < p)
            s_rc[j] = round_consts(make_coef(ang[first + j], ang[p + first + j], COST == 1), M, 0u, 0u);
    };
    auto load_chunk = [&](int k) {
        if (k / kChunk == chunk) return;
        chunk = k / kChunk;
        __syncthreads();
        if (tid < kChunk) form(chunk * kChunk, tid);
        __syncthreads();
    };
    if (tid == 0) s_top = 0;
    __syncthreads();
    if (warp == NW - 1) form(0, lane);
    // cost vector to shared memory (zero beyond 2^n), its largest value
    {
        constexpr int kPer = COST == 0 ? 4 : 16;  // values in 16 bytes
        unsigned top = 0;
        const int have = 1 << n;
        if (have >= kPer) {
#pragma unroll 4
            for (int i = tid; i < N / kPer; i += NT) {
                const uint4 v = i < have / kPer ? __ldg(reinterpret_cast<const uint4 *>(D.cost) + i) : make_uint4(0u, 0u, 0u, 0u);
                reinterpret_cast<uint4 *>(scost)[i] = v;
                if (COST == 1) top = __vmaxu4(top, __vmaxu4(__vmaxu4(v.x, v.y), __vmaxu4(v.z, v.w)));
            }
            top = max(max(top & 255u, (top >> 8) & 255u), max((top >> 16) & 255u, top >> 24));
        } else {
            for (int x = tid; x < N; x += NT) {
                if (COST == 0) {
                    reinterpret_cast<float *>(scost)[x] = x < have ? __ldg(reinterpret_cast<const float *>(D.cost) + x) : 0.f;
                } else {
                    const unsigned c = x < have ? (unsigned)__ldg(reinterpret_cast<const unsigned char *>(D.cost) + x) : 0u;
                    scost[x] = (unsigned char)c;
                    top = max(top, c);
                }
            }
        }
        if (COST == 1) {
            top = __reduce_max_sync(0xffffffffu, top);
            if (lane == 0) atomicMax(&s_top, (int)top);
        }
    }
    bool bad = false;
    for (int k = tid; k < 2 * p; k += NT) bad = bad || !isfinite(ang[k]);
    if (bad) atomicOr(err, DERR_BAD_ANGLE);

    auto coef = [&](int k, float sgn) -> RoundC { return signed_round(s_rc[k % kChunk], sgn); };
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
    __syncthreads();  // costs, their maximum and the first coefficients are there
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
    beside_end();
}

template <int NB>
cudaError_t go_onchip(const SmallDesc *d, int nd, int cost_dtype, int want_grad, int *err, bool beside,
                      cudaStream_t s) {
    const size_t smem = (size_t)Chip<NB>::N * ((want_grad ? 16 : 8) + (cost_dtype == 0 ? 4 : 1));
    auto go = [&](auto kern, int slot) -> cudaError_t {
        static int attr_done[4][kMaxDevices];
        cudaError_t e = smem_attr_once(kern, (int)smem, attr_done[slot]);
        if (e != cudaSuccess) return e;
        if (beside) return launch_chained(kern, nd, Chip<NB>::NT, smem, s, d, err);
        kern<<<nd, Chip<NB>::NT, smem, s>>>(d, err);
        return cudaGetLastError();
    };
    if (cost_dtype == 0) return want_grad ? go(onchip_kernel<NB, 0, 1>, 0) : go(onchip_kernel<NB, 0, 0>, 1);
    return want_grad ? go(onchip_kernel<NB, 1, 1>, 2) : go(onchip_kernel<NB, 1, 0>, 3);
}

}  // namespace

int onchip_class(int n) { return n < 1 || n > kPassTileBits ? 0 : (n < 9 ? 9 : n); }

cudaError_t launch_onchip(const SmallDesc *d, int nd, int cls, int cost_dtype, int want_grad, int *err,
                          bool beside, cudaStream_t s) {
    switch (cls) {
    case 9: return go_onchip<9>(d, nd, cost_dtype, want_grad, err, beside, s);
    case 10: return go_onchip<10>(d, nd, cost_dtype, want_grad, err, beside, s);
    case 11: return go_onchip<11>(d, nd, cost_dtype, want_grad, err, beside, s);
    case 12: return go_onchip<12>(d, nd, cost_dtype, want_grad, err, beside, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace qg
