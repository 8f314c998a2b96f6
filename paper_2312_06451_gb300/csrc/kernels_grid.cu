// Transverse-field mixer on 13..20 qubits, all rounds of an angle set in one
// launch: <C> and the gradient of small batches, where the pass
// kernels are bound by launches and half-empty waves, not by bytes.
//
// A set takes 2^H CTAs, H = n - 12, each holding a tile of 2^12 amplitudes in
// registers.  Even rounds start in the tiling A (local qubits 0..11), odd ones
// in B (local qubits 0..11-H and 12..n-1; the CTA index is the other H qubits).
// A round applies the phase, rotates the twelve local qubits (onchip.cuh),
// exchanges tilings through global memory (L2) -- each CTA writes its tile, the
// set's CTAs meet at a barrier, each reads its tile of the other tiling -- and
// rotates the H qubits that became local, in either tiling local bits 12-H..11.
// So a round costs one exchange.  With gradients every exchange has its own
// buffer, which is the checkpoint the adjoint reads psi from; only lambda is
// exchanged again on the way back.
//
// HI (H > 4): the new bits span layouts P and Q (one more transpose), and the
// set's CTAs meet through arrivals counted in global memory (a cooperative
// launch keeps them resident together; the wait is bounded); else P alone, and
// the set is a thread-block cluster with a hardware barrier.  Latency bounds
// both: a meeting in global memory takes about 4000 cycles with the stores it
// publishes, the rotations of a round 1800 forward and 5000 in the adjoint.
// Gradients at p = 6, float32 costs, one set, a call: n = 13 140 -> 62 us, n = 16
// 155 -> 67, n = 18 170 -> 89, n = 20 210 -> 128 (the passes: 2 (p + 1) launches).
#include "onchip.cuh"

namespace qg {
namespace {

constexpr int kNB = kPassTileBits;
using GPos = Pos<kNB>;

// Descriptor of block b (the blocks of descriptor d: begin[d] .. begin[d + 1] - 1).
__device__ __forceinline__ int grid_desc(const uint32_t *__restrict__ begin, int nd, uint32_t b) {
    int lo = 0, hi = nd - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (begin[mid] <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// The set's CTAs meet: what any of them wrote to global memory before its
// arrive is visible to all after the wait.  Up to 16 CTAs (n <= 16) are one
// thread-block cluster and meet at its hardware barrier; more count arrivals in
// global memory (`target`: those that complete the meeting).  wait returns
// false when the bounded wait gave up (the same for the whole block).
template <int HI>
__device__ __forceinline__ void set_arrive(unsigned *bar) {
    if (HI) {
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(bar, 1u);
        }
    } else {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
}
template <int HI>
__device__ __forceinline__ bool set_wait(const unsigned *bar, unsigned target, int *s_fail) {
    if (HI) {
        if (threadIdx.x == 0) {
            const uint64_t t0 = global_ns();
            for (uint32_t i = 0;; i++) {
                unsigned v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
                if (v >= target) break;
                if ((i & 255u) == 255u && global_ns() - t0 > kWaitLimitNs) {
                    *s_fail = 1;
                    break;
                }
            }
            __threadfence();
        }
        __syncthreads();
        return *s_fail == 0;
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    return true;
}

template <int COST, int GRAD, int HI>
__global__ void __launch_bounds__(kNT, 2)
grid_kernel(const GridDesc *__restrict__ descs, const uint32_t *__restrict__ begin, int nd, int *err) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float2 *sa = reinterpret_cast<float2 *>(smem_raw);
    float2 *sl = sa + (GRAD ? kTile : 0);
    unsigned char *scost = reinterpret_cast<unsigned char *>(sl + kTile);  // tiling A, then B
    __shared__ RoundC s_rc[kChunk];
    __shared__ float2 stab[2][kPhaseTable];  // by round parity: filled while the previous round's may still be read
    __shared__ double s_red[2][2][kNW];  // [round parity][beta, gamma][warp]
    __shared__ double s_E;
    __shared__ int s_fail, s_top;
    __shared__ GridDesc D;
    beside_begin();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int di = grid_desc(begin, nd, blockIdx.x);
    for (int i = tid; i < (int)(sizeof(GridDesc) / 4); i += kNT)
        reinterpret_cast<uint32_t *>(&D)[i] = reinterpret_cast<const uint32_t *>(descs + di)[i];
    if (tid == 0) s_fail = s_top = 0;
    __syncthreads();
    const uint32_t t = blockIdx.x - begin[di];  // this CTA's tile
    const int p = D.p, n = D.n, H = n - kNB, c = kNB - H;
    const unsigned ncta = 1u << H;
    const int64_t N = 1ll << n;
    unsigned target = 0;
    const GPos T;
    const Masks M = {0xFu, 0xFu, 0xFu};
    // rotated bits after an exchange, local bits c..11
    const uint32_t hp = HI ? 0xFu : (0xFu << (4 - H)) & 0xFu, hq = HI ? (0xFu << (8 - H)) & 0xFu : 0u;
    const double *ang = D.angles;

    // global element of local index l in tiling g
    auto gidx = [&](int g, uint32_t l) -> uint32_t {
        return g ? ((l & ((1u << c) - 1u)) | (t << c) | ((l >> c) << kNB)) : ((t << kNB) | l);
    };
    auto first_chunk = [&]() {  // one warp: rounds 0 .. kChunk - 1
        if (lane < p) s_rc[lane] = round_consts(make_coef(ang[lane], ang[p + lane], COST == 1), M, hp, hq);
    };
    {  // the tile's costs in both tilings, 16 bytes at a time (both keep local bits 0..3)
        constexpr int kPer = COST == 0 ? 4 : 16, kWords = 2 * kTile / kPer;
        uint4 w[kWords / kNT];
#pragma unroll
        for (int j = 0; j < kWords / kNT; j++) {
            const uint32_t l = (uint32_t)(tid + j * kNT) * kPer;
            const uint32_t x = gidx((int)(l >> kNB), l & (kTile - 1));
            w[j] = __ldg(reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(D.cost) + (size_t)x * (16 / kPer)));
        }
        if (warp == kNW - 1) first_chunk();  // under the loads
        unsigned top = 0;
#pragma unroll
        for (int j = 0; j < kWords / kNT; j++) {
            reinterpret_cast<uint4 *>(scost)[tid + j * kNT] = w[j];
            if (COST == 1) top = __vmaxu4(top, __vmaxu4(__vmaxu4(w[j].x, w[j].y), __vmaxu4(w[j].z, w[j].w)));
        }
        if (COST == 1) {
            top = max(max(top & 255u, (top >> 8) & 255u), max((top >> 16) & 255u, top >> 24));
            top = __reduce_max_sync(0xffffffffu, top);
            if (lane == 0) atomicMax(&s_top, (int)top);
        }
    }
    if (t == 0) {
        bool bad = false;
        for (int k = tid; k < 2 * p; k += kNT) bad = bad || !isfinite(ang[k]);
        if (bad) atomicOr(err, DERR_BAD_ANGLE);
    }

    int chunk = 0;
    auto load_chunk = [&](int k) {  // coefficients of the kChunk rounds that hold round k
        if (k / kChunk == chunk) return;
        chunk = k / kChunk;
        __syncthreads();
        const int r = chunk * kChunk + tid;
        if (tid < kChunk && r < p) s_rc[tid] = round_consts(make_coef(ang[r], ang[p + r], COST == 1), M, hp, hq);
        __syncthreads();
    };
    auto coef = [&](int k, float sgn) -> RoundC { return signed_round(s_rc[k % kChunk], sgn); };
    auto load_table = [&](int k, const RoundC &C) {
        if (COST == 1) {
            for (int i = tid; i <= s_top; i += kNT) stab[k & 1][i] = phase_turns(C.ghi, C.glo, (float)i);
            __syncthreads();
        }
    };
    // layout F of the phases: Q when HI, else P; the local rotations end in the other one
    auto at = [&](bool inp, int i) -> uint32_t { return inp ? T.lp + ((uint32_t)i << 8) : T.lq + ((uint32_t)i << 4); };
    auto cost_f = [&](int g, int i) -> float {
        const uint32_t x = (uint32_t)g * kTile + at(!HI, i);
        return COST == 0 ? reinterpret_cast<const float *>(scost)[x] : (float)scost[x];
    };
    auto phase_of = [&](int g, int i, const RoundC &C, float &cv) -> float2 {  // g: the round's parity
        const uint32_t x = (uint32_t)g * kTile + at(!HI, i);
        if (COST == 0) {
            cv = reinterpret_cast<const float *>(scost)[x];
            return phase_f32(cv, C.ghi, C.glo);
        }
        const unsigned char u = scost[x];
        cv = (float)u;
        return stab[g][u];
    };
    auto store_to = [&](float2 *dst, int g, bool inp, const float2 (&v)[16]) {
#pragma unroll
        for (int i = 0; i < 16; i++) dst[gidx(g, at(inp, i))] = v[i];
    };
    auto load_from = [&](const float2 *src, int g, bool inp, float2 (&v)[16]) {  // L2: other SMs wrote it
#pragma unroll
        for (int i = 0; i < 16; i++) v[i] = __ldcg(src + gidx(g, at(inp, i)));
    };

    // ---------------- initial state, tiling A, layout F, twisted basis
    float2 a[16], l[16];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; i++) {
        const uint32_t x = gidx(0, at(!HI, i));
        a[i] = twist(D.init ? D.init[x] : make_float2(D.amp0, 0.f), __popc(x));
    }
    // ---------------- forward
    float unused = 0.f, one = 1.f;
    load_table(0, coef(0, 1.f));
    for (int k = 0; k < p; k++) {
        const int g = k & 1;
        const RoundC C = coef(k, 1.f);
#pragma unroll
        for (int i = 0; i < 16; i++) {
            float cv;
            a[i] = cmul(a[i], phase_of(g, i, C, cv));
        }
        rotate_any<kNB, 0, HI>(a, l, sa, sl, C, M, T, unused);
        float2 *X = D.X + (GRAD ? (int64_t)k : (int64_t)g) * N;
        store_to(X, g, HI, a);
        set_arrive<HI>(D.bar);
        if (k + 1 < p) {  // the next round's table meanwhile
            load_chunk(k + 1);
            load_table(k + 1, coef(k + 1, 1.f));
        }
        if (!set_wait<HI>(D.bar, target += ncta, &s_fail)) {
            if (tid == 0) atomicOr(err, DERR_TIMEOUT);
            beside_end();
            return;
        }
        load_from(X, g ^ 1, true, a);
        if (C.R.mode == 0) stage_rot<0, 0>(a, l, hp, C.R, one, unused, true);
        else stage_rot<0, 2>(a, l, hp, C.R, one, unused, true);
        if (HI) {
            if (C.rescale) scale_all<0>(a, l, C.hp);
            put_p<kNB>(a, sa, T);
            __syncthreads();
            get_q<kNB>(a, sa, T);
            if (C.R.mode == 0) stage_rot<0, 0>(a, l, hq, C.R, one, unused, true);
            else stage_rot<0, 2>(a, l, hq, C.R, one, unused, true);
            scale_all<0>(a, l, C.rescale ? C.hq : C.he);
        } else {
            scale_all<0>(a, l, C.rescale ? C.hp : C.he);
        }
    }
    // ---------------- <C>: per-CTA partial sums (float32 within a warp, float64 across)
    const int ge = p & 1;
    float eacc = 0.f;
#pragma unroll
    for (int i = 0; i < 16; i++) eacc = fmaf(cost_f(ge, i), fmaf(a[i].x, a[i].x, a[i].y * a[i].y), eacc);
    {
        const float w = warp_sum_f(eacc);
        if (lane == 0) s_red[0][0][warp] = (double)w;
    }
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int w = 0; w < kNW; w++) s += s_red[0][0][w];
        D.part[t] = s;
    }
    set_arrive<HI>(D.bar);
    if (!set_wait<HI>(D.bar, target += ncta, &s_fail)) {
        if (tid == 0) atomicOr(err, DERR_TIMEOUT);
        beside_end();
        return;
    }
    // sum over the set's CTAs of quantity q (warp-wide, a fixed order)
    auto total_of = [&](int64_t q) -> double {
        double s = 0.0;
        for (unsigned j = lane; j < ncta; j += 32) s += __ldcg(D.part + q * ncta + j);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
    };
    if (warp == 0) {
        const double E = total_of(0);
        if (lane == 0) {
            s_E = E;
            if (t == 0) *D.E_out = E;
        }
    }
    if constexpr (GRAD) {
        __syncthreads();
        // lambda_p = (C - <C>) psi_p (the shift keeps the component <C> psi out of lambda)
        const float c0 = (float)s_E;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const float d = cost_f(ge, i) - c0;
            l[i] = make_float2(d * a[i].x, d * a[i].y);
        }
        auto flush = [&](int k) {  // round k's derivatives, once every warp's sums are in
            if (tid < 2) {
                double s = 0.0;
                for (int w = 0; w < kNW; w++) s += s_red[k & 1][tid][w];
                D.part[(int64_t)(1 + tid * p + k) * ncta + t] = s;
            }
        };
        for (int k = p - 1; k >= 0; k--) {
            const int g = k & 1;
            load_chunk(k);
            const RoundC C = coef(k, -1.f);
            float bacc = 0.f, gacc = 0.f, ps = 1.f;
            // undo the H rotations in tiling g ^ 1 (psi is read back below: it
            // only has to reach the last pair terms)
            if (HI) {
                if (C.R.mode == 0) stage_rot<1, 0>(a, l, hq, C.R, ps, bacc, true);
                else stage_rot<1, 2>(a, l, hq, C.R, ps, bacc, true);
                if (C.rescale) {
                    scale_all<1>(a, l, C.hq);
                    ps = 1.f;
                }
                put_q<kNB>(a, sa, T);
                put_q<kNB>(l, sl, T);
                __syncthreads();
                get_p<kNB>(a, sa, T);
                get_p<kNB>(l, sl, T);
            }
            if (C.R.mode == 0) stage_rot<1, 0>(a, l, hp, C.R, ps, bacc, false);
            else stage_rot<1, 2>(a, l, hp, C.R, ps, bacc, false);
            scale_all<0>(l, l, C.rescale ? C.hp : C.he);
            float2 *L = D.lam + (int64_t)g * N;
            store_to(L, g ^ 1, true, l);
            set_arrive<HI>(D.bar);
            load_from(D.X + (int64_t)k * N, g, HI, a);  // this thread's own stores
            load_table(k, C);
            if (!set_wait<HI>(D.bar, target += ncta, &s_fail)) {
                if (tid == 0) atomicOr(err, DERR_TIMEOUT);
                beside_end();
                return;
            }
            if (k < p - 1) flush(k + 1);
            load_from(L, g, HI, l);
            rotate_any<kNB, 1, !HI>(a, l, sa, sl, C, M, T, bacc);
#pragma unroll
            for (int i = 0; i < 16; i++) {
                float cv;
                const float2 ph = phase_of(g, i, C, cv);
                gacc = fmaf(cv - c0, fmaf(l[i].x, a[i].y, -l[i].y * a[i].x), gacc);
                l[i] = cmul_conj(l[i], ph);
                a[i] = cmul_conj(a[i], ph);
            }
            const float w = warp_sum2_f(bacc, gacc);
            if (lane == 0) s_red[k & 1][0][warp] = (double)w;
            if (lane == 16) s_red[k & 1][1][warp] = (double)w;
        }
        __syncthreads();
        flush(0);
        set_arrive<HI>(D.bar);
        if (!set_wait<HI>(D.bar, target += ncta, &s_fail)) {
            if (tid == 0) atomicOr(err, DERR_TIMEOUT);
            beside_end();
            return;
        }
        // the set's derivatives: output o by warp o of the set
        for (int o = (int)t * kNW + warp; o < 2 * p; o += (int)ncta * kNW) {
            const double s = total_of(1 + o);
            if (lane == 0) D.grad_out[o] = 2.0 * s;
        }
    }
    beside_end();
}

template <int COST, int GRAD, int HI>
struct GridLaunch {
    static constexpr size_t smem = (size_t)kTile * (GRAD ? 16 : 8) + (size_t)2 * kTile * (COST == 0 ? 4 : 1);
    static constexpr auto kern = grid_kernel<COST, GRAD, HI>;

    static cudaError_t attrs() {
        static int smem_done[kMaxDevices], wide_done[kMaxDevices];
        cudaError_t e = smem_attr_once(kern, (int)smem, smem_done);
        if (e != cudaSuccess || HI) return e;
        int dev = 0;
        e = cudaGetDevice(&dev);
        if (e != cudaSuccess || __atomic_load_n(&wide_done[dev], __ATOMIC_ACQUIRE)) return e;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess) __atomic_store_n(&wide_done[dev], 1, __ATOMIC_RELEASE);
        return e;
    }
    static void config(cudaLaunchConfig_t &c, cudaLaunchAttribute (&at)[2], uint32_t ctas, int n, bool beside,
                       cudaStream_t s) {
        c = {};
        c.gridDim = dim3(ctas);
        c.blockDim = dim3(kNT);
        c.dynamicSmemBytes = smem;
        c.stream = s;
        c.attrs = at;
        c.numAttrs = 1;
        if (HI) {  // (cooperative launches stay in stream order)
            at[0].id = cudaLaunchAttributeCooperative;
            at[0].val.cooperative = 1;
            return;
        }
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 1u << (n - kNB);
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        if (beside) {
            at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            at[1].val.programmaticStreamSerializationAllowed = 1;
            c.numAttrs = 2;
        }
    }
    static int room(int n) {
        if (attrs() != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        int dev = 0, nsm = 0, per = 0, coop = 0;
        cudaGetDevice(&dev);
        if (HI) {
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
            cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
            if (!coop || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kNT, smem) != cudaSuccess) per = 0;
            return nsm * per;
        }
        cudaLaunchConfig_t c;
        cudaLaunchAttribute at[2];
        config(c, at, 1u << (n - kNB), n, false, nullptr);
        if (cudaOccupancyMaxActiveClusters(&per, kern, &c) != cudaSuccess) {
            cudaGetLastError();
            per = 0;
        }
        return per << (n - kNB);
    }
    static cudaError_t go(const GridDesc *d, const uint32_t *begin, int nd, uint32_t ctas, int n, int *err,
                          bool beside, cudaStream_t s) {
        cudaError_t e = attrs();
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t c;
        cudaLaunchAttribute at[2];
        config(c, at, ctas, n, beside, s);
        return cudaLaunchKernelEx(&c, kern, d, begin, nd, err);
    }
};

template <class F>
auto grid_pick(int cost_dtype, int want_grad, int hi, F &&f) {
    switch ((cost_dtype ? 4 : 0) | (want_grad ? 2 : 0) | (hi ? 1 : 0)) {
    case 0: return f(GridLaunch<0, 0, 0>());
    case 1: return f(GridLaunch<0, 0, 1>());
    case 2: return f(GridLaunch<0, 1, 0>());
    case 3: return f(GridLaunch<0, 1, 1>());
    case 4: return f(GridLaunch<1, 0, 0>());
    case 5: return f(GridLaunch<1, 0, 1>());
    case 6: return f(GridLaunch<1, 1, 0>());
    default: return f(GridLaunch<1, 1, 1>());
    }
}

}  // namespace

int grid_max_ctas(int cost_dtype, int want_grad, int n) {
    return grid_pick(cost_dtype, want_grad, n > kGridClusterN, [&](auto g) { return decltype(g)::room(n); });
}

cudaError_t launch_grid(const GridDesc *d, const uint32_t *begin, int nd, uint32_t ctas, int cost_dtype,
                        int want_grad, int n, int *err, bool beside, cudaStream_t s) {
    return grid_pick(cost_dtype, want_grad, n > kGridClusterN,
                     [&](auto g) { return decltype(g)::go(d, begin, nd, ctas, n, err, beside, s); });
}

}  // namespace qg
