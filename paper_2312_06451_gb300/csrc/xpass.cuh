// The X mixer's pass kernels (see kernels_xmix.cu for the method) and their
// launches, one translation unit per variant (xpass_*.cu).
#pragma once

#include "xmix.cuh"

namespace qg {
namespace {

__device__ __forceinline__ int find_desc(const uint32_t *__restrict__ tile_begin, int ndesc,
                                         uint32_t b) {
    int lo = 0, hi = ndesc - 1, found = -1;
    while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        if (tile_begin[mid] <= b) {
            found = mid;
            lo = mid + 1;
        } else {
            hi = mid - 1;
        }
    }
    if (found >= 0 && b >= tile_begin[found + 1]) found = -1;
    return found;
}

// ----------------------------------------------------------- TMA / mbarrier
// (mbarrier and bulk-copy wrappers: bulk.cuh)
// One TMA tensor copy of a 4-d box (coordinates c0..c3) global -> shared.
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void *tmap, int c0, int c1, int c2, int c3,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
        "l"(tmap), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}

// --------------------------------------------------------------------------
// The pass kernel (persistent).  A tile is 2^12 amplitudes; 256 threads hold
// 16 amplitudes each (per vector).  Tile-local bit j is global bit gpos[j]
// (bits 0..c-1 are the contiguous run; a gathered tile rotates bits c..11, a
// contiguous one all twelve).  Register layouts (local bits):
//   P: amplitude bits -> 8..11, lanes -> 0..4, warps -> 5..7     (every store)
//   Q: amplitude bits -> 4..7, lanes -> 0..3 and 8, warps -> 9..11
//   R: amplitude bits -> 0..3, lanes -> 4..8, warps -> 9..11     (contiguous only)
// Each layout rotates its amplitude bits.  A pass visits ST of them:
//   ST 1  c >= 8: P alone, no transpose
//   ST 2  c = 4..7: Q, P (one transpose; the rotated bits 4..11 are two
//         layouts' worth, so gathered tiles need no third one)
//   ST 3  contiguous: Q, R, P (two)
// A round-boundary pass starts at P, reaches Q, applies the phase there and
// goes back the same way.
//
// Transposes go through the tile's own buffer.  P and Q access it in natural
// order: 16 lanes cover bits 0..3, one 128-byte line, so 8-byte accesses are
// conflict free, the amplitude bits are immediate offsets, and a thread writes
// back the very slots it read -- one barrier a transpose.  R's 16-byte pairs
// need the 128-byte swizzle (sw) on both sides.  Q and R hold the same 512
// amplitudes per warp, so moving between them takes a warp barrier only.
//
// Shared-memory traffic, instructions and registers bound the adjoint, not
// HBM: an earlier layout rotated {0, 9..11}, {1..4}, {5..8} for every tile and
// so took two transposes (four at a round boundary) whatever was rotated.
// n = 28, p = 8 gradient, float32 costs: 43.6 -> 39.1 ms; 4 sets of <C> at n = 24,
// p = 10, uint8 costs: 4.69 -> 4.05 ms; 64 uneven gradients (n = 14..22, p = 6):
// 7.5 -> 6.2 ms (all with chained launches).
//
// Pipeline: warp 0 loads the tiles of this CTA with TMA copies into NBUF
// shared-memory buffers (completion on one mbarrier per buffer; the tile's
// descriptor index and base offset travel with it through the barrier); the
// buffer goes back to the loader as soon as its last layout has been read.

template <int BWD, int COST>
struct PassGeom {
    static constexpr uint32_t kPsiB = kTile * 8;
    static constexpr uint32_t kCostB = kTile * (COST == 0 ? 4 : 1);
    static constexpr uint32_t kBufB = kPsiB * (BWD ? 2 : 1) + kCostB;
    static constexpr uint32_t kStashB = (BWD && COST == 0) ? kTile * 4 : 0;  // after the buffers
    static constexpr uint32_t kHead = 256 + kPhaseTable * 8;  // barriers, tile info, phase table
};

struct TileInfo {
    int di;
    uint32_t tl;    // tile index within the descriptor
    uint32_t base;  // global element offset of local index 0
    uint32_t pad;
};

template <int BWD>
__device__ __forceinline__ bool needs_cost(uint32_t flags) {
    return BWD ? (flags & (PF_LAM_FROM_C | PF_PHASE | PF_FUSED)) != 0 : (flags & (PF_PHASE | PF_E | PF_FUSED)) != 0;
}

// Descriptor of tile t for the loader.  A CTA claims its tiles in
// increasing order, so the search walks forward from the previous answer
// (`cursor`, warp 0's own) for a few descriptors, and bisects when the claim
// jumped further (small descriptors: a CTA's claims are about a grid apart).
__device__ __forceinline__ int next_desc(const uint32_t *__restrict__ tile_begin, int ndesc, uint32_t t,
                                         int &cursor) {
    int di = cursor;
    if (di < 0 || di >= ndesc || t < tile_begin[di]) {
        di = find_desc(tile_begin, ndesc, t);
    } else {
        int steps = 0;
        while (di < ndesc && t >= tile_begin[di + 1] && steps < 4) {
            di++;
            steps++;
        }
        if (di < ndesc && t >= tile_begin[di + 1]) di = find_desc(tile_begin, ndesc, t);
    }
    if (di >= ndesc) di = -1;
    if (di >= 0) cursor = di;
    return di;
}

// Global offset of local index 0 of tile tl: the tile index's bits fill the
// free qubits in increasing order, which are c..lo-1 and lo+h..n-1 for a pass
// keeping qubits 0..c-1 contiguous and gathering lo..lo+h-1 (h = T - c).
__device__ __forceinline__ uint32_t tile_base(uint32_t tl, int c, int lo) {
    if (c >= kT) return tl << kT;
    const int h = kT - c, nb = lo - c;
    const uint32_t hi = lo + h < 32 ? (tl >> nb) << (lo + h) : 0u;  // nothing above a top block
    return ((tl & ((1u << nb) - 1u)) << c) | hi;
}

// Warp 0: start the loads of tile t into buffer buf (all 32 lanes call).
template <int BWD, int COST>
// The descriptor the CTA is working on sits in shared memory (Ds) with its
// tile range and index in s_tr = {first tile, end tile, index}; a next tile in
// that range (the common case) needs no global load at all.
__device__ __forceinline__ void issue_tile(uint32_t t, unsigned char *buf, uint32_t bar, TileInfo *info,
                                           const PassDesc *__restrict__ descs,
                                           const uint32_t *__restrict__ tile_begin, int ndesc, int &cursor,
                                           const PassDesc *Ds, const uint32_t *s_tr) {
    using G = PassGeom<BWD, COST>;
    const int lane = threadIdx.x & 31;
    const bool here = Ds && t >= s_tr[0] && t < s_tr[1];
    const int di = here ? (int)s_tr[2] : next_desc(tile_begin, ndesc, t, cursor);
    fence_proxy_async();
    if (di < 0) {
        if (lane == 0) {
            info->di = -1;
            mbar_arrive_tx(bar, 0);
        }
        return;
    }
    const PassDesc *Dg = here ? Ds : descs + di;
    const uint32_t flags = Dg->flags;
    const int c = Dg->c;
    const uint32_t tl = t - (here ? s_tr[0] : tile_begin[di]);
    const uint32_t base = tile_base(tl, c, Dg->gpos[c < kT ? c : 0]);
    const bool ld_psi = BWD || !(flags & PF_GEN_INIT);
    const bool ld_lam = BWD && !(flags & PF_LAM_FROM_C);
    const bool ld_cost = needs_cost<BWD>(flags);
    const uint32_t bytes = (ld_psi ? G::kPsiB : 0) + (ld_lam ? G::kPsiB : 0) + (ld_cost ? G::kCostB : 0);
    if (lane == 0) {
        info->di = di;
        info->tl = tl;
        info->base = base;
        mbar_arrive_tx(bar, bytes);
    }
    __syncwarp();
    const uint32_t sb = smem_u32(buf);
    const float2 *psi = Dg->psi_in;
    const float2 *lam = Dg->lam_in;
    const unsigned char *cost = static_cast<const unsigned char *>(Dg->cost);
    constexpr uint32_t cb = COST == 0 ? 4 : 1;
    // Gathered tile with a tensor map: one TMA op per operand.  Box = 2^c
    // contiguous elements x 2^(T-c) rows at stride 2^lo; tile coordinates
    // are the free bits below lo (dim 1) and above lo + T - c (dim 3).
    const void *tm_psi = Dg->tm_psi, *tm_lam = Dg->tm_lam, *tm_cost = Dg->tm_cost;
    bool seg_psi = ld_psi, seg_lam = ld_lam, seg_cost = ld_cost;
    if (lane == 0 && (tm_psi || tm_lam || tm_cost)) {
        const int lo = Dg->gpos[c];  // gathered pass: lo > c
        const int c1 = (int)(tl & ((1u << (lo - c)) - 1u)), c3 = (int)(tl >> (lo - c));
        if (ld_psi && tm_psi) tma_load_4d(sb, tm_psi, 0, c1, 0, c3, bar);
        if (ld_lam && tm_lam) tma_load_4d(sb + G::kPsiB, tm_lam, 0, c1, 0, c3, bar);
        if (ld_cost && tm_cost) tma_load_4d(sb + G::kPsiB * (BWD ? 2 : 1), tm_cost, 0, c1, 0, c3, bar);
    }
    seg_psi = seg_psi && !tm_psi;
    seg_lam = seg_lam && !tm_lam;
    seg_cost = seg_cost && !tm_cost;
    if (!(seg_psi || seg_lam || seg_cost)) return;
    const int nseg = 1 << (kT - c);
    const uint32_t segn = 1u << c;
    const int glo = c < kT ? Dg->gpos[c] : 0;  // segment s starts at base + s 2^lo
    for (int s = lane; s < nseg; s += 32) {
        const uint32_t off = base + ((uint32_t)s << glo);
        const uint32_t ls = (uint32_t)s << c;
        if (seg_psi) bulk_g2s(sb + ls * 8, psi + off, segn * 8, bar);
        if (seg_lam) bulk_g2s(sb + G::kPsiB + ls * 8, lam + off, segn * 8, bar);
        if (seg_cost)
            bulk_g2s(sb + G::kPsiB * (BWD ? 2 : 1) + ls * cb, cost + (size_t)off * cb, segn * cb, bar);
    }
}

// Tiles are handed out dynamically: the first NBUF per CTA statically
// (blockIdx + k gridDim), the rest from a per-launch counter in the order CTAs
// ask for them, so CTAs that run faster take more tiles and the launch ends
// with every CTA within about one tile of the others.  Partial sums sit in
// per-tile slots, so the results do not depend on which CTA took a tile.
// A claim past the last tile posts an end marker through the buffer's barrier.
constexpr int kTileEnd = -2;

__device__ __forceinline__ void post_end(uint32_t bar, TileInfo *info) {
    if ((threadIdx.x & 31) == 0) {
        info->di = kTileEnd;
        mbar_arrive_tx(bar, 0);
    }
}

// Warp 0: claim the next tile for a buffer and start its loads.
template <int BWD, int COST, int NBUF>
__device__ __forceinline__ void claim_issue(unsigned char *buf, uint32_t bar, uint32_t *sched, uint32_t total,
                                            TileInfo *info, const PassDesc *__restrict__ descs,
                                            const uint32_t *__restrict__ tile_begin, int ndesc, int &cursor,
                                            const PassDesc *Ds, const uint32_t *s_tr) {
    uint32_t tn = 0;
    if ((threadIdx.x & 31) == 0) tn = (uint32_t)NBUF * gridDim.x + atomicAdd(sched, 1u);
    tn = __shfl_sync(0xffffffffu, tn, 0);
    if (tn < total) issue_tile<BWD, COST>(tn, buf, bar, info, descs, tile_begin, ndesc, cursor, Ds, s_tr);
    else post_end(bar, info);
}

// Constants of the descriptor being processed, in shared memory (one per
// round of a boundary pass).
struct PassConst {
    Rot R;
    float ghi, glo, amp0;
    float c0;                  // adjoint: cost shift (C - c0 as the operator)
    float fsq, fsr, fsp, fse;  // cos b factors of the Q, R and P rotations, and of all of them
    uint32_t flags, mq, mp;    // pass flags; rotated amplitude bits in Q and P
    int rescale;
};

// A thread's place in the three layouts (local index of amplitude 0).
struct ThreadPos {
    uint32_t lp, lq, lr;
};
__device__ __forceinline__ ThreadPos thread_pos() {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    return {lane | (warp << 5), (lane & 15u) | ((lane >> 4) << 8) | (warp << 9), (lane << 4) | (warp << 9)};
}
// The 128-byte swizzle: bits 1..3 flipped by bits 4..6 (16-byte pairs stay whole).
__device__ __forceinline__ uint32_t sw(uint32_t l) { return l ^ (((l >> 4) & 7u) << 1); }

template <int SWZ>
__device__ __forceinline__ void get_p(float2 (&v)[16], const float2 *s, uint32_t lp) {
    const float2 *q = s + (SWZ ? sw(lp) : lp);
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = q[i << 8];
}
template <int SWZ>
__device__ __forceinline__ void put_p(const float2 (&v)[16], float2 *s, uint32_t lp) {
    float2 *q = s + (SWZ ? sw(lp) : lp);
#pragma unroll
    for (int i = 0; i < 16; i++) q[i << 8] = v[i];
}
template <int SWZ>
__device__ __forceinline__ void get_q(float2 (&v)[16], const float2 *s, uint32_t lq) {
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = s[(SWZ ? lq ^ ((i & 7) << 1) : lq) + (i << 4)];
}
template <int SWZ>
__device__ __forceinline__ void put_q(const float2 (&v)[16], float2 *s, uint32_t lq) {
#pragma unroll
    for (int i = 0; i < 16; i++) s[(SWZ ? lq ^ ((i & 7) << 1) : lq) + (i << 4)] = v[i];
}
__device__ __forceinline__ void get_r(float2 (&v)[16], const float2 *s, uint32_t lr) {
#pragma unroll
    for (int r = 0; r < 8; r++) {
        const float4 w = *reinterpret_cast<const float4 *>(s + (sw(lr) ^ (r << 1)));
        v[2 * r] = make_float2(w.x, w.y);
        v[2 * r + 1] = make_float2(w.z, w.w);
    }
}
__device__ __forceinline__ void put_r(const float2 (&v)[16], float2 *s, uint32_t lr) {
#pragma unroll
    for (int r = 0; r < 8; r++)
        *reinterpret_cast<float4 *>(s + (sw(lr) ^ (r << 1))) =
            make_float4(v[2 * r].x, v[2 * r].y, v[2 * r + 1].x, v[2 * r + 1].y);
}

// Global element offset of local index l within a tile.
__device__ __forceinline__ uint32_t tile_offset(uint32_t l, int c, int lo) {
    return c >= kT ? l : ((l & ((1u << c) - 1u)) | ((l >> c) << lo));
}

// One tile: rotations in the layouts Q, R, P (see above), fused epilogue.
// MODE is the rotation form (0 tan, 2 direct); the forms are separate copies
// of this body so the common one stays compact in the instruction cache.
// Optional work (initial state, phase, epilogue) sits in loops of its own that
// are skipped as a whole when a pass does not need them.  QF: Q rotates all
// four bits (c = 4 or contiguous), known at compile time.
template <int BWD, int COST, int NBUF, int MODE, int VAR, int ST, int QF>
__device__ __forceinline__ void tile_body(const PassConst &K, const PassDesc &D, const uint32_t (&rs)[4], uint32_t gp,
                                          const float2 *stab, const float4 *s_rot, const float4 *s_w,
                                          unsigned char *bufs, int b, uint32_t bar, uint32_t *sched,
                                          uint32_t total, uint32_t base, uint32_t tl, TileInfo *tinfo,
                                          const PassDesc *__restrict__ descs,
                                          const uint32_t *__restrict__ tile_begin, int ndesc, int &cursor,
                                          const uint32_t *s_tr) {
    using G = PassGeom<BWD, COST>;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const ThreadPos T = thread_pos();
    const uint32_t lf = ST == 1 ? T.lp : T.lq;  // first layout
    constexpr int kF = ST == 1 ? 8 : 4;
    const uint32_t flags = K.flags;
    const uint32_t mq = QF ? 0xFu : K.mq, mp = ST >= 2 ? 0xFu : K.mp;

    float2 *sp = reinterpret_cast<float2 *>(bufs + b * G::kBufB);
    float2 *sl = sp + kTile;
    const unsigned char *scost = bufs + b * G::kBufB + G::kPsiB * (BWD ? 2 : 1);
    float2 a[16];
    float2 l[16];
    float pscale = 1.f, bacc = 0.f;
    constexpr bool MA = VAR == 1;  // multi-angle
    constexpr bool GM = VAR == 2;  // general X mixer: fixed half-round rotations, no pair terms
    float bq[MA ? 12 : 1];         // multi-angle: pair terms per local bit
#pragma unroll
    for (int j = 0; j < (MA ? 12 : 1); j++) bq[j] = 0.f;

    // ---------------- read the landed tile
    if (!BWD && (flags & PF_GEN_INIT)) {
        if (GM) {  // the general mixer's passes keep plain amplitudes
#pragma unroll
            for (int i = 0; i < 16; i++) a[i] = make_float2(K.amp0, 0.f);
        } else {
            // uniform state in the twisted basis: amp0 * (-i)^{|x|}, |x| = |base| + |local|
            const float2 a0 = twist(make_float2(K.amp0, 0.f), __popc(base) + __popc(lf));
#pragma unroll
            for (int i = 0; i < 16; i++) a[i] = twist(a0, __popc(i));
        }
    } else {
        if (ST == 1) get_p<0>(a, sp, T.lp);
        else get_q<0>(a, sp, T.lq);
        if (!GM && !BWD && (flags & PF_TWIST_IN)) {
            const float2 w0 = twist(make_float2(1.f, 0.f), __popc(base) + __popc(lf));
#pragma unroll
            for (int i = 0; i < 16; i++) a[i] = cmul(twist(a[i], __popc(i)), w0);
        }
    }
    if (BWD && !(flags & PF_LAM_FROM_C)) {
        if (ST == 1) get_p<0>(l, sl, T.lp);
        else get_q<0>(l, sl, T.lq);
    }
    if (BWD ? (flags & PF_LAM_FROM_C) : (flags & PF_PHASE)) {
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const uint32_t ci = lf + ((uint32_t)i << kF);
            const float C = COST == 0 ? reinterpret_cast<const float *>(scost)[ci] : (float)scost[ci];
            if (BWD) {
                const float d = C - K.c0;
                l[i] = __fmul2_rn(make_float2(d, d), a[i]);
            } else {
                a[i] = cmul(a[i], COST == 0 ? phase_f32(C, K.ghi, K.glo) : stab[scost[ci]]);
            }
        }
    }
    if (GM && !BWD && (flags & PF_WDIAG)) {
        // general X mixer: e^{-i b G(|x|)} on the global index x of every amplitude
        const int c = D.c, lo = c < kT ? D.gpos[c] : 0;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const float4 t = s_w[__popc(base + tile_offset(lf + ((uint32_t)i << kF), c, lo))];
            a[i] = cmul(a[i], make_float2(t.x, t.y));
        }
    }
    // ---------------- Q (and R), back through the buffer to P
    if constexpr (ST >= 2) {
        if constexpr (MA) stage_rot_ma<BWD, MODE, 4, 5, 6, 7>(a, l, mq, s_rot, bq, pscale, true);
        else stage_rot<BWD, MODE>(a, l, mq, K.R, pscale, bacc, true, !GM);
        if (K.rescale) {
            scale_all<BWD>(a, l, K.fsq);
            pscale = 1.f;
        }
        if constexpr (ST == 3) {
            __syncwarp();  // the warp's 512 amplitudes are read: rewrite them swizzled
            put_q<1>(a, sp, T.lq);
            if (BWD) put_q<1>(l, sl, T.lq);
            __syncwarp();
            get_r(a, sp, T.lr);
            if (BWD) get_r(l, sl, T.lr);
            if constexpr (MA) stage_rot_ma<BWD, MODE, 0, 1, 2, 3>(a, l, 0xFu, s_rot, bq, pscale, true);
            else stage_rot<BWD, MODE>(a, l, 0xFu, K.R, pscale, bacc, true, !GM);
            if (K.rescale) {
                scale_all<BWD>(a, l, K.fsr);
                pscale = 1.f;
            }
            put_r(a, sp, T.lr);
            if (BWD) put_r(l, sl, T.lr);
        } else {
            put_q<0>(a, sp, T.lq);
            if (BWD) put_q<0>(l, sl, T.lq);
        }
        __syncthreads();
        get_p<ST == 3>(a, sp, T.lp);
        if (BWD) get_p<ST == 3>(l, sl, T.lp);
    }
    // Cost values of this thread's P amplitudes, read before the buffer goes
    // back to the loader: uint8 costs packed four to a register; float costs of
    // the adjoint copied to this thread's own slots of a stash that the loader
    // never writes (16 live registers there cause spills).
    const bool epi_c = BWD ? (flags & PF_PHASE) : (flags & PF_E);
    float cst[16];
    uint32_t cpk[4];
    float *stash = reinterpret_cast<float *>(bufs + NBUF * G::kBufB);
    if (epi_c) {
        if (COST == 1) {
#pragma unroll
            for (int q = 0; q < 4; q++) cpk[q] = 0u;
#pragma unroll
            for (int i = 0; i < 16; i++) cpk[i >> 2] |= (uint32_t)scost[T.lp + (i << 8)] << (8 * (i & 3));
        } else if (BWD) {
#pragma unroll
            for (int i = 0; i < 16; i++)
                stash[T.lp + (i << 8)] = reinterpret_cast<const float *>(scost)[T.lp + (i << 8)];
        } else {
#pragma unroll
            for (int i = 0; i < 16; i++) cst[i] = reinterpret_cast<const float *>(scost)[T.lp + (i << 8)];
        }
    }
    auto cost_at = [&](int i) -> float {
        if (COST == 1) return (float)((cpk[i >> 2] >> (8 * (i & 3))) & 255u);
        if (BWD) return stash[T.lp + (i << 8)];
        return cst[i];
    };
    // the buffer is consumed: start the tile NBUF ahead
    __syncthreads();
    if (warp == 0)
        claim_issue<BWD, COST, NBUF>(bufs + b * G::kBufB, bar, sched, total, &tinfo[b], descs, tile_begin, ndesc,
                                     cursor, &D, s_tr);
    // psi after the last rotation is needed only when it is stored or meets the
    // phase epilogue (the adjoint with per-pass checkpoints stores lambda only)
    const bool psi_live = !BWD || D.psi_out != nullptr || (flags & PF_PHASE) || (GM && (flags & PF_WDIAG));
    if constexpr (MA) stage_rot_ma<BWD, MODE, 8, 9, 10, 11>(a, l, mp, s_rot, bq, pscale, psi_live);
    else stage_rot<BWD, MODE>(a, l, mp, K.R, pscale, bacc, psi_live, !GM);
    scale_all<BWD>(a, l, K.rescale ? K.fsp : K.fse);

    // ---------------- fused epilogue, coalesced store
    // offset of amplitude i: i rs[0] where the four amplitude bits are
    // consecutive global bits (ST >= 2)
    auto off = [&](int i) -> uint32_t {
        if (ST >= 2) return (uint32_t)i * rs[0];
        return ((i & 1) ? rs[0] : 0) + ((i & 2) ? rs[1] : 0) + ((i & 4) ? rs[2] : 0) + ((i & 8) ? rs[3] : 0);
    };
    const uint32_t g = base + gp;
    if (GM && BWD && (flags & PF_WDIAG)) {
        // general X mixer: the beta partial sum_x G(|x|) Im(conj(lam) psi) in
        // the frame between the two half rounds, then the diagonal undone
        float wacc = 0.f;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const float4 t = s_w[__popc(g + off(i))];
            wacc = fmaf(t.z, fmaf(l[i].x, a[i].y, -l[i].y * a[i].x), wacc);
            l[i] = cmul_conj(l[i], make_float2(t.x, t.y));
            if (D.psi_out) a[i] = cmul_conj(a[i], make_float2(t.x, t.y));
        }
        bacc += wacc;
    }
    float eacc = 0.f;
    if (epi_c) {
        if (!BWD) {
#pragma unroll
            for (int i = 0; i < 16; i++) eacc = fmaf(cost_at(i), fmaf(a[i].x, a[i].x, a[i].y * a[i].y), eacc);
        } else {
            const bool un_psi = flags & PF_UNPHASE_PSI;
#pragma unroll
            for (int i = 0; i < 16; i++) {
                const float C = cost_at(i);
                const float2 ph = COST == 0 ? phase_f32(C, K.ghi, K.glo) : stab[(int)C];
                eacc = fmaf(C - K.c0, fmaf(l[i].x, a[i].y, -l[i].y * a[i].x), eacc);
                l[i] = cmul_conj(l[i], ph);
                if (un_psi) a[i] = cmul_conj(a[i], ph);
            }
        }
    }
    if (D.psi_out) {
        float2 *out = D.psi_out + g;
#pragma unroll
        for (int i = 0; i < 16; i++) __stcs(out + off(i), a[i]);
    }
    if (BWD && D.lam_out) {
        float2 *out = D.lam_out + g;
#pragma unroll
        for (int i = 0; i < 16; i++) __stcs(out + off(i), l[i]);
    }
    // per-warp partial sums: slot tile * 8 + warp (no block barrier)
    if (BWD) {
        if constexpr (MA) {  // slot (local bit j, tile, warp); j's total in lane 2j
            float v[16];
#pragma unroll
            for (int j = 0; j < 16; j++) v[j] = j < 12 ? bq[j < 12 ? j : 0] : 0.f;
            const float tb = warp_sum16_f(v);
            const uint32_t j = (uint32_t)lane >> 1;
            if (!(lane & 1) && j < 12u && ((D.active >> j) & 1u) && D.part_beta)
                D.part_beta[((size_t)j * D.ntiles + tl) * kNW + warp] = (double)tb;
            if (flags & PF_PHASE) {
                const float tg = warp_sum_f(eacc);
                if (lane == 0 && D.part_gamma) D.part_gamma[tl * kNW + warp] = (double)tg;
            }
        } else {  // beta's total in lane 0, gamma's in lane 16
            const float t = warp_sum2_f(bacc, eacc);
            if (lane == 0 && D.part_beta) D.part_beta[tl * kNW + warp] = (double)t;
            if ((flags & PF_PHASE) && lane == 16 && D.part_gamma) D.part_gamma[tl * kNW + warp] = (double)t;
        }
    } else if (flags & PF_E) {
        const float te = warp_sum_f(eacc);
        if (lane == 0 && D.part_E) D.part_E[tl * kNW + warp] = (double)te;
    }
}

// Rotation and phase constants of one round for the tiles of a descriptor
// (K.mq and K.mp must be set): rotation form, the cos factors per layout and
// of the whole pass.  `all`: a contiguous tile (R rotates its four bits too).
__device__ __forceinline__ void set_round(PassConst &K, const RoundCoef &cf, float sgn, bool all) {
    const bool tan = cf.bmode == 0;
    K.R.mode = cf.bmode;
    K.R.tt = make_float2(sgn * cf.bt, sgn * cf.bt);
    K.R.ntt = make_float2(-sgn * cf.bt, -sgn * cf.bt);
    K.R.c = cf.cb;
    K.R.s = sgn * cf.sb;
    K.R.psc = tan ? cf.pw[2] : 1.f;
    K.rescale = (tan && cf.rescale) ? 1 : 0;
    const int nq = __popc(K.mq), np = __popc(K.mp), nr = all ? 4 : 0;
    K.fsq = tan ? cf.pw[nq] : 1.f;
    K.fsr = tan ? cf.pw[nr] : 1.f;
    K.fsp = tan ? cf.pw[np] : 1.f;
    K.fse = tan && !K.rescale ? cf.pw[nq + nr + np] : 1.f;
    K.ghi = cf.g_hi;
    K.glo = cf.g_lo;
}

// Round-boundary tile (PF_FUSED).  The tile's bits are the last qubit group
// of round k and the first of round k+1, so one pass applies round k's
// rotations, the phase of round k+1 and round k+1's rotations (forward), or
// undoes them in reverse order with both rounds' pair terms and the gamma
// partial in between (adjoint).  The layouts run P, R, Q, the phase at Q (P
// for ST 1; cost values in the tile buffer, natural order), then Q, R, P.  KA
// is the round applied first (forward: k; adjoint: k+1), KB the second; KP
// holds the phase (round k+1).
template <int BWD, int COST, int NBUF, int MA, int MB, int ST, int QF>
__device__ __forceinline__ void tile_body_fused_impl(const PassConst &KA, const PassConst &KB, const PassConst &KP,
                                                     const uint32_t (&rs)[4], uint32_t gp,
                                                     const PassDesc &D, const float2 *stab, unsigned char *bufs, int b,
                                                     uint32_t bar, uint32_t *sched, uint32_t total, uint32_t base,
                                                     uint32_t tl, TileInfo *tinfo, const PassDesc *__restrict__ descs,
                                                     const uint32_t *__restrict__ tile_begin, int ndesc, int &cursor,
                                                     const uint32_t *s_tr) {
    using G = PassGeom<BWD, COST>;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const ThreadPos T = thread_pos();
    float2 *sp = reinterpret_cast<float2 *>(bufs + b * G::kBufB);
    float2 *sl = sp + kTile;
    const unsigned char *scost = bufs + b * G::kBufB + G::kPsiB * (BWD ? 2 : 1);
    float2 a[16], l[16];
    float pscale = 1.f, bA = 0.f, bB = 0.f, eacc = 0.f;
    const uint32_t mq = QF ? 0xFu : KA.mq, mp = ST >= 2 ? 0xFu : KA.mp;

    // ---------------- round A: P, R, Q
    get_p<0>(a, sp, T.lp);
    if (BWD) get_p<0>(l, sl, T.lp);
    stage_rot<BWD, MA>(a, l, mp, KA.R, pscale, bA, true);
    if constexpr (ST >= 2) {
        if (KA.rescale) {
            scale_all<BWD>(a, l, KA.fsp);
            pscale = 1.f;
        }
        if (ST == 3) __syncwarp();  // swizzled slots: those of the same 16 lanes
        put_p<ST == 3>(a, sp, T.lp);
        if (BWD) put_p<ST == 3>(l, sl, T.lp);
        __syncthreads();
        if constexpr (ST == 3) {
            get_r(a, sp, T.lr);
            if (BWD) get_r(l, sl, T.lr);
            stage_rot<BWD, MA>(a, l, 0xFu, KA.R, pscale, bA, true);
            if (KA.rescale) {
                scale_all<BWD>(a, l, KA.fsr);
                pscale = 1.f;
            }
            put_r(a, sp, T.lr);
            if (BWD) put_r(l, sl, T.lr);
            __syncwarp();
        }
        get_q<ST == 3>(a, sp, T.lq);
        if (BWD) get_q<ST == 3>(l, sl, T.lq);
        stage_rot<BWD, MA>(a, l, mq, KA.R, pscale, bA, true);
    }
    scale_all<BWD>(a, l, KA.rescale ? (ST >= 2 ? KA.fsq : KA.fsp) : KA.fse);
    pscale = 1.f;

    // ---------------- the phase of round k+1 between the two rounds
    {
        const uint32_t lx = ST == 1 ? T.lp : T.lq;
        constexpr int kX = ST == 1 ? 8 : 4;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const uint32_t ci = lx + ((uint32_t)i << kX);
            const float C = COST == 0 ? reinterpret_cast<const float *>(scost)[ci] : (float)scost[ci];
            const float2 ph = COST == 0 ? phase_f32(C, KP.ghi, KP.glo) : stab[scost[ci]];
            if (BWD) {
                eacc = fmaf(C - KP.c0, fmaf(l[i].x, a[i].y, -l[i].y * a[i].x), eacc);
                l[i] = cmul_conj(l[i], ph);
                a[i] = cmul_conj(a[i], ph);
            } else {
                a[i] = cmul(a[i], ph);
            }
        }
    }

    // ---------------- round B: Q, R, P
    if constexpr (ST >= 2) {
        stage_rot<BWD, MB>(a, l, mq, KB.R, pscale, bB, true);
        if (KB.rescale) {
            scale_all<BWD>(a, l, KB.fsq);
            pscale = 1.f;
        }
        put_q<ST == 3>(a, sp, T.lq);
        if (BWD) put_q<ST == 3>(l, sl, T.lq);
        if constexpr (ST == 3) {
            __syncwarp();
            get_r(a, sp, T.lr);
            if (BWD) get_r(l, sl, T.lr);
            stage_rot<BWD, MB>(a, l, 0xFu, KB.R, pscale, bB, true);
            if (KB.rescale) {
                scale_all<BWD>(a, l, KB.fsr);
                pscale = 1.f;
            }
            put_r(a, sp, T.lr);
            if (BWD) put_r(l, sl, T.lr);
        }
        __syncthreads();
        get_p<ST == 3>(a, sp, T.lp);
        if (BWD) get_p<ST == 3>(l, sl, T.lp);
    }
    // the buffer is consumed: start the tile NBUF ahead
    __syncthreads();
    if (warp == 0)
        claim_issue<BWD, COST, NBUF>(bufs + b * G::kBufB, bar, sched, total, &tinfo[b], descs, tile_begin, ndesc,
                                     cursor, &D, s_tr);
    // psi is dead after the last adjoint pair terms
    stage_rot<BWD, MB>(a, l, mp, KB.R, pscale, bB, !BWD);
    if (BWD) scale_all<0>(l, l, KB.rescale ? KB.fsp : KB.fse);
    else scale_all<0>(a, a, KB.rescale ? KB.fsp : KB.fse);
    float2 *out = BWD ? D.lam_out : D.psi_out;
    if (out) {
        const float2 *v = BWD ? l : a;
        out += base + gp;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const uint32_t o = ST >= 2 ? (uint32_t)i * rs[0]
                                       : ((i & 1) ? rs[0] : 0u) + ((i & 2) ? rs[1] : 0u) + ((i & 4) ? rs[2] : 0u) +
                                             ((i & 8) ? rs[3] : 0u);
            __stcs(out + o, v[i]);
        }
    }
    if (BWD) {  // round k+1's beta total in lane 0, round k's in lane 16; gamma by its own tree
        const float t = warp_sum2_f(bA, bB);
        if (lane == 0 && D.part_beta) D.part_beta[tl * kNW + warp] = (double)t;
        if (lane == 16 && D.part_beta2) D.part_beta2[tl * kNW + warp] = (double)t;
        const float tg = warp_sum_f(eacc);
        if (lane == 0 && D.part_gamma) D.part_gamma[tl * kNW + warp] = (double)tg;
    }
}

// The common case (both rounds in the tan form) inline; the direct form
// (|cos b| tiny, rare) out of line, so that its registers do not set the
// register allocation of the common path.
template <int BWD, int COST, int NBUF, int MA, int MB, int ST, int QF, class... Args>
__device__ __forceinline__ void tile_body_fused(Args &&...args) {
    tile_body_fused_impl<BWD, COST, NBUF, MA, MB, ST, QF>(args...);
}
template <int BWD, int COST, int NBUF, int MA, int MB, int ST>
__device__ __noinline__ void tile_body_fused_rare(const PassConst &KA, const PassConst &KB, const PassConst &KP,
                                                  const uint32_t (&rs)[4], uint32_t gp,
                                                  const PassDesc &D, const float2 *stab, unsigned char *bufs, int b,
                                                  uint32_t bar, uint32_t *sched, uint32_t total, uint32_t base,
                                                  uint32_t tl, TileInfo *tinfo, const PassDesc *__restrict__ descs,
                                                  const uint32_t *__restrict__ tile_begin, int ndesc, int &cursor,
                                                  const uint32_t *s_tr) {
    tile_body_fused_impl<BWD, COST, NBUF, MA, MB, ST, 0>(KA, KB, KP, rs, gp, D, stab, bufs, b, bar, sched, total,
                                                         base, tl, tinfo, descs, tile_begin, ndesc, cursor, s_tr);
}

// GATH: the launch's tiles are gathered ones (ST 1 or 2 by descriptor), else
// contiguous (ST 3).
template <int BWD, int COST, int NBUF, int VAR, int FUSED, int GATH>
__global__ void __launch_bounds__(kNT, (BWD && NBUF > 1) ? 1 : 2)
xpass_kernel(const PassDesc *__restrict__ descs, const uint32_t *__restrict__ tile_begin, int ndesc,
             uint32_t total, int *err, uint32_t *__restrict__ sched) {
    using G = PassGeom<BWD, COST>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_raw);
    TileInfo *tinfo = reinterpret_cast<TileInfo *>(smem_raw + 64);
    float2 *stab = reinterpret_cast<float2 *>(smem_raw + 256);
    unsigned char *bufs = smem_raw + G::kHead;
    __shared__ PassDesc D;
    __shared__ float4 s_rot[12];  // multi-angle: (cos, +-sin, +-tan, cos^2) per local bit
    __shared__ float2 s_cc[12];   // multi-angle: cosines as float pairs (1 where not rotated)
    __shared__ float4 s_w[33];    // general X mixer: weight phases and G(w)
    __shared__ uint32_t s_tr[3];  // D's first tile, end tile and index
    __shared__ PassConst s_k[2];  // the round's constants (round-boundary launches: rounds k and k+1)

    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid == 0) {
        for (int b = 0; b < NBUF; b++) mbar_init(smem_u32(&bars[b]), 1);
        fence_mbar_init();
    }
    __syncthreads();
    chain_begin();
    const uint32_t stride = gridDim.x;
    int cursor = 0;  // loader's descriptor search position (warp 0)
    if (warp == 0) {
        for (int k = 0; k < NBUF; k++) {
            const uint32_t t = blockIdx.x + (uint32_t)k * stride;
            if (t < total)
                issue_tile<BWD, COST>(t, bufs + k * G::kBufB, smem_u32(&bars[k]), &tinfo[k], descs, tile_begin,
                                      ndesc, cursor, nullptr, nullptr);
            else
                post_end(smem_u32(&bars[k]), &tinfo[k]);
        }
    }
    int cur = -1;
    uint32_t gp = 0, rs[4] = {0, 0, 0, 0};

    for (uint32_t it = 0;; it++) {
        const int b = (int)(it % NBUF);
        const uint32_t bar = smem_u32(&bars[b]);
        const bool ok = mbar_wait(bar, (it / NBUF) & 1u);
        const TileInfo ti = tinfo[b];
        if (ok && ti.di == kTileEnd) break;  // uniform; later claims are end markers too
        const int di = ok ? ti.di : -1;
        if (di != cur) {  // uniform: every thread read the same tile info
            __syncthreads();  // the previous tile's epilogue is done with D / stab
            if (di < 0) {
                if (tid == 0) atomicOr(err, ok ? DERR_BAD_DESC : DERR_TIMEOUT);
                // let every load this CTA started land before the block exits
                // (each of the other buffers holds a claimed tile or an end marker)
                for (int k = 1; k < NBUF; k++)
                    mbar_wait(smem_u32(&bars[(it + k) % NBUF]), ((it + k) / NBUF) & 1u);
                if (!ok) mbar_wait(bar, (it / NBUF) & 1u);
                return;
            }
            const uint32_t *src = reinterpret_cast<const uint32_t *>(descs + di);
            uint32_t *dst = reinterpret_cast<uint32_t *>(&D);
            for (int i = tid; i < (int)(sizeof(PassDesc) / 4); i += kNT) dst[i] = src[i];
            if (tid == 0) {
                s_tr[0] = tile_begin[di];
                s_tr[1] = tile_begin[di + 1];
                s_tr[2] = (uint32_t)di;
            }
            __syncthreads();
            // undoing a round (adjoint) uses the coefficients of -b
            const float sgn = BWD ? -1.f : 1.f;
            if (tid < (FUSED ? 2 : 1)) {
                PassConst K;
                K.flags = D.flags;
                K.mq = (D.active >> 4) & 0xFu;
                K.mp = (D.active >> 8) & 0xFu;
                K.amp0 = D.amp0;
                K.c0 = (BWD && D.c0 && (D.flags & (PF_LAM_FROM_C | PF_PHASE | PF_FUSED))) ? (float)*D.c0 : 0.f;
                set_round(K, tid ? *D.coef2 : *D.coef, sgn, D.c >= kT);
                s_k[tid] = K;
            }
            gp = tile_offset(thread_pos().lp, D.c, D.c < kT ? D.gpos[D.c] : 0);
#pragma unroll
            for (int k = 0; k < 4; k++) rs[k] = 1u << D.gpos[8 + k];
            if (COST == 1 && (D.flags & (PF_PHASE | PF_FUSED)))
                for (int i = tid; i < kPhaseTable; i += kNT) stab[i] = D.table[i];
            if (VAR == 2 && (D.flags & PF_WDIAG))
                for (int i = tid; i <= D.n; i += kNT) s_w[i] = D.wtab[i];
            if (VAR == 1) {
                // per-qubit rotations: D.coef is this round's n entries, indexed
                // by global qubit.  The tan form when every rotated qubit allows
                // it, with the cosines per layout (rescale: any |cos| < 1/4) or
                // once per pass, else the direct form.
                bool tan_ok = true, resc = false;
                if (tid < kT) {
                    const RoundCoef &q = D.coef[D.gpos[tid]];
                    const float c = q.bmode == 0 ? q.pw[1] : q.cb;
                    s_rot[tid] = make_float4(q.cb, sgn * q.sb, sgn * q.bt, c * c);
                    const bool on = (D.active >> tid) & 1u;
                    s_cc[tid] = on ? make_float2(q.pw[1], q.c_lo) : make_float2(1.f, 0.f);
                    tan_ok = !on || q.bmode == 0;
                    resc = on && q.rescale;
                }
                tan_ok = __syncthreads_and(tan_ok);
                resc = __syncthreads_or(resc) && tan_ok;
                if (tid == 0) {
                    // products of the rotated qubits' cosines as float pairs (a
                    // rounding here would scale every amplitude of the pass alike)
                    auto prod = [&](int b0) -> float2 {
                        float2 f = make_float2(1.f, 0.f);
#pragma unroll
                        for (int j = b0; j < b0 + 4; j++) f = pair_mul(f, s_cc[j]);
                        return f;
                    };
                    const float2 fq = prod(4), fr = prod(0), fp = prod(8);
                    PassConst &K = s_k[0];
                    K.R.mode = tan_ok ? 0 : 2;
                    K.rescale = resc ? 1 : 0;
                    K.fsq = tan_ok ? fq.x : 1.f;
                    K.fsr = tan_ok ? fr.x : 1.f;
                    K.fsp = tan_ok ? fp.x : 1.f;
                    K.fse = tan_ok && !resc ? pair_mul(pair_mul(fq, fr), fp).x : 1.f;
                }
            }
            __syncthreads();
            cur = di;
        }
        const int c = D.c;
        if constexpr (FUSED) {
            // forward: round k then round k+1; adjoint: k+1 first; the phase is round k+1's
            const PassConst &KA = s_k[BWD ? 1 : 0], &KB = s_k[BWD ? 0 : 1], &KP = s_k[1];
            const int mk = (KA.R.mode == 0 ? 0 : 1) | (KB.R.mode == 0 ? 0 : 2);
#define QG_FUSED_ARGS                                                                                                \
    KA, KB, KP, rs, gp, D, stab, bufs, b, bar, sched, total, ti.base, ti.tl, tinfo, descs, tile_begin, ndesc, cursor, \
        s_tr
            if constexpr (!GATH) {
                if (mk == 0) tile_body_fused<BWD, COST, NBUF, 0, 0, 3, 1>(QG_FUSED_ARGS);
                else if (mk == 1) tile_body_fused_rare<BWD, COST, NBUF, 2, 0, 3>(QG_FUSED_ARGS);
                else if (mk == 2) tile_body_fused_rare<BWD, COST, NBUF, 0, 2, 3>(QG_FUSED_ARGS);
                else tile_body_fused_rare<BWD, COST, NBUF, 2, 2, 3>(QG_FUSED_ARGS);
            } else if (c >= 8) {
                if (mk == 0) tile_body_fused<BWD, COST, NBUF, 0, 0, 1, 0>(QG_FUSED_ARGS);
                else if (mk == 1) tile_body_fused_rare<BWD, COST, NBUF, 2, 0, 1>(QG_FUSED_ARGS);
                else if (mk == 2) tile_body_fused_rare<BWD, COST, NBUF, 0, 2, 1>(QG_FUSED_ARGS);
                else tile_body_fused_rare<BWD, COST, NBUF, 2, 2, 1>(QG_FUSED_ARGS);
            } else {
                if (mk == 0 && c == 4) tile_body_fused<BWD, COST, NBUF, 0, 0, 2, 1>(QG_FUSED_ARGS);
                else if (mk == 0) tile_body_fused<BWD, COST, NBUF, 0, 0, 2, 0>(QG_FUSED_ARGS);
                else if (mk == 1) tile_body_fused_rare<BWD, COST, NBUF, 2, 0, 2>(QG_FUSED_ARGS);
                else if (mk == 2) tile_body_fused_rare<BWD, COST, NBUF, 0, 2, 2>(QG_FUSED_ARGS);
                else tile_body_fused_rare<BWD, COST, NBUF, 2, 2, 2>(QG_FUSED_ARGS);
            }
#undef QG_FUSED_ARGS
        } else {
            const PassConst &K = s_k[0];
            const bool tan = K.R.mode == 0;
#define QG_TILE_ARGS                                                                                                \
    K, D, rs, gp, stab, s_rot, s_w, bufs, b, bar, sched, total, ti.base, ti.tl, tinfo, descs, tile_begin, ndesc,    \
        cursor, s_tr
            if constexpr (!GATH) {
                if (tan) tile_body<BWD, COST, NBUF, 0, VAR, 3, 1>(QG_TILE_ARGS);
                else tile_body<BWD, COST, NBUF, 2, VAR, 3, 1>(QG_TILE_ARGS);
            } else if (c >= 8) {
                if (tan) tile_body<BWD, COST, NBUF, 0, VAR, 1, 0>(QG_TILE_ARGS);
                else tile_body<BWD, COST, NBUF, 2, VAR, 1, 0>(QG_TILE_ARGS);
            } else {
                if (tan && c == 4) tile_body<BWD, COST, NBUF, 0, VAR, 2, 1>(QG_TILE_ARGS);
                else if (tan) tile_body<BWD, COST, NBUF, 0, VAR, 2, 0>(QG_TILE_ARGS);
                else tile_body<BWD, COST, NBUF, 2, VAR, 2, 0>(QG_TILE_ARGS);
            }
#undef QG_TILE_ARGS
        }
    }
}

template <int BWD, int COST, int NBUF, int VAR, int FUSED, int GATH>
cudaError_t launch_one(const PassDesc *d, const uint32_t *tb, int nd, uint32_t tiles, int *err, uint32_t *sched,
                       cudaStream_t s) {
    using G = PassGeom<BWD, COST>;
    const size_t smem = G::kHead + (size_t)NBUF * G::kBufB + G::kStashB;
    // per device: the shared-memory attribute and the persistent grid size
    static int attr_done[kMaxDevices];
    static int grid_caps[kMaxDevices];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    e = smem_attr_once(xpass_kernel<BWD, COST, NBUF, VAR, FUSED, GATH>, (int)smem, attr_done);
    if (e != cudaSuccess) return e;
    int grid_cap = __atomic_load_n(&grid_caps[dev], __ATOMIC_ACQUIRE);
    if (!grid_cap) {
        int nsm = 0, per_sm = 0;
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, xpass_kernel<BWD, COST, NBUF, VAR, FUSED, GATH>, kNT, smem);
        if (e != cudaSuccess) return e;
        grid_cap = std::max(1, nsm * std::max(1, per_sm));
        __atomic_store_n(&grid_caps[dev], grid_cap, __ATOMIC_RELEASE);
    }
    const uint32_t grid = std::min<uint32_t>(tiles, (uint32_t)grid_cap);
    return launch_chained(xpass_kernel<BWD, COST, NBUF, VAR, FUSED, GATH>, grid, kNT, smem, s, d, tb, nd, tiles, err,
                          sched);
}

template <int VAR, int FUSED, int GATH>
cudaError_t launch_xpass_t(int bwd, int cost_dtype, int nbuf, const PassDesc *d, const uint32_t *tb, int nd,
                           uint32_t tiles, int *err, uint32_t *sched, cudaStream_t s) {
    if (!bwd) return cost_dtype == 0 ? launch_one<0, 0, 2, VAR, FUSED, GATH>(d, tb, nd, tiles, err, sched, s)
                                     : launch_one<0, 1, 2, VAR, FUSED, GATH>(d, tb, nd, tiles, err, sched, s);
    // adjoint: one tile buffer and two CTAs per SM (128 registers a thread),
    // or two buffers and one CTA per SM (no register cap below 255)
    if (nbuf == 2)
        return cost_dtype == 0 ? launch_one<1, 0, 2, VAR, FUSED, GATH>(d, tb, nd, tiles, err, sched, s)
                               : launch_one<1, 1, 2, VAR, FUSED, GATH>(d, tb, nd, tiles, err, sched, s);
    return cost_dtype == 0 ? launch_one<1, 0, 1, VAR, FUSED, GATH>(d, tb, nd, tiles, err, sched, s)
                           : launch_one<1, 1, 1, VAR, FUSED, GATH>(d, tb, nd, tiles, err, sched, s);
}

template <int VAR, int FUSED>
cudaError_t launch_xpass_g(int bwd, int cost_dtype, int nbuf, int gather, const PassDesc *d, const uint32_t *tb,
                           int nd, uint32_t tiles, int *err, uint32_t *sched, cudaStream_t s) {
    return gather ? launch_xpass_t<VAR, FUSED, 1>(bwd, cost_dtype, nbuf, d, tb, nd, tiles, err, sched, s)
                  : launch_xpass_t<VAR, FUSED, 0>(bwd, cost_dtype, nbuf, d, tb, nd, tiles, err, sched, s);
}

}  // namespace
}  // namespace qg
