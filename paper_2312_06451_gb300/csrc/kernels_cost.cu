// Cost-vector pre-computation over the feasible set (arXiv 2312.06451,
// Sec. 2.1: C(x) is evaluated once for every feasible x and stored) and the
// Hamming-weight-k feasible set itself.
//
//   MaxCut   C(x) = #{edges (u, v) : x_u != x_v}, weighted: the sum of their weights.
//   SK       C(x) = sum_{i<j} J_ij z_i z_j, z_i = 1 - 2 x_i.
//            Both are quadratic forms in z.  When the couplings are multiples
//            of one power of two and the sums fit, they are carried exactly in
//            integers and rounded once to the output type (cost_quad_kernel);
//            float32 couplings that spread too far are summed in float64.
//   DkS      C(x) = sum_u x_u popcount(nbr_hi[u] & x) on weight-k states.
//   k-VC     C(x) = m - (the DkS count of the complement of x).
//   Dicke    state of rank r (increasing integer order = colex order of
//            k-subsets) by the combinatorial number system:
//            x = {c_k > ... > c_1}, r = sum_i binom(c_i, i).
#include "common.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace qg {

constexpr int kBinomMax = 41;  // n <= 40 for weight-k problems
__constant__ uint64_t c_binom[kBinomMax][kBinomMax];

int binom_table_max() { return kBinomMax - 1; }

cudaError_t upload_binom_table() {
    static uint64_t h[kBinomMax][kBinomMax];
    for (int a = 0; a < kBinomMax; a++)
        for (int b = 0; b < kBinomMax; b++)
            h[a][b] = (b == 0) ? 1 : (a == 0 ? 0 : h[a - 1][b - 1] + h[a - 1][b]);
    return cudaMemcpyToSymbol(c_binom, h, sizeof(h));
}

namespace {

struct AdjParams {
    uint64_t nbr[64];
    int n;
};

__device__ __forceinline__ uint64_t unrank_colex(int64_t r, int n, int k) {
    uint64_t x = 0;
    int c = n - 1;
    for (int i = k; i >= 1; i--) {
        while (c_binom[c][i] > (uint64_t)r) c--;
        x |= 1ull << c;
        r -= (int64_t)c_binom[c][i];
        c--;
    }
    return x;
}

__device__ __forceinline__ int64_t rank_colex(uint64_t x) {
    int64_t r = 0;
    int i = 1;
    while (x) {
        const int c = __ffsll((long long)x) - 1;
        r += (int64_t)c_binom[c][i];
        i++;
        x &= x - 1;
    }
    return r;
}

__global__ void cost_wmaxcut_kernel(const int32_t *edges, const float *w, int m, int64_t dim,
                                    float *out) {
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < dim;
         x += (int64_t)gridDim.x * blockDim.x) {
        double c = 0.0;
        for (int e = 0; e < m; e++) {
            const int u = __ldg(edges + 2 * e), v = __ldg(edges + 2 * e + 1);
            if (((x >> u) ^ (x >> v)) & 1) c += (double)__ldg(w + e);
        }
        out[x] = (float)c;
    }
}

constexpr int kSkMaxN = 40;

// MaxCut, weighted MaxCut and SK costs on all 2^n states as one integer
// quadratic form: C(x) = 2^-shift (base + sum_{i<j} K_ij z_i z_j), z = 1 - 2 x,
// carried exactly (so the result does not depend on the summation order) and
// rounded once to the output type.  An edge of weight w contributes
// w (1 - z_u z_v) / 2.
//
// One write per state bounds it (256 MiB of float32 at n = 26: 40 us), so a
// state may cost a handful of adds, not one per pair.  Local qubits 0, 1, 10
// and 11 are a thread's 16 outputs of a tile of 2^12, qubits 2..9 its index,
// qubits 12..11+M the 2^M tiles a block walks in Gray-code order, the rest the
// block index.  A thread sums its own qubits' pairs and the fields they exert
// once; a tile then moves by one flipped qubit (a few adds), and the 16
// outputs are +- combinations of five sums: about 4 adds an output instead of
// n(n-1)/2 with a shared-memory load each.  n = 26, int32: a call 12.1 ms -> 81 us.
// The output need only be aligned for one value: vectors that a caller packs one
// behind the other take stores of single values (VEC 0).
template <typename A>
struct QuadParams {
    A K[kQuadMaxN][kQuadMaxN];  // symmetric, zero diagonal, zero beyond n
    A base;
    int n;
    float scale;  // 2^-shift (float32 output)
};

template <typename A, int U8, int M, int VEC>
__global__ void __launch_bounds__(256) cost_quad_kernel(const __grid_constant__ QuadParams<A> Q, int64_t dim, void *out) {
    __shared__ A s_f[12 + M];  // fields of the block's qubits on the local ones
    __shared__ A s_e;          // base + the block qubits' own pairs
    const int tid = threadIdx.x, nb = Q.n - 12 - M;  // block qubits 12 + M ..
    const uint32_t hi = blockIdx.x;
    auto sg = [](uint32_t bit, A v) -> A { return bit ? -v : v; };
    if (tid < 12 + M) {
        A f = 0;
        for (int u = 0; u < nb; u++) f += sg((hi >> u) & 1u, Q.K[tid][12 + M + u]);
        s_f[tid] = f;
    } else if (tid >= 32 && tid < 64) {
        const int u = tid - 32;  // at most kQuadMaxN - 12 block qubits
        A e = 0;
        for (int v = u + 1; v < nb; v++) e += sg(((hi >> u) ^ (hi >> v)) & 1u, Q.K[12 + M + u][12 + M + v]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
        if (u == 0) s_e = e + Q.base;
    }
    __syncthreads();
    // this thread's qubits 2..9: their pairs and fields, and the fields on the
    // output qubits (a) and the tile qubits (g)
    A S = s_e, a[4], g[M > 0 ? M : 1];
    const int rq[4] = {0, 1, 10, 11};
#pragma unroll
    for (int r = 0; r < 4; r++) a[r] = s_f[rq[r]];
#pragma unroll
    for (int j = 0; j < M; j++) g[j] = s_f[12 + j];
#pragma unroll
    for (int i = 2; i < 10; i++) {
        const uint32_t bi = (uint32_t)tid >> (i - 2);
        A f = s_f[i];
#pragma unroll
        for (int j = i + 1; j < 10; j++) f += sg(((uint32_t)tid >> (j - 2)) & 1u, Q.K[i][j]);
        S += sg(bi & 1u, f);
#pragma unroll
        for (int r = 0; r < 4; r++) a[r] += sg(bi & 1u, Q.K[i][rq[r]]);
#pragma unroll
        for (int j = 0; j < M; j++) g[j] += sg(bi & 1u, Q.K[i][12 + j]);
    }
    // the first tile has every tile qubit at z = +1
#pragma unroll
    for (int j = 0; j < M; j++) {
        S += g[j];
#pragma unroll
        for (int l = 0; l < M; l++)
            if (l != j) {
                if (l < j) S += Q.K[12 + j][12 + l];
                g[j] += Q.K[12 + j][12 + l];
            }
#pragma unroll
        for (int r = 0; r < 4; r++) a[r] += Q.K[rq[r]][12 + j];
    }
    const int64_t x0 = ((int64_t)hi << (12 + M)) + 4 * tid;
#pragma unroll
    for (int t = 0; t < (1 << M); t++) {
        if (t) {  // Gray code: flip tile qubit j, from z = +1 to -1 (down) or back
            const int j = (t & 1) ? 0 : (t & 2) ? 1 : (t & 4) ? 2 : 3;
            const bool down = ((t ^ (t >> 1)) >> j) & 1;
            S += down ? -2 * g[j] : 2 * g[j];
#pragma unroll
            for (int l = 0; l < M; l++)
                if (l != j) g[l] += down ? -2 * Q.K[12 + j][12 + l] : 2 * Q.K[12 + j][12 + l];
#pragma unroll
            for (int r = 0; r < 4; r++) a[r] += down ? -2 * Q.K[12 + j][rq[r]] : 2 * Q.K[12 + j][rq[r]];
        }
        const int64_t xt = x0 + ((int64_t)(t ^ (t >> 1)) << 12);
#pragma unroll
        for (int h = 0; h < 4; h++) {  // qubits 10, 11
            const A k1 = Q.K[10][11];
            const A s = S + ((h & 1) ? -a[2] : a[2]) + ((h & 2) ? -a[3] : a[3]) + (((h >> 1) ^ h) & 1 ? -k1 : k1);
            const A b0 = a[0] + ((h & 1) ? -Q.K[0][10] : Q.K[0][10]) + ((h & 2) ? -Q.K[0][11] : Q.K[0][11]);
            const A b1 = a[1] + ((h & 1) ? -Q.K[1][10] : Q.K[1][10]) + ((h & 2) ? -Q.K[1][11] : Q.K[1][11]);
            const A p = s + Q.K[0][1], m = s - Q.K[0][1], u = b0 + b1, v = b1 - b0;
            const A c[4] = {p + u, m + v, m - v, p - u};  // (z_0, z_1) = ++, -+, +-, --
            const int64_t x = xt + ((int64_t)h << 10);
            if (U8) {
                const uchar4 o = make_uchar4((unsigned char)(c[0] >> 1), (unsigned char)(c[1] >> 1),
                                             (unsigned char)(c[2] >> 1), (unsigned char)(c[3] >> 1));
                unsigned char *dst = reinterpret_cast<unsigned char *>(out) + x;
                if (VEC && x + 4 <= dim) __stcs(reinterpret_cast<uchar4 *>(dst), o);
                else
                    for (int i = 0; i < 4; i++)
                        if (x + i < dim) dst[i] = i == 0 ? o.x : i == 1 ? o.y : i == 2 ? o.z : o.w;
            } else {
                float f[4];
#pragma unroll
                for (int i = 0; i < 4; i++) f[i] = (sizeof(A) == 8 ? __ll2float_rn((long long)c[i]) : __int2float_rn((int)c[i])) * Q.scale;
                float *dst = reinterpret_cast<float *>(out) + x;
                if (VEC && x + 4 <= dim) __stcs(reinterpret_cast<float4 *>(dst), make_float4(f[0], f[1], f[2], f[3]));
                else
                    for (int i = 0; i < 4; i++)
                        if (x + i < dim) dst[i] = f[i];
            }
        }
    }
}

__global__ void cost_sk_f64_kernel(int n, const double *Jd, int64_t dim, float *out) {
    __shared__ double J[kSkMaxN * kSkMaxN];
    for (int i = threadIdx.x; i < n * n; i += blockDim.x) J[i] = Jd[i];
    __syncthreads();
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < dim;
         x += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t ux = (uint64_t)x;
        double acc = 0.0;
        for (int i = 0; i < n; i++) {
            const uint64_t xi = (ux >> i) & 1;
            for (int j = i + 1; j < n; j++) {
                const double v = J[i * n + j];
                acc += (((ux >> j) & 1) ^ xi) ? -v : v;
            }
        }
        out[x] = (float)acc;
    }
}

// kvc = 0: edges inside the chosen set (densest k-subgraph); kvc = 1: edges
// with an end in the set (k-vertex cover) = m - edges inside the complement.
__global__ void cost_dks_kernel(AdjParams A, int k, int64_t dim, void *out, int dtype, int kvc, int m) {
    const uint64_t full = A.n == 64 ? ~0ull : ((1ull << A.n) - 1);
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < dim;
         a += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t x0 = unrank_colex(a, A.n, k);
        const uint64_t x = kvc ? (full ^ x0) : x0;
        int c = 0;
        for (int u = 0; u < A.n; u++)
            if ((x >> u) & 1) c += __popcll(A.nbr[u] & x);
        if (kvc) c = m - c;
        if (dtype == 1)
            reinterpret_cast<unsigned char *>(out)[a] = (unsigned char)c;
        else
            reinterpret_cast<float *>(out)[a] = (float)c;
    }
}

__global__ void dicke_states_kernel(int n, int k, int64_t dim, uint64_t *out) {
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < dim;
         a += (int64_t)gridDim.x * blockDim.x)
        out[a] = unrank_colex(a, n, k);
}

// Row a of the ring mixer restricted to weight-k states: for every ring edge
// (i, i+1 mod n) whose bits differ, X_i X_j + Y_i Y_j maps |x> to 2|x'> with
// the two bits swapped.  Row a is written only by thread a.
__global__ void ring_h_kernel(int n, int k, int64_t dim, double *H) {
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < dim;
         a += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t x = unrank_colex(a, n, k);
        for (int i = 0; i < n; i++) {
            const int j = (i + 1) % n;
            if (((x >> i) ^ (x >> j)) & 1) {
                const uint64_t y = x ^ (1ull << i) ^ (1ull << j);
                H[a * dim + rank_colex(y)] += 2.0;
            }
        }
    }
}

// Row a of the clique mixer restricted to weight-k states: the same swap
// term on every pair i < j whose bits differ.
__global__ void clique_h_kernel(int n, int k, int64_t dim, double *H) {
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < dim;
         a += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t x = unrank_colex(a, n, k);
        for (int i = 0; i < n; i++) {
            if (!((x >> i) & 1)) continue;  // i: a set bit, j: a clear bit
            for (int j = 0; j < n; j++) {
                if ((x >> j) & 1) continue;
                const uint64_t y = x ^ (1ull << i) ^ (1ull << j);
                H[a * dim + rank_colex(y)] += 2.0;
            }
        }
    }
}

unsigned grid_for(int64_t dim, int threads) {
    int64_t b = (dim + threads - 1) / threads;
    if (b > 152 * 64) b = 152 * 64;
    if (b < 1) b = 1;
    return (unsigned)b;
}

AdjParams make_adj(int n, const uint64_t *nbr_hi) {
    AdjParams A;
    for (int i = 0; i < 64; i++) A.nbr[i] = (i < n) ? nbr_hi[i] : 0;
    A.n = n;
    return A;
}

}  // namespace

namespace {

template <typename A, int U8>
cudaError_t go_quad(const CostQuad &C, int64_t dim, void *d_out, cudaStream_t s) {
    QuadParams<A> Q;
    for (int i = 0; i < kQuadMaxN; i++)
        for (int j = 0; j < kQuadMaxN; j++) Q.K[i][j] = i < C.n && j < C.n ? (A)C.K[i][j] : (A)0;
    Q.base = (A)C.base;
    Q.n = std::max(C.n, 12);  // qubits a small instance lacks: no couplings, states past dim not written
    Q.scale = ldexpf(1.f, -C.shift);
    if (reinterpret_cast<uintptr_t>(d_out) & (U8 ? 3 : 15)) {
        cost_quad_kernel<A, U8, 0, 0><<<1u << (Q.n - 12), 256, 0, s>>>(Q, dim, d_out);
        return cudaGetLastError();
    }
    // 2^M tiles a block: all 16 once that leaves two or more blocks an SM (M = 4 from n = 25), fewer
    // tiles and more blocks below
    const int M = std::max(0, std::min(4, Q.n - 21));
    const unsigned grid = 1u << (Q.n - 12 - M);
    switch (M) {
    case 0: cost_quad_kernel<A, U8, 0, 1><<<grid, 256, 0, s>>>(Q, dim, d_out); break;
    case 1: cost_quad_kernel<A, U8, 1, 1><<<grid, 256, 0, s>>>(Q, dim, d_out); break;
    case 2: cost_quad_kernel<A, U8, 2, 1><<<grid, 256, 0, s>>>(Q, dim, d_out); break;
    case 3: cost_quad_kernel<A, U8, 3, 1><<<grid, 256, 0, s>>>(Q, dim, d_out); break;
    default: cost_quad_kernel<A, U8, 4, 1><<<grid, 256, 0, s>>>(Q, dim, d_out); break;
    }
    return cudaGetLastError();
}

}  // namespace

bool cost_quad_exact(CostQuad &C, const double *w, int n, bool cut) {
    if (n > kQuadMaxN) return false;
    // the grid 2^-shift that holds every coupling
    int shift = 0;
    for (int i = 0; i < n; i++)
        for (int j = i + 1; j < n; j++) {
            const double v = w[i * n + j];
            if (!std::isfinite(v)) return false;
            if (v == 0.0) continue;
            int e = 0;
            const double f = std::frexp(v, &e);  // v = f 2^e, f of at most 53 bits
            const int64_t m = (int64_t)std::ldexp(f, 53);
            shift = std::max(shift, 53 - e - __builtin_ctzll((unsigned long long)m));
        }
    if (shift > 90) return false;  // float32 results stay far from the subnormals
    // sums below 2^50 on the grid: exact in int64, and in the float64 sums they stand for
    double total = 0.0;
    for (int i = 0; i < n; i++)
        for (int j = i + 1; j < n; j++) total += std::ldexp(std::fabs(w[i * n + j]), shift);
    if (!(total < 1125899906842624.0)) return false;
    std::memset(&C, 0, sizeof(C));
    C.n = n;
    C.shift = shift + (cut ? 1 : 0);
    for (int i = 0; i < n; i++)
        for (int j = i + 1; j < n; j++) {
            const int64_t k = (int64_t)std::ldexp(w[i * n + j], shift);
            C.K[i][j] = C.K[j][i] = cut ? -k : k;
            C.base += cut ? k : 0;
        }
    C.wide = total + std::fabs((double)C.base) >= 1073741824.0;  // a thread's running sums reach twice this at most
    return true;
}

cudaError_t launch_cost_quad(const CostQuad &C, int64_t dim, void *d_out, int dtype, cudaStream_t s) {
    if (C.n < 1 || C.n > kQuadMaxN || (dtype == 1 && (C.shift != 1 || C.wide))) return cudaErrorInvalidValue;
    if (dtype == 1) return go_quad<int32_t, 1>(C, dim, d_out, s);
    return C.wide ? go_quad<int64_t, 0>(C, dim, d_out, s) : go_quad<int32_t, 0>(C, dim, d_out, s);
}

cudaError_t launch_cost_wmaxcut(const float *d_w, const int32_t *d_edges, int m, int64_t dim, float *d_out,
                                cudaStream_t s) {
    cost_wmaxcut_kernel<<<grid_for(dim, 256), 256, 0, s>>>(d_edges, d_w, m, dim, d_out);
    return cudaGetLastError();
}

cudaError_t launch_cost_sk(int n, const double *d_Jd, int64_t dim, float *d_out, cudaStream_t s) {
    if (n > kSkMaxN) return cudaErrorInvalidValue;
    cost_sk_f64_kernel<<<grid_for(dim, 256), 256, 0, s>>>(n, d_Jd, dim, d_out);
    return cudaGetLastError();
}

cudaError_t launch_cost_dks(int n, int k, const uint64_t *nbr_hi, int64_t dim, void *d_out, int dtype,
                            int kvc, int m, cudaStream_t s) {
    cost_dks_kernel<<<grid_for(dim, 256), 256, 0, s>>>(make_adj(n, nbr_hi), k, dim, d_out, dtype, kvc, m);
    return cudaGetLastError();
}

cudaError_t launch_dicke_states(int n, int k, int64_t dim, uint64_t *d_out, cudaStream_t s) {
    dicke_states_kernel<<<grid_for(dim, 256), 256, 0, s>>>(n, k, dim, d_out);
    return cudaGetLastError();
}

cudaError_t launch_ring_hamiltonian(int n, int k, int64_t dim, double *d_H, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(d_H, 0, (size_t)dim * (size_t)dim * sizeof(double), s);
    if (e != cudaSuccess) return e;
    ring_h_kernel<<<grid_for(dim, 128), 128, 0, s>>>(n, k, dim, d_H);
    return cudaGetLastError();
}

cudaError_t launch_clique_hamiltonian(int n, int k, int64_t dim, double *d_H, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(d_H, 0, (size_t)dim * (size_t)dim * sizeof(double), s);
    if (e != cudaSuccess) return e;
    clique_h_kernel<<<grid_for(dim, 128), 128, 0, s>>>(n, k, dim, d_H);
    return cudaGetLastError();
}

}  // namespace qg
