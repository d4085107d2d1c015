// Exact separable solver of the discrete problems: the inner solver of the
// mixed-precision defect correction, the FP64 direct correction, and the
// coarse-grid solve of the V-cycles.
//
// xi depends on z only (Sect. 2.1, eq. scalar_pot) and the side faces are
// Dirichlet (Sect. 2.2), so the discrete sine vectors
//   s_m(i) = sin(pi m i / (nx - 1)),  m = 1 .. nx-2
// diagonalise the horizontal second differences: on plane k the operator
// cx_k (E + W - 2) + cy_k (N + S - 2) becomes cx_k mu_x(m) + cy_k mu_y(n)
// with mu(m) = -4 sin^2(pi m / (2 (n - 1))).  A = f on one level then splits
// into one tridiagonal system along z per mode (m, n):
//   cz (e[k-1] + e[k+1]) + D_k e[k] = rhat[k],
//   D_k = (alpha^2 - 2 cz) + cx_k mu_x(m) + cy_k mu_y(n),
// and the lower-boundary problem (eq. lower_bound) into a division per mode.
// Every multigrid level is a rediscretisation with the same structure, so
// the same solver applies on any level.  The sine transforms are
// - dense products with folded sine matrices, both transforms of a plane in one
//   launch (plane_body), on planes of at most 128 cells a side that have no fast
//   transform or a slower one (dense_planes_faster in launch_rules.h);
// - exact digit products on the tensor cores in the FP64 direct correction of 128
//   and 256 cells and on coarse FP64 levels of 64 x 64 cells, where the FP64 pipe
//   bounds the fast transforms (kernels_split.cu);
// - fast transforms (kernels_dst.cu) on other planes whose nx - 1 and ny - 1 are
//   powers of two;
// - in FP32 batched GEMMs with the (symmetric) sine matrices otherwise (in FP64
//   such levels are refused, sep_level_ok).
// The inverse is the same transform scaled by (2/(nx-1)) (2/(ny-1)).  In FP32 the
// solve is accurate to about 1e-6 relative, which the double-float outer loop of
// mixed mode then corrects.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

#include "device_util.cuh"
#include "dst_body.cuh"
#include "group.h"
#include "launch_rules.h"
#include "mhs_internal.h"
#include "per_device.h"
#include "solver.h"

namespace mhs {

namespace {

// C_b = scale A_b B_b (+ C_b): TB x TB output tile per block of 256 threads,
// TB/16 x TB/16 outputs per thread (rows ty + 16 r, columns tx + 16 c), K
// staged through shared memory TK at a time; block (bx, by, bz) = (column
// tile, row tile, batch).  Every output is one FMA chain over increasing k,
// whatever the tile, so the results do not depend on it.
template <typename T, int TB, int TK>
__device__ __forceinline__ void gemm_tile(const GemmArgs<T>& g, int bx, int by, int bz, T* smem) {
    constexpr int R = TB / 16, LD = TB + (TB > 16 ? 4 : 1);
    T* As = smem;               // [TK][LD]
    T* Bs = smem + TK * LD;     // [TK][LD]
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int row0 = by * TB, col0 = bx * TB;
    const long long b = bz;
    const T* A = g.A + b * g.sA;
    const T* B = g.B + b * g.sB;
    T* C = g.C + b * g.sC;
    T acc[R][R] = {};
    for (int k0 = 0; k0 < g.K; k0 += TK) {
        // A tile: TB rows x TK k (k fastest in global memory)
#pragma unroll 4
        for (int e = threadIdx.x; e < TB * TK; e += 256) {
            const int r = e / TK, kk = e % TK;
            const int gr = row0 + r, gk = k0 + kk;
            As[kk * LD + r] = (gr < g.M && gk < g.K) ? A[(long long)gr * g.lda + gk] : T(0);
        }
        // B tile: TK k x TB columns (columns fastest)
#pragma unroll 4
        for (int e = threadIdx.x; e < TK * TB; e += 256) {
            const int kk = e / TB, c = e % TB;
            const int gk = k0 + kk, gc = col0 + c;
            Bs[kk * LD + c] = (gk < g.K && gc < g.N) ? B[(long long)gk * g.ldb + gc] : T(0);
        }
        __syncthreads();
        const int kn = min(TK, g.K - k0);
#pragma unroll 8
        for (int kk = 0; kk < kn; ++kk) {
            T a[R], bb[R];
#pragma unroll
            for (int r = 0; r < R; ++r) a[r] = As[kk * LD + ty + 16 * r];
#pragma unroll
            for (int c = 0; c < R; ++c) bb[c] = Bs[kk * LD + tx + 16 * c];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < R; ++c) acc[r][c] = fma(a[r], bb[c], acc[r][c]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int gr = row0 + ty + 16 * r;
        if (gr >= g.M) continue;
#pragma unroll
        for (int c = 0; c < R; ++c) {
            const int gc = col0 + tx + 16 * c;
            if (gc < g.N) {
                const T v = g.scale * acc[r][c];
                const long long at = (long long)gr * g.ldc + gc;
                C[at] = g.accumulate ? C[at] + v : v;
            }
        }
    }
}

// The tile of a product (GemmArgs::tile): the largest that still gives two
// blocks per SM (one plane's product in 64 x 64 tiles ran on a few SMs alone).
// FP32 only: the FP64 levels without a fast transform are planes of at most 65
// cells, which plane_body serves.
constexpr int TK64 = 16, TK32 = 32, TK16 = 64;
constexpr int GEMM_SMEM = 2 * TK32 * 36;   // the 32 x 32 tiles' two operands, the largest
static_assert(GEMM_SMEM >= 2 * TK16 * 17 && GEMM_SMEM >= 2 * TK64 * 68, "shared memory of the other tiles");

int gemm_tile_size(int M, int N, int batch) {
    for (int tb : {64, 32})
        if ((long long)((M + tb - 1) / tb) * ((N + tb - 1) / tb) * batch >= 2 * 152) return tb;
    return 16;
}

template <typename T>
__device__ __forceinline__ void gemm_body(const GemmArgs<T>& g, int bx, int by, int bz) {
    __shared__ T smem[GEMM_SMEM];
    if (g.tile == 16) gemm_tile<T, 16, TK16>(g, bx, by, bz, smem);
    else if (g.tile == 32) gemm_tile<T, 32, TK32>(g, bx, by, bz, smem);
    else gemm_tile<T, 64, TK64>(g, bx, by, bz, smem);
}

template <typename T>
__global__ void __launch_bounds__(256) gemm_kernel(GemmArgs<T> g) {
    gemm_body(g, int(blockIdx.x), int(blockIdx.y), int(blockIdx.z));
}

// Both sine transforms of a plane as dense products with folded matrices.
//
// With M elements (M + 1 = N), s_i = x_i + x_{N-i} and d_i = x_i - x_{N-i}, the
// odd results need only the s_i (and the middle element when N is even), the
// even ones only the d_i: two matrices of half the side, Ko = ceil(M/2) and
// Ke = floor(M/2), half the products.  A block takes sp odd and sp even results
// b of the first transform (along the lines) for all A lines, and transforms
// those along the lines' index: no other block's data is needed, so a plane is
// one launch without clusters or exchanges, and every block loads the whole
// plane (from L2).  The sums run in blocks of eight (one FMA chain each), whose
// sums are added in order: a rounding error that grows with the number of
// blocks rather than of terms, no larger than the fast transforms'.
//
// Fast transforms need fewer operations, but on the planes of coarse levels
// they are a chain of short barrier-separated steps.  Per launch, forward or
// inverse: FP32 65^3 9.6 us (fast transforms 14), 33^3 6.9 (8.3), FP64 17^3 5.9
// (14); the 65^2 lower-boundary solve in one cluster 22.6 us in FP64 (31); as
// stages of ragged 49 x 41 planes 14 us instead of two products of 9.5.  Whole
// mixed solves with fields 1.25 -> 1.17 ms (129^3), FP64 33^3 1.01 -> 0.88 ms.
// Errors against the exact solution, random and smooth right-hand sides, 17^3
// to 129 x 129 x 17: FP32 1.0e-7 .. 2.4e-7 (fast transforms 1.0e-7 .. 2.8e-7).
// FP32: four results per thread share each loaded element (R = 4).  FP64 is
// bound by its pipe, so one result per thread spreads a plane furthest.
constexpr int PLANE_T = 256;
constexpr int PLANE_CELLS = 128;   // most cells of a side

// shared memory of plane_body (elements; every part a multiple of four)
template <typename T>
struct PlaneLayout {
    int s1, g, x, total;   // offsets after the matrix of the second transform
    __host__ __device__ PlaneLayout(int A, int M1, int sp) {
        const int Ko2 = (A + 1) / 2, Ke2 = A / 2;
        auto up = [](int n) { return (n + 3) / 4 * 4; };
        s1 = up(Ko2 * Ko2 + Ke2 * Ke2);
        g = s1 + up(M1 * sp);
        x = g + up(A * 2 * sp);
        total = x + up(M1 * (A | 1));
    }
};

// blocked dot products: out[q] = sum over i < K of m(i)[q] x(i)
template <typename T, int R, typename FX, typename FM>
__device__ __forceinline__ void plane_dot(int K, FX&& x, FM&& m, T (&tot)[R]) {
#pragma unroll
    for (int q = 0; q < R; ++q) tot[q] = T(0);
    int i = 0;
    for (; i + 8 <= K; i += 8) {
        T p[R] = {};
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const T xv = x(i + u);
            T mv[R];
            m(i + u, mv);
#pragma unroll
            for (int q = 0; q < R; ++q) p[q] = fma(mv[q], xv, p[q]);
        }
#pragma unroll
        for (int q = 0; q < R; ++q) tot[q] += p[q];
    }
    if (i < K) {
        T p[R] = {};
        for (; i < K; ++i) {
            const T xv = x(i);
            T mv[R];
            m(i, mv);
#pragma unroll
            for (int q = 0; q < R; ++q) p[q] = fma(mv[q], xv, p[q]);
        }
#pragma unroll
        for (int q = 0; q < R; ++q) tot[q] += p[q];
    }
}

template <int R, typename T>
__device__ __forceinline__ void plane_ld(const T* p, T (&v)[R]) {
    if constexpr (R == 4 && sizeof(T) == 4) {
        const float4 w = *reinterpret_cast<const float4*>(p);
        v[0] = w.x, v[1] = w.y, v[2] = w.z, v[3] = w.w;
    } else {
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = p[q];
    }
}

template <typename T>
constexpr int plane_r() { return sizeof(T) == 4 ? 4 : 1; }

// matrix of n elements to shared memory, 16 bytes at a time (both aligned)
template <typename T>
__device__ __forceinline__ void plane_matrix(T* dst, const T* __restrict__ src, int n) {
    constexpr int V = 16 / sizeof(T);
#pragma unroll 4
    for (int e = threadIdx.x; e < n / V; e += PLANE_T)
        reinterpret_cast<uint4*>(dst)[e] = __ldg(reinterpret_cast<const uint4*>(src) + e);
    for (int e = n / V * V + threadIdx.x; e < n; e += PLANE_T) dst[e] = src[e];
}

// the block's columns of the first transform's matrix: [Ko1][sp] odd, [Ke1][sp] even results from p0
template <typename T>
__device__ __forceinline__ void plane_columns(T* S1, const T* __restrict__ s1, int M1, int sp, int p0) {
    const int Ko1 = (M1 + 1) / 2, Ke1 = M1 / 2;
#pragma unroll 4
    for (int e = threadIdx.x; e < M1 * sp; e += PLANE_T) {
        const int i = e / sp, p = p0 + (e - i * sp);
        const bool odd = i < Ko1;
        S1[e] = p < (odd ? Ko1 : Ke1) ? __ldg(s1 + (odd ? i * Ko1 : Ko1 * Ko1 + (i - Ko1) * Ke1) + p) : T(0);
    }
}

// lines a < A of M1 elements ld(a, i), folded: X[i][a] the sums (and the
// middle element), X[M1 - 1 - i][a] the differences.  A warp takes whole
// lines, eight at a time, all loads before the stores.
template <typename T, typename LD>
__device__ __forceinline__ void plane_fold(T* X, int pA, int A, int M1, LD&& ld) {
    constexpr int B = 8;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = PLANE_T / 32, Ko1 = (M1 + 1) / 2;
    for (int i = lane; i < Ko1; i += 32) {
        const int j = M1 - 1 - i;
        for (int a0 = w; a0 < A; a0 += B * nw) {
            T lo[B], hi[B];
#pragma unroll
            for (int q = 0; q < B; ++q) {
                const int a = a0 + q * nw;
                lo[q] = a < A ? ld(a, i) : T(0);
                hi[q] = a < A && i != j ? ld(a, j) : T(0);
            }
#pragma unroll
            for (int q = 0; q < B; ++q) {
                const int a = a0 + q * nw;
                if (a >= A) continue;
                X[i * pA + a] = i == j ? lo[q] : lo[q] + hi[q];
                if (i != j) X[j * pA + a] = lo[q] - hi[q];
            }
        }
    }
}

// first transform: G[a][parity sp + q] = results p0 + q of line a, from X and S1
template <typename T>
__device__ __forceinline__ void plane_first(const T* X, const T* S1, T* G, int A, int M1, int sp) {
    constexpr int R = plane_r<T>();
    const int Ko1 = (M1 + 1) / 2, Ke1 = M1 / 2, pA = A | 1, A32 = (A + 31) / 32 * 32, per = sp / R;
    for (int u = threadIdx.x; u < A32 * 2 * per; u += PLANE_T) {
        const int a = u % A32, h = u / A32, par = h / per, q0 = (h - par * per) * R;
        if (a >= A) continue;
        const T* S = S1 + (par ? Ko1 * sp : 0) + q0;
        const T* Xa = X + (par ? (M1 - 1) * pA : 0) + a;
        const int step = par ? -pA : pA;
        T v[R];
        plane_dot<T, R>(
            par ? Ke1 : Ko1, [&](int i) { return Xa[i * step]; }, [&](int i, T(&m)[R]) { plane_ld<R>(S + i * sp, m); },
            v);
#pragma unroll
        for (int q = 0; q < R; ++q) G[a * 2 * sp + par * sp + q0 + q] = v[q];
    }
}

// fold along the lines' index: row a the sums, row A - 1 - a the differences
template <typename T>
__device__ __forceinline__ void plane_refold(T* G, int A, int sp) {
    for (int e = threadIdx.x; e < A / 2 * 2 * sp; e += PLANE_T) {
        const int a = e / (2 * sp), q = e - a * 2 * sp;
        const T lo = G[a * 2 * sp + q], hi = G[(A - 1 - a) * 2 * sp + q];
        G[a * 2 * sp + q] = lo + hi;
        G[(A - 1 - a) * 2 * sp + q] = lo - hi;
    }
}

// second transform, of the refolded G along the lines' index: st(b, c, value) for result c of the
// block's column b (0 .. 2 sp - 1, odd results first)
template <typename T, typename ST>
__device__ __forceinline__ void plane_second(const T* G, const T* S2, int A, int sp, ST&& st) {
    constexpr int R = plane_r<T>();
    const int Ko2 = (A + 1) / 2, Ke2 = A / 2, C32 = (Ko2 + 31) / 32 * 32, groups = 2 * sp / R;
    for (int u = threadIdx.x; u < C32 * 2 * groups; u += PLANE_T) {
        const int c = u % C32, h = u / C32, par = h / groups, b0 = (h - par * groups) * R;
        const int K = par ? Ke2 : Ko2;
        if (c >= K) continue;
        const T* S = S2 + (par ? Ko2 * Ko2 : 0) + c;
        const T* Gb = G + (par ? (A - 1) * 2 * sp : 0) + b0;
        const int step = par ? -2 * sp : 2 * sp;
        T v[R];
        plane_dot<T, R>(K, [&](int i) { return S[i * K]; }, [&](int i, T(&m)[R]) { plane_ld<R>(Gb + i * step, m); }, v);
#pragma unroll
        for (int q = 0; q < R; ++q) st(b0 + q, 2 * c + par, v[q]);
    }
}

// block bx: results p0 = sp bx .. of either parity; by: the plane
template <typename T>
__device__ __forceinline__ void plane_body(const PlaneArgs<T>& g, int bx, int by) {
    extern __shared__ __align__(16) unsigned char psep_smem[];
    const int A = g.A, M1 = g.M1, sp = g.sp;
    const PlaneLayout<T> L(A, M1, sp);
    const int Ko1 = (M1 + 1) / 2, Ke1 = M1 / 2, Ko2 = (A + 1) / 2, Ke2 = A / 2;
    T* S2 = reinterpret_cast<T*>(psep_smem);
    T *S1 = S2 + L.s1, *G = S2 + L.g, *X = S2 + L.x;
    const int p0 = bx * sp;
    const T* in = g.in + by * g.in_plane;
    plane_matrix(S2, g.s2, Ko2 * Ko2 + Ke2 * Ke2);
    plane_columns(S1, g.s1, M1, sp, p0);
    plane_fold(X, A | 1, A, M1, [&](int a, int i) { return in[a * g.in_line + i]; });
    __syncthreads();
    plane_first(X, S1, G, A, M1, sp);
    __syncthreads();
    plane_refold(G, A, sp);
    __syncthreads();
    T* out = g.out + by * g.out_plane;
    plane_second(G, S2, A, sp, [&](int b, int c, T v) {
        const int par = b >= sp, p = p0 + b - par * sp;
        if (p >= (par ? Ke1 : Ko1)) return;
        T* o = out + (long long)(2 * p + par) * g.out_line + c;
        *o = dst_result(g.scale, v, g.accumulate != 0, g.accumulate ? *o : T(0));
    });
}

template <typename T>
__global__ void __launch_bounds__(PLANE_T) sep_dense_kernel(PlaneArgs<T> a) {
    plane_body(a, int(blockIdx.x), int(blockIdx.y));
}

// elements of the cluster kernel's X, which serves as [nxi][nyi | 1], [nyi][2 sp] and [nxi][2 so]
template <typename T>
__host__ __device__ inline size_t dense2d_x(int nxi, int nyi, int sp, int so) {
    size_t n = size_t(nxi) * (nyi | 1);
    if (size_t(nyi) * 2 * sp > n) n = size_t(nyi) * 2 * sp;
    if (size_t(nxi) * 2 * so > n) n = size_t(nxi) * 2 * so;
    return (n + 3) / 4 * 4;
}

// The whole solve of a lower-boundary level in one cluster (one CTA per slab
// of results): x and y transforms of the CTA's x modes, the division by the
// mode eigenvalues, the y transform back (still the CTA's own modes), one
// exchange through distributed shared memory, and the x transform back of the
// CTA's rows.  The operations of the plane stages and the division in their
// order.  f = forward stage (x lines), b = the way back (y lines).
template <typename T>
__global__ void __launch_bounds__(PLANE_T) sep_dense2d_kernel(PlaneArgs<T> f, PlaneArgs<T> b, T cf, T cs,
                                                              const T* __restrict__ mufast,
                                                              const T* __restrict__ muslow) {
    extern __shared__ __align__(16) unsigned char psep_smem[];
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = int(cl.block_rank());
    const int nyi = f.A, nxi = f.M1, sp = f.sp, so = b.sp;
    const int Kox = (nxi + 1) / 2, Kex = nxi / 2, Koy = (nyi + 1) / 2, Key = nyi / 2;
    const PlaneLayout<T> L(nyi, nxi, sp);
    // the matrices of y (S2) and of x (after everything else), whole
    T* Sy = reinterpret_cast<T*>(psep_smem);
    T *S1 = Sy + L.s1, *G = Sy + L.g, *X = Sy + L.x, *Sx = X + dense2d_x<T>(nxi, nyi, sp, so);
    T* C = Sx + (Kox * Kox + Kex * Kex + 3) / 4 * 4;   // [2 sp][nyi]: this CTA's modes, back in y
    const int p0 = rank * sp;
    plane_matrix(Sy, f.s2, Koy * Koy + Key * Key);
    plane_matrix(Sx, f.s1, Kox * Kox + Kex * Kex);
    plane_columns(S1, f.s1, nxi, sp, p0);
    plane_fold(X, nyi | 1, nyi, nxi, [&](int a, int i) { return f.in[a * f.in_line + i]; });
    __syncthreads();
    plane_first(X, S1, G, nyi, nxi, sp);
    __syncthreads();
    plane_refold(G, nyi, sp);
    __syncthreads();
    // x mode of column q (past the last one: the results are not used)
    auto mode = [&](int q) { return q < sp ? 2 * (p0 + q) : 2 * (p0 + q - sp) + 1; };
    T* H = X;   // [nyi][2 sp]: mode n of column q, divided (X is no longer read)
    plane_second(G, Sy, nyi, sp, [&](int q, int n, T v) {
        const int m = mode(q);
        H[n * 2 * sp + q] = m < nxi ? mode_divide(dst_result(T(1), v, false, T(0)), cf, mufast[n], cs, muslow[m]) : T(0);
    });
    __syncthreads();
    plane_refold(H, nyi, sp);
    __syncthreads();
    plane_second(H, Sy, nyi, sp, [&](int q, int j, T v) { C[q * nyi + j] = v; });
    cl.sync();
    // rows j of this CTA (so odd and so even indexes), all modes from their owners
    const int r0 = rank * so, rows = 2 * so;
    T* Y = X;   // [nxi][2 so]: element m of row column r
    for (int e = threadIdx.x; e < nxi * rows; e += PLANE_T) {
        const int r = e / nxi, m = e - r * nxi;
        const int j = r < so ? 2 * (r0 + r) : 2 * (r0 + r - so) + 1;
        const int p = m >> 1, owner = p / sp, q = (p - owner * sp) + ((m & 1) ? sp : 0);
        Y[m * rows + r] = j < nyi ? cl.map_shared_rank(C, owner)[q * nyi + j] : T(0);
    }
    cl.sync();   // every remote read done before any CTA of the cluster exits
    plane_refold(Y, nxi, so);
    __syncthreads();
    plane_second(Y, Sx, nxi, so, [&](int r, int i, T v) {
        const int j = r < so ? 2 * (r0 + r) : 2 * (r0 + r - so) + 1;
        if (j >= nyi) return;
        T* o = b.out + (long long)j * b.out_line + i;
        *o = dst_result(b.scale, v, b.accumulate != 0, b.accumulate ? *o : T(0));
    });
}

// shared memory of the cluster kernel: plane_body's, the x matrix and the exchanged modes after it
template <typename T>
size_t dense2d_smem(int nxi, int nyi, int sp, int so) {
    const int Kox = (nxi + 1) / 2, Kex = nxi / 2;
    return (size_t(PlaneLayout<T>(nyi, nxi, sp).x) + dense2d_x<T>(nxi, nyi, sp, so) +
            (size_t(Kox) * Kox + size_t(Kex) * Kex + 3) / 4 * 4 + size_t(2) * sp * nyi) *
           sizeof(T);
}

// One transform per launch (the staged form): plane_dot's sums on folded lines.
// A block folds LINE_Y plane_r lines into shared memory once, then each thread forms one
// result of plane_r of them, a warp's results of one parity, every element of the
// matrix loaded for all of them (folding at each result took two loads and an
// addition per term: staged mixed solves of 129 x 129 x 33 772 us, now 573 us, FP64
// ones of 65 x 65 x 33 773 and 570 us).  Blocks of 64 x LINE_Y threads.
constexpr int LINE_Y = 4;
template <typename T>
__global__ void __launch_bounds__(64 * LINE_Y)
sep_line_kernel(int lines, int M, const T* __restrict__ in, long long in_plane, long long in_line, T* __restrict__ out,
                long long out_plane, long long out_line, long long out_elem, const T* __restrict__ s, T scale,
                int accumulate) {
    constexpr int R = plane_r<T>(), LB = LINE_Y * R, LD = LB + R;
    __shared__ __align__(16) T F[PLANE_CELLS * LD];   // [element][line]: sums, then differences
    const int Ko = (M + 1) / 2, Ke = M / 2, l0 = blockIdx.y * LB, k = blockIdx.z;
    const T* x = in + k * in_plane + l0 * in_line;
    for (int e = threadIdx.x + 64 * threadIdx.y; e < Ko * LB; e += 64 * LINE_Y) {
        const int q = e / Ko, i = e - q * Ko, j = M - 1 - i;
        const bool on = l0 + q < lines;
        const T lo = on ? x[q * in_line + i] : T(0), hi = on && i != j ? x[q * in_line + j] : T(0);
        F[i * LD + q] = i == j ? lo : lo + hi;
        if (i != j) F[(Ko + i) * LD + q] = lo - hi;
    }
    __syncthreads();
    const int m = blockIdx.x * 64 + 2 * (threadIdx.x & 31) + (threadIdx.x >> 5), q0 = threadIdx.y * R;
    if (m >= M || l0 + q0 >= lines) return;
    const int par = m & 1, p = m >> 1, K = par ? Ke : Ko;
    const T* S = s + (par ? Ko * Ko : 0) + p;
    const T* f = F + (par ? Ko * LD : 0) + q0;
    T v[R];
    plane_dot<T, R>(K, [&](int i) { return __ldg(S + i * K); }, [&](int i, T(&w)[R]) { plane_ld<R>(f + i * LD, w); }, v);
#pragma unroll
    for (int q = 0; q < R; ++q) {
        if (l0 + q0 + q >= lines) break;
        T* o = out + k * out_plane + (l0 + q0 + q) * out_line + m * out_elem;
        *o = dst_result(scale, v[q], accumulate != 0, accumulate ? *o : T(0));
    }
}

constexpr size_t PLANE_SMEM = 227 * 1024;

// Elimination factors of the mode systems of one 3D level, one thread per
// mode (fast index m, slow index n; the layout of the transformed data),
// formed in FP64 from the FP64 plane coefficients and rounded to T:
//   D_k = base_k + c_k^fast mu_fast(m) + c_k^slow mu_slow(n),
//   pivot_1 = D_1, pivot_k = D_k - cz sup_{k-1}, inv_k = 1 / pivot_k,
//   sup_k = cz inv_k,
// with mu(m) = -4 sin^2(pi (m + 1) / (2 (n_nodes - 1))).  ytrans: the fast
// index is the y mode (fast transforms), else the x mode (dense transforms).
template <typename T>
__global__ void sep_pivot_kernel(int nfast, int nslow, int nzi, int nodes_fast, int nodes_slow,
                                 const PlaneCoef<double>* __restrict__ coef, int ytrans, T* __restrict__ inv,
                                 T* __restrict__ sup) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    const int n = blockIdx.y;
    if (m >= nfast) return;
    const double sf = sinpi(double(m + 1) / (2.0 * (nodes_fast - 1)));
    const double ss = sinpi(double(n + 1) / (2.0 * (nodes_slow - 1)));
    const double af = -4.0 * sf * sf, as = -4.0 * ss * ss;
    const double cz = coef[1].cz;
    const size_t stride = size_t(nfast) * nslow, o = size_t(n) * nfast + m;
    double prev = 0.0;
    for (int k = 0; k < nzi; ++k) {
        const PlaneCoef<double> c = coef[k + 1];
        const double d = ytrans ? c.base + c.cy * af + c.cx * as : c.base + c.cx * af + c.cy * as;
        const double iv = 1.0 / (k ? d - cz * prev : d);
        prev = cz * iv;
        inv[k * stride + o] = T(iv);
        sup[k * stride + o] = T(prev);
    }
}

// One thread per mode (m fast, n slow) of the transformed data t[k][n][m]
// (k = 0 .. nzi-1 standing for planes 1 .. nzi): the mode's tridiagonal
// system along k solved with its precomputed elimination factors,
//   forward  e_k <- (t_k - cz e_{k-1}) inv_k,
//   backward e_k <- e_k - sup_k e_{k+1},
// t overwritten by the solution.  U planes of right-hand sides (and, going
// back, of eliminated values) are loaded before the recursion consumes them,
// so U memory round trips overlap (the factor tables through the read-only
// path); the recursion is an FMA and a multiply per plane.
template <typename T>
__device__ __forceinline__ void thomas_body(const ModeArgs<T>& a, int bx, int by) {
    constexpr int U = 16;
    const int m = bx * blockDim.x + threadIdx.x;
    const int n = by;
    if (m >= a.nfast) return;
    const int nzi = a.nzi;
    const size_t stride = size_t(a.nfast) * a.nslow, o = size_t(n) * a.nfast + m;
    T* tc = a.t + o;
    const T* ic = a.inv + o;
    const T* sc = a.sup + o;
    const T cz = a.coef[1].cz;
    T dp = T(0);
    for (int k0 = 0; k0 < nzi; k0 += U) {
        T rhs[U], iv[U];
#pragma unroll
        for (int q = 0; q < U; ++q)
            if (k0 + q < nzi) {
                rhs[q] = tc[(k0 + q) * stride];
                iv[q] = __ldg(ic + (k0 + q) * stride);
            }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int k = k0 + q;
            if (k < nzi) {
                dp = (k ? fma(-cz, dp, rhs[q]) : rhs[q]) * iv[q];
                tc[k * stride] = dp;
            }
        }
    }
    T x = dp;
    for (int k0 = nzi - 2; k0 >= 0; k0 -= U) {
        T dd[U], cc[U];
#pragma unroll
        for (int q = 0; q < U; ++q)
            if (k0 - q >= 0) {
                dd[q] = tc[(k0 - q) * stride];
                cc[q] = __ldg(sc + (k0 - q) * stride);
            }
#pragma unroll
        for (int q = 0; q < U; ++q)
            if (k0 - q >= 0) {
                x = fma(-cc[q], x, dd[q]);
                tc[(k0 - q) * stride] = x;
            }
    }
}

template <typename T>
__global__ void sep_thomas_kernel(ModeArgs<T> a) {
    thomas_body(a, int(blockIdx.x), int(blockIdx.y));
}

// The same mode systems with more parallelism, for levels whose planes fit
// shared memory: a block takes 32 consecutive fast modes of one slow index,
// stages their right-hand sides and factors for every plane through shared
// memory (coalesced rows; the tile is padded to 33 columns), and a warp solves
// one mode at a time with its lanes over the planes.  Each recurrence of the
// elimination is affine in its carried value,
//   forward  e_k = a_k e_{k-1} + b_k,  a_k = -cz inv_k (a_0 = 0), b_k = t_k inv_k,
//   backward e_k = alpha_k e_{k+1} + e_k,  alpha_k = -sup_k (0 on the top plane),
// so every lane composes the maps of its run of consecutive planes, a warp
// scan of the composed maps (shuffles) gives each lane the value entering its
// run, and the lane then repeats the sequential steps of its run from it.
template <typename T>
__device__ __forceinline__ void scan_body(const ModeArgs<T>& ma, int bx, int by) {
    extern __shared__ __align__(16) unsigned char scan_smem[];
    const int nfast = ma.nfast, nslow = ma.nslow, nzi = ma.nzi;
    const T* __restrict__ inv = ma.inv;
    const T* __restrict__ sup = ma.sup;
    T* __restrict__ t = ma.t;
    constexpr int W = 33;
    T* st = reinterpret_cast<T*>(scan_smem);   // [nzi][W]: right-hand sides, then solution
    T* si = st + size_t(nzi) * W;              // inverse pivots
    T* ss = si + size_t(nzi) * W;              // eliminated super-diagonals
    const int m0 = bx * 32, n = by;
    const int nc = min(32, nfast - m0);
    const size_t stride = size_t(nfast) * nslow, base = size_t(n) * nfast + m0;
    const T cz = ma.coef[1].cz;
    // rows in batches of R per thread, every load of a batch issued before its
    // values are stored (one memory round trip per batch instead of per row)
    constexpr int R = 8;
    const int c_ld = threadIdx.x & 31, r_ld = threadIdx.x >> 5, rstep = blockDim.x >> 5;
    for (int k0 = r_ld; k0 < nzi; k0 += R * rstep) {
        T vt[R], vi[R], vs[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int k = k0 + q * rstep;
            if (k < nzi && c_ld < nc) {
                const size_t gi = k * stride + base + c_ld;
                vt[q] = t[gi];
                vi[q] = __ldg(inv + gi);
                vs[q] = __ldg(sup + gi);
            }
        }
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int k = k0 + q * rstep;
            if (k < nzi && c_ld < nc) {
                st[k * W + c_ld] = vt[q];
                si[k * W + c_ld] = vi[q];
                ss[k * W + c_ld] = vs[q];
            }
        }
    }
    __syncthreads();
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int run = (nzi + 31) / 32;
    const int k0 = min(nzi, lane * run), k1 = min(nzi, k0 + run);
    for (int c = warp; c < nc; c += nw) {
        // forward: compose this lane's maps, scan, then the sequential steps
        T A = T(1), B = T(0);
        for (int k = k0; k < k1; ++k) {
            const T iv = si[k * W + c];
            const T a = k ? -cz * iv : T(0);
            B = fma(a, B, st[k * W + c] * iv);
            A = a * A;
        }
        for (int off = 1; off < 32; off <<= 1) {
            const T Ap = __shfl_up_sync(full, A, off), Bp = __shfl_up_sync(full, B, off);
            if (lane >= off) {
                B = fma(A, Bp, B);
                A = A * Ap;
            }
        }
        T d = __shfl_up_sync(full, B, 1);
        if (lane == 0) d = T(0);
        for (int k = k0; k < k1; ++k) {
            const T iv = si[k * W + c];
            d = (k ? fma(-cz, d, st[k * W + c]) : st[k * W + c]) * iv;
            st[k * W + c] = d;
        }
        __syncwarp();
        // backward: the same from the top plane down
        A = T(1);
        B = T(0);
        for (int k = k1 - 1; k >= k0; --k) {
            const T al = k == nzi - 1 ? T(0) : -ss[k * W + c];
            B = fma(al, B, st[k * W + c]);
            A = al * A;
        }
        for (int off = 1; off < 32; off <<= 1) {
            const T An = __shfl_down_sync(full, A, off), Bn = __shfl_down_sync(full, B, off);
            if (lane + off < 32) {
                B = fma(A, Bn, B);
                A = A * An;
            }
        }
        T x = __shfl_down_sync(full, B, 1);
        if (lane == 31) x = T(0);
        for (int k = k1 - 1; k >= k0; --k) {
            x = k == nzi - 1 ? st[k * W + c] : fma(-ss[k * W + c], x, st[k * W + c]);
            st[k * W + c] = x;
        }
        __syncwarp();
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nzi * 32; e += blockDim.x) {
        const int k = e >> 5, c = e & 31;
        if (c < nc) t[k * stride + base + c] = st[k * W + c];
    }
}

template <typename T>
__global__ void __launch_bounds__(1024) sep_scan_kernel(ModeArgs<T> a) {
    scan_body(a, int(blockIdx.x), int(blockIdx.y));
}

constexpr size_t SCAN_SMEM_MAX = 200 * 1024;
template <typename T>
size_t scan_smem_bytes(int nzi) { return size_t(3) * size_t(nzi) * 33 * sizeof(T); }

// lower-boundary plane: that = rhat / (cf mu_fast(m) + cs mu_slow(n))
template <typename T>
__device__ __forceinline__ void divide_body(const ModeArgs<T>& a, int bx, int by) {
    const int m = bx * blockDim.x + threadIdx.x;
    const int n = by;
    if (m >= a.nfast) return;
    T& t = a.t[size_t(n) * a.nfast + m];
    t = mode_divide(t, a.cf, a.mufast[m], a.cs, a.muslow[n]);
}

template <typename T>
__global__ void sep_divide_kernel(ModeArgs<T> a) {
    divide_body(a, int(blockIdx.x), int(blockIdx.y));
}

// one stage of every item's separable solve (grouped launches)
template <typename T, int KIND>
__global__ void __launch_bounds__(1024) g_sep_kernel(const GSepItem<T>* items, int n, int fmg_step, int gate) {
    int lb;
    const GSepItem<T>* it = glocate(items, n, gate, fmg_step, lb);
    if (!it) return;
    const int bx = lb % it->gx, by = lb / it->gx;
    if constexpr (KIND == SEP_SCAN) scan_body(it->st.mode, bx, by);
    else if constexpr (KIND == SEP_THOMAS) thomas_body(it->st.mode, bx, by);
    else if constexpr (KIND == SEP_PLANE) plane_body(it->st.plane, bx, by);
    else divide_body(it->st.mode, bx, by);
}

bool pow2(int v) { return v > 0 && (v & (v - 1)) == 0; }
int ilog2(int v) {
    int b = 0;
    while ((1 << b) < v) ++b;
    return b;
}

// the mode-solve stage on transformed data t (fast index nfast): tridiagonal
// systems along z with the level's elimination factors (3D; a warp scan per
// mode on FP32 levels whose planes fit shared memory, the plain recurrence
// otherwise) or a division per mode (2D)
template <typename T>
SepStage<T> mode_stage(const Geom& g, int dim, const PlaneCoef<T>* coef, const SepTables& tab, int nfast, int nslow,
                       const T* mufast, const T* muslow, bool ytrans, T* t) {
    SepStage<T> s;
    ModeArgs<T>& m = s.mode;
    m.nfast = nfast;
    m.nslow = nslow;
    m.nzi = dim == 3 ? g.nz - 2 : 1;
    m.coef = coef;
    m.t = t;
    if (dim == 3) {
        m.inv = static_cast<const T*>(tab.inv);
        m.sup = static_cast<const T*>(tab.sup);
        // the scan costs about four times the arithmetic of the plain
        // recurrence: FP32 levels only (in FP64 the plain recurrence is faster)
        if (sizeof(T) == 4 && scan_smem_bytes<T>(m.nzi) <= SCAN_SMEM_MAX) {
            s.kind = SEP_SCAN;
            s.threads = 32 * std::min(32, nfast);   // a warp per mode of the block's 32
            s.grid = dim3((nfast + 31) / 32, nslow);
            s.smem = scan_smem_bytes<T>(m.nzi);
            return s;
        }
        s.kind = SEP_THOMAS;
    } else {
        s.kind = SEP_DIVIDE;
        m.mufast = mufast;
        m.muslow = muslow;
        m.cf = T(1.0 / (ytrans ? g.hy * g.hy : g.hx * g.hx));
        m.cs = T(1.0 / (ytrans ? g.hx * g.hx : g.hy * g.hy));
    }
    s.threads = nfast <= 64 ? 64 : 128;
    s.grid = dim3((nfast + s.threads - 1) / s.threads, nslow);
    return s;
}

template <typename T>
SepStage<T> gemm_stage(const GemmArgs<T>& g, int batch) {
    SepStage<T> s;
    s.kind = SEP_GEMM;
    s.gemm = g;
    s.threads = 256;
    const int tb = s.gemm.tile = gemm_tile_size(g.M, g.N, batch);
    s.grid = dim3((g.N + tb - 1) / tb, (g.M + tb - 1) / tb, batch);
    return s;
}

// The plane transforms as one stage, both directions: along lines of M1
// elements first.  Blocks of plane_results results of either parity (FP64:
// down to one, FP32: four).
template <typename T>
SepStage<T> plane_stage(const PlaneArgs<T>& p, int planes, bool grouped) {
    SepStage<T> s;
    s.kind = SEP_PLANE;
    s.plane = p;
    s.threads = PLANE_T;
    const int Ko1 = (p.M1 + 1) / 2, least = sizeof(T) == 4 ? 4 : 1;
    int sp = plane_results(Ko1, planes, least, grouped);
    while (sp > least && PlaneLayout<T>(p.A, p.M1, sp).total * sizeof(T) > PLANE_SMEM) sp /= 2;
    s.plane.sp = sp;
    s.smem = PlaneLayout<T>(p.A, p.M1, sp).total * sizeof(T);
    s.grid = dim3((Ko1 + sp - 1) / sp, planes);
    return s;
}

// The stages of A e = f on one level, e = out (stored, or added with
// accumulate), f and out pitched level arrays (interior read / written), t1
// and t2 dense scratch of the interior size (t2 may be the array of f).
// Fast transforms: x lines of f -> t1[k][m][j] (transposed), y lines ->
// t2[k][m][n], mode solves, inverse y -> t1[k][j][m] (transposed), inverse
// x -> out, scaled.
// Dense transforms: t1[k][j][m] = sum_i f[k][j][i] Sx[m][i], t2[k][n][m] =
// sum_j Sy[n][j] t1[k][j][m], mode solves, and back the same way.
template <typename T>
void plan_level(const Geom& g, int dim, const PlaneCoef<T>* coef, const SepTables& tab, const T* f, T* t1, T* t2,
                T* out, bool accumulate, std::vector<SepStage<T>>& stages, bool split = false, bool lines = false,
                bool grouped = false) {
    const int nxi = g.nx - 2, nyi = g.ny - 2, nzi = dim == 3 ? g.nz - 2 : 1;
    if (nxi < 1 || nyi < 1 || nzi < 1) return;
    const long long pl = (long long)nxi * nyi;
    const long long off = dim == 3 ? (long long)g.plane + g.px + 1 : (long long)g.px + 1;
    const long long sA = dim == 3 ? (long long)g.plane : 0;
    const T* mux = static_cast<const T*>(tab.mux);
    const T* muy = static_cast<const T*>(tab.muy);
    const T scale = T((2.0 / (g.nx - 1)) * (2.0 / (g.ny - 1)));
    const bool planes = tab.fx || (tab.gp && !lines);
    auto plane = [&](const PlaneArgs<T>& p) {
        if constexpr (sizeof(T) == 8)
            if (tab.gp) return split_plane_stage(p, tab.gp, nzi);
        return plane_stage<T>(p, nzi, grouped);
    };
    if (planes) {   // x lines of f -> t1[k][m][n], mode solves, y lines back and x -> out, scaled
        PlaneArgs<T> p;
        p.A = nyi;
        p.M1 = nxi;
        p.in = f + off;
        p.in_plane = sA;
        p.in_line = g.px;
        p.out = t1;
        p.out_plane = pl;
        p.out_line = nyi;
        p.s1 = static_cast<const T*>(tab.fx);
        p.s2 = static_cast<const T*>(tab.fy);
        stages.push_back(plane(p));
        stages.push_back(mode_stage<T>(g, dim, coef, tab, nyi, nxi, muy, mux, true, t1));
        p.A = nxi;
        p.M1 = nyi;
        p.in = t1;
        p.in_plane = pl;
        p.in_line = nyi;
        p.out = out + off;
        p.out_plane = sA;
        p.out_line = g.px;
        p.s1 = static_cast<const T*>(tab.fy);
        p.s2 = static_cast<const T*>(tab.fx);
        p.scale = scale;
        p.accumulate = accumulate ? 1 : 0;
        stages.push_back(plane(p));
        return;
    }
    if (tab.twx || tab.gp) {
        auto dst = [&](const DstArgs<T>& a) {
            SepStage<T> s;
            s.dst = a;
            if (tab.gp || (split && tab.gx && tab.gy)) {
                s.kind = SEP_SPLIT;
                s.digits = tab.gp ? tab.gp : a.L == g.nx - 1 ? tab.gx : tab.gy;
            } else {
                s.kind = SEP_DST;
                dst_shape<T>(s.dst, s.grid, s.threads, s.smem);
            }
            stages.push_back(s);
        };
        const int Lx = g.nx - 1, Ly = g.ny - 1;
        DstArgs<T> a{};
        a.L = Lx; a.log2n = ilog2(Lx); a.lines = nyi; a.planes = nzi; a.tw = tab.twx; a.scale = T(1);
        a.in = f + off; a.in_plane = sA; a.in_line = g.px;
        a.out = t1; a.out_plane = pl; a.out_line = 1; a.out_elem = nyi;
        dst(a);
        DstArgs<T> b{};
        b.L = Ly; b.log2n = ilog2(Ly); b.lines = nxi; b.planes = nzi; b.tw = tab.twy; b.scale = T(1);
        b.in = t1; b.in_plane = pl; b.in_line = nyi;
        b.out = t2; b.out_plane = pl; b.out_line = nyi; b.out_elem = 1;
        dst(b);
        stages.push_back(mode_stage<T>(g, dim, coef, tab, nyi, nxi, muy, mux, true, t2));
        b.in = t2; b.out = t1; b.out_line = 1; b.out_elem = nxi;
        dst(b);
        a.in = t1; a.in_plane = pl; a.in_line = nxi;
        a.out = out + off; a.out_plane = sA; a.out_line = g.px; a.out_elem = 1;
        a.scale = scale;
        a.accumulate = accumulate ? 1 : 0;
        dst(a);
        return;
    }
    if (sizeof(T) == 8) throw Error(MHS_ERR_BAD_STATE, "separable solve: no FP64 transforms for this level");
    const T* Sx = static_cast<const T*>(tab.sx);
    const T* Sy = static_cast<const T*>(tab.sy);
    stages.push_back(gemm_stage<T>(GemmArgs<T>{nyi, nxi, nxi, f + off, g.px, sA, Sx, nxi, 0, t1, nxi, pl, T(1), 0}, nzi));
    stages.push_back(gemm_stage<T>(GemmArgs<T>{nyi, nxi, nyi, Sy, nyi, 0, t1, nxi, pl, t2, nxi, pl, T(1), 0}, nzi));
    stages.push_back(mode_stage<T>(g, dim, coef, tab, nxi, nyi, mux, muy, false, t2));
    stages.push_back(gemm_stage<T>(GemmArgs<T>{nyi, nxi, nyi, Sy, nyi, 0, t2, nxi, pl, t1, nxi, pl, T(1), 0}, nzi));
    stages.push_back(gemm_stage<T>(
        GemmArgs<T>{nyi, nxi, nxi, t1, nxi, pl, Sx, nxi, 0, out + off, g.px, sA, scale, accumulate ? 1 : 0}, nzi));
}

template <typename T>
void launch_stage(const SepStage<T>& s, cudaStream_t st) {
    switch (s.kind) {
    case SEP_DST: launch_dst_stage<T>(s, st); return;
    case SEP_SPLIT_PLANE:
        if constexpr (sizeof(T) == 8) launch_split_plane(s, st);
        break;
    case SEP_SPLIT:
        if constexpr (sizeof(T) == 8) launch_dst_split(s.dst, s.digits, st);
        return;
    case SEP_GEMM:
        if constexpr (sizeof(T) == 4) gemm_kernel<T><<<s.grid, s.threads, 0, st>>>(s.gemm);
        break;
    case SEP_SCAN:
        allow_smem(sep_scan_kernel<T>, SCAN_SMEM_MAX);
        sep_scan_kernel<T><<<s.grid, s.threads, s.smem, st>>>(s.mode);
        break;
    case SEP_THOMAS: sep_thomas_kernel<T><<<s.grid, s.threads, 0, st>>>(s.mode); break;
    case SEP_PLANE:
        allow_smem(sep_dense_kernel<T>, PLANE_SMEM);
        sep_dense_kernel<T><<<s.grid, s.threads, s.smem, st>>>(s.plane);
        break;
    default: sep_divide_kernel<T><<<s.grid, s.threads, 0, st>>>(s.mode); break;
    }
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

}  // namespace

template <typename T>
void launch_sep_stage(const SepStage<T>& s, cudaStream_t st) {
    launch_stage<T>(s, st);
}
template void launch_sep_stage<double>(const SepStage<double>&, cudaStream_t);
template void launch_sep_stage<float>(const SepStage<float>&, cudaStream_t);

namespace {

template <typename T>
void level_solve(mhs_ctx* c, const Geom& g, int dim, const PlaneCoef<T>* coef, const SepTables& tab, const T* f,
                 T* t1, T* t2, T* out, bool accumulate, bool split = false, bool lines = false) {
    std::vector<SepStage<T>> stages;
    plan_level<T>(g, dim, coef, tab, f, t1, t2, out, accumulate, stages, split, lines);
    for (const SepStage<T>& s : stages) launch_stage<T>(s, c->stream);
}

// the stages of a level with folded matrices, one transform per launch (same results)
template <typename T>
void staged_lines(mhs_ctx* c, const Geom& g, int dim, const SepTables& tab, const SepStage<T>& modes, const T* f, T* t,
                  T* w, T* out) {
    const int nxi = g.nx - 2, nyi = g.ny - 2, nzi = dim == 3 ? g.nz - 2 : 1;
    const long long pl = (long long)nxi * nyi;
    const long long off = dim == 3 ? (long long)g.plane + g.px + 1 : (long long)g.px + 1;
    const long long sA = dim == 3 ? (long long)g.plane : 0;
    const T *sx = static_cast<const T*>(tab.fx), *sy = static_cast<const T*>(tab.fy);
    auto pass = [&](int lines, int M, const T* in, long long ip, long long il, T* o, long long op, long long ol,
                    long long oe, const T* s, T scale) {
        constexpr int LB = LINE_Y * plane_r<T>();
        sep_line_kernel<T><<<dim3((M + 63) / 64, (lines + LB - 1) / LB, nzi), dim3(64, LINE_Y), 0, c->stream>>>(
            lines, M, in, ip, il, o, op, ol, oe, s, scale, 0);
        count_launches(1);
        MHS_CUDA(cudaGetLastError());
    };
    pass(nyi, nxi, f + off, sA, g.px, w, pl, 1, nyi, sx, T(1));        // x lines -> w[k][m][j]
    pass(nxi, nyi, w, pl, nyi, t, pl, nyi, 1, sy, T(1));               // y lines -> t[k][m][n]
    launch_stage<T>(modes, c->stream);
    pass(nxi, nyi, t, pl, nyi, w, pl, 1, nxi, sy, T(1));               // back along y -> w[k][j][m]
    pass(nyi, nxi, w, pl, nxi, out + off, sA, g.px, 1, sx, T((2.0 / (g.nx - 1)) * (2.0 / (g.ny - 1))));
}

// a lower-boundary level with folded matrices in one cluster; false when no
// cluster of the kernel fits (nothing launched)
template <typename T>
bool dense2d_solve(const std::vector<SepStage<T>>& st, cudaStream_t stream) {
    PlaneArgs<T> f = st[0].plane, b = st[2].plane;
    const ModeArgs<T>& m = st[1].mode;
    const int Kox = (f.M1 + 1) / 2, Koy = (f.A + 1) / 2, r = plane_r<T>();
    const void* fn = reinterpret_cast<const void*>(&sep_dense2d_kernel<T>);
    auto slab = [&](int K, int c) { return ((K + c - 1) / c + r - 1) / r * r; };
    static PerDevice<std::pair<int, int>, int> sizes;   // cluster size of (nxi, nyi), 0: none
    const int c = sizes.get(current_device(), {f.M1, f.A}, [&] {
        int size = 0;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(PLANE_SMEM)) == cudaSuccess &&
            cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
            for (int n = 16; n >= 1 && !size; n /= 2) {
                const size_t smem = dense2d_smem<T>(f.M1, f.A, slab(Kox, n), slab(Koy, n));
                if (smem > PLANE_SMEM) break;
                if (n > 1 && (n / 2) * r >= std::max(Kox, Koy)) continue;   // fewer CTAs suffice
                cudaLaunchConfig_t cfg{};
                cudaLaunchAttribute attr{};
                attr.id = cudaLaunchAttributeClusterDimension;
                attr.val.clusterDim.x = n;
                attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
                cfg.gridDim = dim3(n, 1, 1);
                cfg.blockDim = dim3(PLANE_T, 1, 1);
                cfg.dynamicSmemBytes = smem;
                cfg.attrs = &attr;
                cfg.numAttrs = 1;
                int clusters = 0;
                if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) == cudaSuccess && clusters > 0) size = n;
            }
        (void)cudaGetLastError();
        return size;
    });
    if (c == 0) return false;
    f.sp = slab(Kox, c);
    b.sp = slab(Koy, c);
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = c;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.gridDim = dim3(c, 1, 1);
    cfg.blockDim = dim3(PLANE_T, 1, 1);
    cfg.dynamicSmemBytes = dense2d_smem<T>(f.M1, f.A, f.sp, b.sp);
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    MHS_CUDA(cudaLaunchKernelEx(&cfg, sep_dense2d_kernel<T>, f, b, m.cf, m.cs, m.mufast, m.muslow));
    count_launches(1);
    return true;
}

template <typename T>
LevelArrays<T>& arrays_of(Hierarchy& H, int l);
template <>
LevelArrays<double>& arrays_of<double>(Hierarchy& H, int l) { return H.d[l]; }
template <>
LevelArrays<float>& arrays_of<float>(Hierarchy& H, int l) { return H.s[l]; }
template <typename T>
std::vector<SepTables>& tables_of(Hierarchy& H) { return sizeof(T) == 8 ? H.sep64 : H.sep32; }

// elimination factors of level l's mode systems from the current coefficients
template <typename T>
void compute_pivots(mhs_ctx* c, Hierarchy& H, int l, SepTables& t) {
    const Geom& g = H.g[l];
    if (H.dim != 3 || !t.inv) return;
    const bool ytrans = t.twx != nullptr || t.fx != nullptr || t.gp != nullptr;
    const int nxi = g.nx - 2, nyi = g.ny - 2;
    const int nfast = ytrans ? nyi : nxi, nslow = ytrans ? nxi : nyi;
    const int threads = nfast <= 64 ? 64 : 128;
    sep_pivot_kernel<T><<<dim3((nfast + threads - 1) / threads, nslow), threads, 0, c->stream>>>(
        nfast, nslow, g.nz - 2, ytrans ? g.ny : g.nx, ytrans ? g.nx : g.ny, H.d[l].coef, ytrans ? 1 : 0,
        static_cast<T*>(t.inv), static_cast<T*>(t.sup));
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

template <typename T>
const SepTables& tables(Hierarchy& H, int l) {
    std::vector<SepTables>& v = tables_of<T>(H);
    if (size_t(l) >= v.size() || !v[l].ready) throw Error(MHS_ERR_BAD_STATE, "separable solver tables not built");
    return v[l];
}

}  // namespace

bool sep_level_ok(const Geom& g) {
    return (pow2(g.nx - 1) && pow2(g.ny - 1)) || (g.nx <= 66 && g.ny <= 66);
}

// The levels whose planes are transformed by plane_body: at most 128 cells a
// side, where there are no fast transforms or they are slower.
template <typename T>
static bool dense_planes(const Geom& g, int dim) {
    const int big = std::max(g.nx, g.ny) - 1, least = sizeof(T) == 4 ? 4 : 1;
    if (big > PLANE_CELLS || PlaneLayout<T>(g.ny - 2, g.nx - 2, least).total * sizeof(T) > PLANE_SMEM ||
        PlaneLayout<T>(g.nx - 2, g.ny - 2, least).total * sizeof(T) > PLANE_SMEM)
        return false;
    return !(pow2(g.nx - 1) && pow2(g.ny - 1)) ||
           dense_planes_faster(sizeof(T) == 8, dim, g.nx - 1, g.ny - 1, dim == 3 ? g.nz - 2 : 1);
}

// Mode eigenvalues, and twiddles or sine matrices, of level l in T, built once
// (FP64 on the host, rounded to T).  Any level: the dense transforms serve
// whatever the node counts (the mixed-mode finest-level solve of long
// non-power-of-two rows among them); the callers that must stay cheap check
// sep_level_ok first.
template <typename T>
void sep_tables(mhs_ctx* c, Hierarchy& H, int l) {
    std::vector<SepTables>& v = tables_of<T>(H);
    if (v.size() < size_t(H.nlev())) v.resize(H.nlev());
    SepTables& t = v[l];
    if (t.ready) return;
    const Geom& g = H.g[l];
    auto upload = [&](const std::vector<T>& h) {
        void* p = nullptr;
        MHS_CUDA(cudaMalloc(&p, std::max<size_t>(h.size(), 1) * sizeof(T)));
        c->allocations.push_back(p);
        c->dev_bytes += round_up(std::max<size_t>(h.size(), 1) * sizeof(T), 256);
        MHS_CUDA(cudaMemcpy(p, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice));
        return p;
    };
    auto mu = [](int n) {
        std::vector<T> m(n - 2);
        for (int q = 1; q <= n - 2; ++q) {
            const double s = std::sin(M_PI * q / (2.0 * (n - 1)));
            m[q - 1] = T(-4.0 * s * s);
        }
        return m;
    };
    auto sine = [](int n) {   // S[m-1][i-1] = sin(pi m i / (n - 1))
        const int ni = n - 2;
        std::vector<T> s(size_t(ni) * ni);
        for (int m = 1; m <= ni; ++m)
            for (int i = 1; i <= ni; ++i) {
                // reduce m i modulo 2 (n - 1) before the sine for an accurate argument
                const long long p = (long long)m * i % (2LL * (n - 1));
                s[size_t(m - 1) * ni + (i - 1)] = T(std::sin(M_PI * double(p) / double(n - 1)));
            }
        return s;
    };
    // folded: element (i, p) of the odd results' matrix is S[2p][i], of the even ones' S[2p+1][i]
    auto folded = [&](int n) {
        const int M = n - 2, Ko = (M + 1) / 2, Ke = M / 2;
        const std::vector<T> S = sine(n);
        std::vector<T> s(size_t(Ko) * Ko + size_t(Ke) * Ke);
        for (int i = 0; i < Ko; ++i)
            for (int p = 0; p < Ko; ++p) s[size_t(i) * Ko + p] = S[size_t(2 * p) * M + i];
        for (int i = 0; i < Ke; ++i)
            for (int p = 0; p < Ke; ++p) s[size_t(Ko) * Ko + size_t(i) * Ke + p] = S[size_t(2 * p + 1) * M + i];
        return s;
    };
    t.mux = upload(mu(g.nx));
    t.muy = upload(mu(g.ny));
    if (dense_planes<T>(g, H.dim)) {
        t.fx = upload(folded(g.nx));
        t.fy = upload(folded(g.ny));
    } else if (sizeof(T) == 8 && H.dim == 3 && l > 0 && split_planes(g)) {   // (direct corrections, l = 0, keep the fast form)
        size_t bytes = 0;
        t.gp = make_split_table(g.nx - 1, &bytes);
        c->allocations.push_back(t.gp);
        c->dev_bytes += round_up(bytes, 256);
    } else if (pow2(g.nx - 1) && pow2(g.ny - 1)) {
        size_t tb = 0;
        t.twx = make_twiddles<T>(g.nx - 1, &tb);
        c->allocations.push_back(t.twx);
        c->dev_bytes += round_up(tb, 256);
        t.twy = make_twiddles<T>(g.ny - 1, &tb);
        c->allocations.push_back(t.twy);
        c->dev_bytes += round_up(tb, 256);
        // the direct solves of the finest level (the lower boundary's lines are as long as the volume's)
        if (sizeof(T) == 8 && l == 0 && split_length(g.nx - 1) && split_length(g.ny - 1)) {
            const std::vector<SepTables>& twin = tables_of<T>(H.dim == 2 ? c->h3 : c->h2);
            const SepTables o = twin.empty() ? SepTables{} : twin[0];
            auto digits = [&](int n, void* have) {
                if (have) return have;
                size_t bytes = 0;
                void* p = make_split_table(n, &bytes);
                c->allocations.push_back(p);
                c->dev_bytes += round_up(bytes, 256);
                return p;
            };
            t.gx = digits(g.nx - 1, o.gx);
            t.gy = digits(g.ny - 1, o.gy ? o.gy : g.ny == g.nx ? t.gx : nullptr);
        }
    } else {
        t.sx = upload(sine(g.nx));
        t.sy = upload(sine(g.ny));
    }
    if (H.dim == 3 && g.nz > 2) {
        const size_t n = size_t(g.nx - 2) * size_t(g.ny - 2) * size_t(g.nz - 2);
        for (void** p : {&t.inv, &t.sup}) {
            MHS_CUDA(cudaMalloc(p, n * sizeof(T)));
            c->allocations.push_back(*p);
            c->dev_bytes += round_up(n * sizeof(T), 256);
        }
        compute_pivots<T>(c, H, l, t);
    }
    t.ready = true;
}

void sep_refresh(mhs_ctx* c, Hierarchy& H) {
    for (size_t l = 0; l < H.sep64.size(); ++l)
        if (H.sep64[l].ready) compute_pivots<double>(c, H, int(l), H.sep64[l]);
    for (size_t l = 0; l < H.sep32.size(); ++l)
        if (H.sep32[l].ready) compute_pivots<float>(c, H, int(l), H.sep32[l]);
}

template <typename T>
void sep_exact(mhs_ctx* c, Hierarchy& H, int l) {
    LevelArrays<T>& A = arrays_of<T>(H, l);
    const Geom& g = H.g[l];
    const SepTables& tab = tables<T>(H, l);
    if (!(c->opts.flags & MHS_FLAG_STAGED_TRANSFORMS) && tab.twx) {
        // per-plane transforms in thread-block clusters (same results as the staged passes)
        const SepStage<T> ms = mode_stage<T>(g, H.dim, A.coef, tab, g.ny - 2, g.nx - 2, static_cast<const T*>(tab.muy),
                                             static_cast<const T*>(tab.mux), true, A.t);
        if (plane_level_solve<T>(g, H.dim, tab, A.f, A.t, A.u, false, &ms, c->stream)) return;
    }
    if (tab.fx) {
        std::vector<SepStage<T>> st;
        plan_level<T>(g, H.dim, A.coef, tab, A.f, A.t, A.r, A.u, false, st);
        if (c->opts.flags & MHS_FLAG_STAGED_TRANSFORMS) {
            staged_lines<T>(c, g, H.dim, tab, st[1], A.f, A.t, A.r, A.u);
            return;
        }
        if (H.dim == 2 && dense2d_solve<T>(st, c->stream)) return;
        for (const SepStage<T>& q : st) launch_stage<T>(q, c->stream);
        return;
    }
    level_solve<T>(c, g, H.dim, A.coef, tab, A.f, A.r, A.t, A.u, false, false,
                   (c->opts.flags & MHS_FLAG_STAGED_TRANSFORMS) != 0);
}

template <typename T>
void sep_exact_plan(mhs_ctx* c, Hierarchy& H, int l, std::vector<SepStage<T>>& stages) {
    (void)c;
    LevelArrays<T>& A = arrays_of<T>(H, l);
    plan_level<T>(H.g[l], H.dim, A.coef, tables<T>(H, l), A.f, A.r, A.t, A.u, false, stages, false, false, true);
}

template <typename T>
void glaunch_sep(const GSepTable<T>& t, int fmg_step, int gate, cudaStream_t st) {
    if (t.n == 0) return;
    switch (t.kind) {
    case SEP_DST: glaunch_dst<T>(t, fmg_step, gate, st); return;
    case SEP_SCAN:
        allow_smem(g_sep_kernel<T, SEP_SCAN>, SCAN_SMEM_MAX);
        g_sep_kernel<T, SEP_SCAN><<<t.blocks, t.threads, t.smem, st>>>(t.items, t.n, fmg_step, gate);
        break;
    case SEP_THOMAS: g_sep_kernel<T, SEP_THOMAS><<<t.blocks, t.threads, 0, st>>>(t.items, t.n, fmg_step, gate); break;
    case SEP_PLANE:
        allow_smem(g_sep_kernel<T, SEP_PLANE>, PLANE_SMEM);
        g_sep_kernel<T, SEP_PLANE><<<t.blocks, t.threads, t.smem, st>>>(t.items, t.n, fmg_step, gate);
        break;
    case SEP_SPLIT_PLANE:
        if constexpr (sizeof(T) == 8) glaunch_split_plane(t, fmg_step, gate, st);
        break;
    default: g_sep_kernel<T, SEP_DIVIDE><<<t.blocks, t.threads, 0, st>>>(t.items, t.n, fmg_step, gate); break;
    }
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

void sep_prepare(mhs_ctx* c, int mode) {
    for (Hierarchy* H : {&c->h3, &c->h2}) {
        if (mode == MHS_MIXED) sep_tables<float>(c, *H, 0);
        else if (sep_fp64_available(c)) sep_tables<double>(c, *H, 0);
    }
}

// e = A^{-1} f on the finest FP32 level of H (interior; e's boundary is left
// as it is); the level's r and t arrays are scratch.
void sep_solve(mhs_ctx* c, Hierarchy& H) { sep_exact<float>(c, H, 0); }

bool sep_fp64_available(const mhs_ctx* c) { return sep_level_ok(c->h3.g[0]); }

// FP64 mode: P += A^{-1} r on the finest level of H, r the residual of the
// latest check (in A.r, consumed), the level's twin t as scratch.
void sep_correct64(mhs_ctx* c, Hierarchy& H) {
    LevelArrays<double>& A = H.d[0];
    level_solve<double>(c, H.g[0], H.dim, A.coef, tables<double>(H, 0), A.r, A.t, A.r, A.u, true, true);
}

template void sep_tables<double>(mhs_ctx*, Hierarchy&, int);
template void sep_tables<float>(mhs_ctx*, Hierarchy&, int);
template void sep_exact<double>(mhs_ctx*, Hierarchy&, int);
template void sep_exact<float>(mhs_ctx*, Hierarchy&, int);
template void sep_exact_plan<double>(mhs_ctx*, Hierarchy&, int, std::vector<SepStage<double>>&);
template void sep_exact_plan<float>(mhs_ctx*, Hierarchy&, int, std::vector<SepStage<float>>&);
template void glaunch_sep<double>(const GSepTable<double>&, int, int, cudaStream_t);
template void glaunch_sep<float>(const GSepTable<float>&, int, int, cudaStream_t);

}  // namespace mhs
