// Post-processing of an equilibrium: the quantities the paper's figures show
// (Sect. 3): current density j = curl B / mu0 with its magnitude, |B|, and
// magnetic field lines.
//
// current_kernel: one thread per node, the difference operators of the
// field recovery (central inside, second-order one-sided at the first and
// last node of an axis), FP64.
//
// trace_kernel: one thread per seed; classical fourth-order Runge-Kutta
// along dr/ds = dir B/|B| with B interpolated trilinearly (x, then y, then
// z) from the nodes of the cell holding the point.  A step is taken only
// when its four stage points and its end point lie in the closed box and
// |B| does not vanish at the stage points; otherwise the line ends.  All
// arithmetic uses explicitly rounded FP64 operations (no fused
// multiply-add), in a fixed order, so that a line depends only on B and the
// seed, not on how the compiler schedules the arithmetic.
#include <algorithm>

#include "device_util.cuh"
#include "mhs_internal.h"

namespace mhs {

namespace {

constexpr int BX = 32, BY = 8;

// numerator of d/dx_a at node t of n along one axis, element stride s (times
// 1/(2h): the derivative); the three-point form of either end and the central
// one share their first two terms
__device__ __forceinline__ double num1(const double* __restrict__ f, size_t c, ptrdiff_t s, int t, int n) {
    const bool lo = t == 0, hi = t == n - 1, end = lo || hi;
    const double w0 = lo ? -3.0 : hi ? 3.0 : -1.0, w1 = lo ? 4.0 : hi ? -4.0 : 1.0;
    double v = fma(w1, f[hi ? c - s : c + s], w0 * f[end ? c : c - s]);
    if (end) v += lo ? -f[c + 2 * s] : f[c - 2 * s];
    return v;
}

// j and the magnitudes on dense arrays; wx, wy, wz = 1/(2 h mu0).  A block
// owns 256 consecutive nodes of a plane and `per` consecutive planes.  Bound
// by the FP64 pipe (12 instructions per node for j, 22 for the two
// magnitudes): the scale 1/mu0 is folded into the difference weights, and a
// warp without an edge node takes plain central differences (129^3: 366 ->
// 192 us).
__global__ void __launch_bounds__(BX * BY)
current_kernel(int nx, int ny, int nz, int per, double wx, double wy, double wz, const double* __restrict__ Bx,
               const double* __restrict__ By, const double* __restrict__ Bz, double* __restrict__ jx,
               double* __restrict__ jy, double* __restrict__ jz, double* __restrict__ jmag, double* __restrict__ bmag) {
    const size_t sz = size_t(nx) * ny;
    const size_t e = blockIdx.x * size_t(BX * BY) + threadIdx.x;
    const bool node = e < sz;
    const int j = node ? int(unsigned(e) / unsigned(nx)) : 0;
    const int i = node ? int(unsigned(e) - unsigned(j) * unsigned(nx)) : 0;
    const bool edge = node && (i == 0 || i == nx - 1 || j == 0 || j == ny - 1);
    const int edges = __any_sync(0xffffffffu, edge);
    if (!node) return;
    const ptrdiff_t sy = nx;
    const int k0 = blockIdx.y * per, k1 = min(nz, k0 + per);
    size_t c = e + sz * size_t(k0);
    for (int k = k0; k < k1; ++k, c += sz) {
        double xy, xz, yx, yz, zx, zy;   // differences of B along x of By, Bz; y of Bx, Bz; z of Bx, By
        if (edges || k == 0 || k == nz - 1) {
            xy = num1(By, c, 1, i, nx);
            xz = num1(Bz, c, 1, i, nx);
            yx = num1(Bx, c, sy, j, ny);
            yz = num1(Bz, c, sy, j, ny);
            zx = num1(Bx, c, (ptrdiff_t)sz, k, nz);
            zy = num1(By, c, (ptrdiff_t)sz, k, nz);
        } else {
            xy = By[c + 1] - By[c - 1];
            xz = Bz[c + 1] - Bz[c - 1];
            yx = Bx[c + sy] - Bx[c - sy];
            yz = Bz[c + sy] - Bz[c - sy];
            zx = Bx[c + sz] - Bx[c - sz];
            zy = By[c + sz] - By[c - sz];
        }
        const double cx = fma(yz, wy, -(zy * wz));
        const double cy = fma(zx, wz, -(xz * wx));
        const double cz = fma(xy, wx, -(yx * wy));
        if (jx) jx[c] = cx;
        if (jy) jy[c] = cy;
        if (jz) jz[c] = cz;
        if (jmag) jmag[c] = sqrt_mid(fma(cx, cx, fma(cy, cy, cz * cz)));
        if (bmag) bmag[c] = sqrt_mid(fma(Bx[c], Bx[c], fma(By[c], By[c], Bz[c] * Bz[c])));
    }
}

struct TraceGeom {
    int n[3];
    double L[3];
    size_t px, plane;   // element strides of the B arrays along y and z
};

__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }

// dir * B/|B| at r; false outside the closed box or where |B| = 0
__device__ bool trace_dir(const TraceGeom& G, const double* __restrict__ Bx, const double* __restrict__ By,
                          const double* __restrict__ Bz, double dir, const double r[3], double v[3]) {
    int c[3];
    double f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (!(r[a] >= 0.0 && r[a] <= G.L[a])) return false;
        const double h = __ddiv_rn(G.L[a], double(G.n[a] - 1));
        const double s = __ddiv_rn(r[a], h);
        int i = int(floor(s));
        if (i > G.n[a] - 2) i = G.n[a] - 2;
        if (i < 0) i = 0;
        c[a] = i;
        f[a] = sub(s, double(i));
    }
    const double* B[3] = {Bx, By, Bz};
    double b[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const double* F = B[q];
        double e[2][2];
#pragma unroll
        for (int dz = 0; dz < 2; ++dz)
#pragma unroll
            for (int dy = 0; dy < 2; ++dy) {
                const size_t o = size_t(c[0]) + G.px * size_t(c[1] + dy) + G.plane * size_t(c[2] + dz);
                e[dz][dy] = add(mul(F[o], sub(1.0, f[0])), mul(F[o + 1], f[0]));
            }
        const double e0 = add(mul(e[0][0], sub(1.0, f[1])), mul(e[0][1], f[1]));
        const double e1 = add(mul(e[1][0], sub(1.0, f[1])), mul(e[1][1], f[1]));
        b[q] = add(mul(e0, sub(1.0, f[2])), mul(e1, f[2]));
    }
    const double m = __dsqrt_rn(add(add(mul(b[0], b[0]), mul(b[1], b[1])), mul(b[2], b[2])));
    if (!(m > 0.0)) return false;
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] = __ddiv_rn(mul(dir, b[q]), m);
    return true;
}

__global__ void trace_kernel(TraceGeom G, const double* __restrict__ Bx, const double* __restrict__ By,
                             const double* __restrict__ Bz, const double* __restrict__ seeds, int n, double ds,
                             int max_steps, double dir, double* __restrict__ points, int* __restrict__ lengths) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    double r[3] = {seeds[3 * size_t(q)], seeds[3 * size_t(q) + 1], seeds[3 * size_t(q) + 2]};
    double* out = points + size_t(q) * size_t(max_steps + 1) * 3;
    bool inside = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) inside = inside && r[a] >= 0.0 && r[a] <= G.L[a];
    if (!inside) {
        lengths[q] = 0;
        return;
    }
    out[0] = r[0];
    out[1] = r[1];
    out[2] = r[2];
    int len = 1;
    const double hs = mul(0.5, ds), s6 = __ddiv_rn(ds, 6.0);
    for (int step = 0; step < max_steps; ++step) {
        double k1[3], k2[3], k3[3], k4[3], t[3], e[3];
        if (!trace_dir(G, Bx, By, Bz, dir, r, k1)) break;
#pragma unroll
        for (int a = 0; a < 3; ++a) t[a] = add(r[a], mul(hs, k1[a]));
        if (!trace_dir(G, Bx, By, Bz, dir, t, k2)) break;
#pragma unroll
        for (int a = 0; a < 3; ++a) t[a] = add(r[a], mul(hs, k2[a]));
        if (!trace_dir(G, Bx, By, Bz, dir, t, k3)) break;
#pragma unroll
        for (int a = 0; a < 3; ++a) t[a] = add(r[a], mul(ds, k3[a]));
        if (!trace_dir(G, Bx, By, Bz, dir, t, k4)) break;
        bool ok = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            e[a] = add(r[a], mul(s6, add(add(add(k1[a], mul(2.0, k2[a])), mul(2.0, k3[a])), k4[a])));
            ok = ok && e[a] >= 0.0 && e[a] <= G.L[a];
        }
        if (!ok) break;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            r[a] = e[a];
            out[3 * size_t(len) + a] = e[a];
        }
        ++len;
    }
    lengths[q] = len;
}

// The same lines with four lanes per line: lane a (a < 3) owns coordinate a
// of the point and component a of B, the fourth mirrors the third; cell
// indices, cell fractions and squares of B's components travel by shuffles
// within the four.  Every value is formed by the operations of trace_dir in
// their order, so the lines equal trace_kernel's bit for bit.
//
// Bound by the FP64 pipe (16 cycles of an SM's pipe per warp instruction,
// whatever its active lanes) on few warps: one thread per line runs about 200
// FP64 instructions per stage and 2048 lines fill 64 warps; here a warp
// runs about 60 per stage for its eight lines and 2048 lines make 256 warps.
// 2048 lines of 200 steps through a 129^3 field: 4.59 -> 1.82 ms; what is
// left is the dependent FP64 chain of a stage (32 % of the pipe's cycles).
__device__ __forceinline__ bool trace_dir4(const TraceGeom& G, const double* __restrict__ F, double L, double h, int n,
                                           int a, int base, double dir, double r, double& v) {
    const unsigned full = 0xffffffffu;
    const bool in = r >= 0.0 && r <= L;
    const double s = __ddiv_rn(r, h);
    int i = int(floor(s));
    if (i > n - 2) i = n - 2;
    if (i < 0) i = 0;
    const double f = sub(s, double(i));
    const int cx = __shfl_sync(full, i, base), cy = __shfl_sync(full, i, base + 1), cz = __shfl_sync(full, i, base + 2);
    const double f0 = __shfl_sync(full, f, base), f1 = __shfl_sync(full, f, base + 1), f2 = __shfl_sync(full, f, base + 2);
    const size_t o = size_t(cx) + G.px * size_t(cy) + G.plane * size_t(cz);
    double e[2][2];
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            const size_t q = o + G.px * size_t(dy) + G.plane * size_t(dz);
            e[dz][dy] = add(mul(F[q], sub(1.0, f0)), mul(F[q + 1], f0));
        }
    const double e0 = add(mul(e[0][0], sub(1.0, f1)), mul(e[0][1], f1));
    const double e1 = add(mul(e[1][0], sub(1.0, f1)), mul(e[1][1], f1));
    const double b = add(mul(e0, sub(1.0, f2)), mul(e1, f2));
    const double bb = mul(b, b);
    const double b0 = __shfl_sync(full, bb, base), b1 = __shfl_sync(full, bb, base + 1),
                 b2 = __shfl_sync(full, bb, base + 2);
    const double m = __dsqrt_rn(add(add(b0, b1), b2));
    v = __ddiv_rn(mul(dir, b), m);
    // every coordinate in the box (the four lanes of the line) and |B| > 0
    const unsigned inside = __ballot_sync(full, in) >> base;
    return (inside & 15u) == 15u && m > 0.0;
}

constexpr int TRACE4_THREADS = 32;

__global__ void __launch_bounds__(TRACE4_THREADS)
trace4_kernel(TraceGeom G, const double* __restrict__ Bx, const double* __restrict__ By, const double* __restrict__ Bz,
              const double* __restrict__ seeds, int n, double ds, int max_steps, double dir, double* __restrict__ points,
              int* __restrict__ lengths) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, base = lane & ~3, a = min(lane & 3, 2);
    const int q = blockIdx.x * (TRACE4_THREADS / 4) + threadIdx.x / 4;
    const bool line = q < n, own = line && (lane & 3) < 3;
    const double* F = a == 0 ? Bx : a == 1 ? By : Bz;
    const double L = a == 0 ? G.L[0] : a == 1 ? G.L[1] : G.L[2];
    const int na = a == 0 ? G.n[0] : a == 1 ? G.n[1] : G.n[2];
    const double h = __ddiv_rn(L, double(na - 1));
    double r = line ? seeds[3 * size_t(q) + a] : 0.0;
    double* out = points + size_t(line ? q : 0) * size_t(max_steps + 1) * 3 + a;
    // the warp's lines advance together; a line that has ended idles
    // (warp votes stand in statements of their own: every lane takes part)
    const unsigned start = __ballot_sync(full, r >= 0.0 && r <= L) >> base;
    bool alive = line && (start & 15u) == 15u;
    int len = alive ? 1 : 0;
    if (alive && own) out[0] = r;
    const double hs = mul(0.5, ds), s6 = __ddiv_rn(ds, 6.0);
    for (int step = 0; step < max_steps; ++step) {
        const int any = __any_sync(full, alive);
        if (!any) break;
        double k1, k2, k3, k4;
        bool ok = trace_dir4(G, F, L, h, na, a, base, dir, r, k1);
        ok &= trace_dir4(G, F, L, h, na, a, base, dir, add(r, mul(hs, k1)), k2);
        ok &= trace_dir4(G, F, L, h, na, a, base, dir, add(r, mul(hs, k2)), k3);
        ok &= trace_dir4(G, F, L, h, na, a, base, dir, add(r, mul(ds, k3)), k4);
        const double e = add(r, mul(s6, add(add(add(k1, mul(2.0, k2)), mul(2.0, k3)), k4)));
        const unsigned taken = __ballot_sync(full, ok && e >= 0.0 && e <= L) >> base;
        alive = alive && (taken & 15u) == 15u;
        if (alive) {
            r = e;
            if (own) out[3 * size_t(len)] = e;
            ++len;
        }
    }
    if (line && (lane & 3) == 0) lengths[q] = len;
}

}  // namespace

void launch_current(const Geom& g, double mu0, const double* Bx, const double* By, const double* Bz, double* jx,
                    double* jy, double* jz, double* jmag, double* bmag, cudaStream_t st) {
    // about eight blocks per SM, chunks of at most 16 planes
    const long long pl = ((long long)g.nx * g.ny + BX * BY - 1) / (BX * BY);
    const int per = int(std::min<long long>(16, std::max<long long>(1, pl * g.nz / (152 * 8))));
    const double m = 1.0 / mu0;
    current_kernel<<<dim3(unsigned(pl), (g.nz + per - 1) / per), BX * BY, 0, st>>>(
        g.nx, g.ny, g.nz, per, 0.5 / g.hx * m, 0.5 / g.hy * m, 0.5 / g.hz * m, Bx, By, Bz, jx, jy, jz, jmag, bmag);
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

// Four lanes per line up to the count of lines that gives the one-lane form a
// warp per SM; past it the one-lane form's smaller total (no duplicated
// square roots and votes) wins, as both then keep every SM's FP64 pipe busy.
constexpr int TRACE4_LINES = 32 * 152;

void launch_trace(int nx, int ny, int nz, double Lx, double Ly, double Lz, size_t px, size_t plane, const double* Bx,
                  const double* By, const double* Bz, const double* seeds, int n, double ds, int max_steps,
                  double dir, double* points, int* lengths, cudaStream_t st) {
    if (n <= 0) return;
    TraceGeom G{{nx, ny, nz}, {Lx, Ly, Lz}, px, plane};
    if (n <= TRACE4_LINES) {
        constexpr int per = TRACE4_THREADS / 4;
        trace4_kernel<<<(n + per - 1) / per, TRACE4_THREADS, 0, st>>>(G, Bx, By, Bz, seeds, n, ds, max_steps, dir,
                                                                      points, lengths);
    } else {
        trace_kernel<<<(n + 31) / 32, 32, 0, st>>>(G, Bx, By, Bz, seeds, n, ds, max_steps, dir, points, lengths);
    }
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

}  // namespace mhs
