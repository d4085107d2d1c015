// Field recovery (Sect. 2.2, eqs. b_iden, t, pressure, density), FP64.
//
//   B_x = alpha dP/dy + d2P/dxdz,  B_y = -alpha dP/dx + d2P/dydz,
//   B_z = -(d2P/dx2 + d2P/dy2),
//   p   = p_b(z) - xi(z) B_z^2 / (2 mu0),
//   rho = rho_b(z) + [xi'(z) B_z^2/(2 mu0) + xi(z) B.grad(B_z) / mu0] / g.
//
// Derivatives are second-order finite differences: central at inner nodes,
// one-sided three-point (first derivative) and four-point (second
// derivative) stencils on the first and last node of an axis; the mixed
// derivative applies the first-derivative operator along x (or y) to the
// first derivative along z.  B_z takes the compact three-point second
// difference (the operator of eq. lower_bound) or, with bz_mode = 1, the
// first-difference operator applied twice.
//
// P is the pitched level array; the five fields are dense [nz][ny][nx], the
// layout callers receive, so a caller's device array is written by the
// kernels themselves.
#include <algorithm>

#include "device_util.cuh"
#include "mhs_internal.h"

namespace mhs {

namespace {

// Difference weights, formed on the host.
struct FieldWeights {
    double hi[3];      // 1/(2 h) per axis: first differences
    double h2[2];      // 1/h^2 along x and y: second differences
    double m2[2];      // 1/(4 h^2) along x and y: first differences applied twice
    double ax, ay;     // alpha/(2 hy), alpha/(2 hx): alpha dP/dy and alpha dP/dx
    double mxz, myz;   // 1/(4 hx hz), 1/(4 hy hz): mixed derivatives
};

// numerator of the first derivative at node t of n along one axis (times
// 1/(2 h): the derivative) of the values g(o) at element o, stride st; q: the
// offset in nodes.  The three-point form of either end and the central one
// share their first two terms (weights 1 and -1 in the middle), so a warp
// that holds both pays one instruction for it.
template <typename F>
__device__ __forceinline__ double num1(F&& g, size_t o, ptrdiff_t st, int t, int n) {
    const bool lo = t == 0, hi = t == n - 1, end = lo || hi;
    const int q0 = end ? 0 : -1, q1 = hi ? -1 : 1;
    const double w0 = lo ? -3.0 : hi ? 3.0 : -1.0, w1 = lo ? 4.0 : hi ? -4.0 : 1.0;
    double v = fma(w1, g(o + q1 * st, q1), w0 * g(o + q0 * st, q0));
    if (end) {
        const int q2 = lo ? 2 : -2;
        const double last = g(o + q2 * st, q2);
        v += lo ? -last : last;
    }
    return v;
}

// numerator of the compact second derivative (times 1/h^2)
__device__ __forceinline__ double num2(const double* __restrict__ f, size_t o, ptrdiff_t st, int t, int n) {
    if (t == 0 || t == n - 1) {
        const ptrdiff_t q = t == 0 ? st : -st;
        return fma(4.0, f[o + 2 * q], fma(-5.0, f[o + q], fma(2.0, f[o], -f[o + 3 * q])));
    }
    return fma(-2.0, f[o], f[o + st] + f[o - st]);
}

// Per-plane constants: prof[8k + ...] = xi, xi', p_b, rho_b, xi/(2 mu0),
// xi'/(2 mu0 g), xi/(mu0 g).
// Generic path for node (i,j,k): any position, one-sided stencils where needed.
__device__ __noinline__ void field_b_node(const Geom& g, const FieldWeights& w, const double* __restrict__ prof,
                             const double* __restrict__ P, double* __restrict__ Bx, double* __restrict__ By,
                             double* __restrict__ Bz, double* __restrict__ p, int bz_mode, int i, int j, int k) {
    const size_t o = at(g, i, j, k), d = size_t(i) + size_t(g.nx) * (size_t(j) + size_t(g.ny) * size_t(k));
    const ptrdiff_t sy = g.px, sz = (ptrdiff_t)g.plane;
    auto v = [&](size_t q, int) { return P[q]; };
    auto Pz = [&](size_t q, int) { return num1(v, q, sz, k, g.nz); };
    const double bx = fma(w.ax, num1(v, o, sy, j, g.ny), num1(Pz, o, 1, i, g.nx) * w.mxz);
    const double by = fma(-w.ay, num1(v, o, 1, i, g.nx), num1(Pz, o, sy, j, g.ny) * w.myz);
    double bz;
    if (bz_mode == 1) {
        auto Px = [&](size_t q, int s) { return num1(v, q, 1, i + s, g.nx); };
        auto Py = [&](size_t q, int s) { return num1(v, q, sy, j + s, g.ny); };
        bz = -fma(w.m2[0], num1(Px, o, 1, i, g.nx), w.m2[1] * num1(Py, o, sy, j, g.ny));
    } else {
        bz = -fma(w.h2[0], num2(P, o, 1, i, g.nx), w.h2[1] * num2(P, o, sy, j, g.ny));
    }
    Bx[d] = bx;
    By[d] = by;
    Bz[d] = bz;
    if (p) p[d] = fma(-prof[8 * k + 4], bz * bz, prof[8 * k + 2]);
}

// Boundary nodes (the six faces), enumerated as a flat list so that every
// warp runs the generic path together: planes k = 0 and nz-1, then rows
// j = 0 and ny-1 of the inner planes, then the columns i = 0 and those i = nx-1 of the
// remaining nodes (faces one after the other, so that a warp's nodes take the
// same stencils).
__device__ bool face_node(const Geom& g, long long q, int& i, int& j, int& k) {
    const long long pl = (long long)g.nx * g.ny;
    if (q < 2 * pl) {
        k = q < pl ? 0 : g.nz - 1;
        const unsigned r = unsigned(q < pl ? q : q - pl);
        j = int(r / unsigned(g.nx));
        i = int(r - unsigned(j) * unsigned(g.nx));
        return true;
    }
    q -= 2 * pl;
    const long long rows = (long long)(g.nz - 2) * 2 * g.nx;
    if (q < rows) {
        k = 1 + int(q / (2 * g.nx));
        const int r = int(q % (2 * g.nx));
        j = r < g.nx ? 0 : g.ny - 1;
        i = r < g.nx ? r : r - g.nx;
        return true;
    }
    q -= rows;
    const long long cols = (long long)(g.nz - 2) * (g.ny - 2) * 2;
    if (q < cols) {
        const long long half = cols / 2;
        i = q < half ? 0 : g.nx - 1;
        const unsigned r = unsigned(q < half ? q : q - half);
        k = int(r / unsigned(g.ny - 2));
        j = 1 + int(r - unsigned(k) * unsigned(g.ny - 2));
        ++k;
        return true;
    }
    return false;
}

// Launch shape of the pass over B and p: blocks of 32 x 8 threads, the first
// `faces` blocks over the face list, the rest one tile of 32 x 8 inner
// columns and `per` consecutive inner planes each.
struct FieldGrid {
    int faces, tx, ty, per;
};
constexpr int FIELD_PLANES = 16;   // most planes of a block

// B and p.  Inner nodes (1 <= i, j, k <= n-2) take fixed central stencils: a
// block marches up its planes with the tile and its one-node rim of P in
// shared memory, and the difference dP(k+1) - dP(k-1) of every tile and rim
// node formed once (it enters the mixed derivatives of four neighbours; the
// values are those of differencing at each node).  The FP64 pipe bounds the
// pass: 17.4 instructions per inner node, 20 with the vertical differences
// formed per node; a block runs its pipe at 81 %.  129^3 with the faces, which
// were a launch of their own dividing by h at every node: 146 -> 94 us, 257^3:
// 997 -> 660 us.
constexpr int FT_X = 34, FT_Y = 10;

__global__ void __launch_bounds__(256)
field_b_kernel(Geom g, FieldWeights w, FieldGrid fg, const double* __restrict__ prof,
               const double* __restrict__ P, double* __restrict__ Bx, double* __restrict__ By, double* __restrict__ Bz,
               double* __restrict__ p, int bz_mode) {
    __shared__ double sP[2][FT_Y][FT_X], sD[2][FT_Y][FT_X];
    const int tid = threadIdx.x;
    int b = blockIdx.x;
    if (b < fg.faces) {
        int i, j, k;
        for (long long q = b * 256LL + tid; face_node(g, q, i, j, k); q += fg.faces * 256LL)
            field_b_node(g, w, prof, P, Bx, By, Bz, p, bz_mode, i, j, k);
        return;
    }
    b -= fg.faces;
    const int bx = b % fg.tx, by = (b / fg.tx) % fg.ty, bz = b / (fg.tx * fg.ty);
    const int i0 = bx * 32, j0 = by * 8;   // first rim node
    const int k0 = 1 + bz * fg.per, k1 = min(g.nz - 2, k0 + fg.per - 1);
    const int tx = tid & 31, ty = tid >> 5;
    const int i = i0 + 1 + tx, j = j0 + 1 + ty;
    const bool node = i <= g.nx - 2 && j <= g.ny - 2;
    if (bz_mode != 0) {
        if (node)
            for (int k = k0; k <= k1; ++k) field_b_node(g, w, prof, P, Bx, By, Bz, p, bz_mode, i, j, k);
        return;
    }
    // tile and rim elements of this thread: tid and tid + 256
    const int ha = tid % FT_X, va = tid / FT_X;
    const int e2 = tid + 256, hb = e2 % FT_X, vb = e2 / FT_X;
    const bool la = i0 + ha < g.nx && j0 + va < g.ny;
    const bool lb = e2 < FT_X * FT_Y && i0 + hb < g.nx && j0 + vb < g.ny;
    const double* qa = P + at(g, la ? i0 + ha : 0, la ? j0 + va : 0, k0);
    const double* qb = P + at(g, lb ? i0 + hb : 0, lb ? j0 + vb : 0, k0);
    const size_t pl = g.plane;
    double pa = 0.0, ca = 0.0, na = 0.0, pb = 0.0, cb = 0.0, nb = 0.0;
    if (la) {
        pa = *(qa - pl);
        ca = *qa;
        na = *(qa + pl);
    }
    if (lb) {
        pb = *(qb - pl);
        cb = *qb;
        nb = *(qb + pl);
    }
    size_t o = size_t(i) + size_t(g.nx) * (size_t(j) + size_t(g.ny) * size_t(k0));
    const size_t dpl = size_t(g.nx) * size_t(g.ny);
    for (int k = k0; k <= k1; ++k, o += dpl) {
        const int u = k & 1;
        sP[u][va][ha] = ca;
        sD[u][va][ha] = na - pa;
        if (lb) {
            sP[u][vb][hb] = cb;
            sD[u][vb][hb] = nb - pb;
        }
        pa = ca;
        ca = na;
        pb = cb;
        cb = nb;
        if (k < k1) {   // the plane after next
            qa += pl;
            qb += pl;
            if (la) na = *(qa + pl);
            if (lb) nb = *(qb + pl);
        }
        // the buffers alternate: a plane's are written again only after the next plane's barrier
        __syncthreads();
        if (!node) continue;
        const double c = sP[u][ty + 1][tx + 1];
        const double e = sP[u][ty + 1][tx + 2], ww = sP[u][ty + 1][tx], n = sP[u][ty + 2][tx + 1], s = sP[u][ty][tx + 1];
        const double pxz = (sD[u][ty + 1][tx + 2] - sD[u][ty + 1][tx]) * w.mxz;
        const double pyz = (sD[u][ty + 2][tx + 1] - sD[u][ty][tx + 1]) * w.myz;
        const double vz = -fma(w.h2[0], fma(-2.0, c, e + ww), w.h2[1] * fma(-2.0, c, n + s));
        Bx[o] = fma(w.ax, n - s, pxz);
        By[o] = fma(-w.ay, e - ww, pyz);
        Bz[o] = vz;
        if (p) p[o] = fma(-prof[8 * k + 4], vz * vz, prof[8 * k + 2]);
    }
}

// rho on dense arrays: a block owns 256 consecutive nodes of a plane (whole
// planes, edges among them) and `per` consecutive planes.  With D. = B_z
// differences without their 1/(2 h),
//   rho = rho_b + c5 B_z^2 + c6 (B_x Dx / 2hx + B_y Dy / 2hy + B_z Dz / 2hz),
// the spacings folded into per-plane factors of c6 and the B_z terms
// collected: 10 FP64 instructions per node (9 with h_x = h_y) instead of 12.
// A warp without an edge node takes plain central differences.  The FP64
// pipe bounds the pass: 129^3 with the faces 65 -> 53 us.
// SAME: h_x = h_y (a template parameter, as a runtime choice between two FP64
// expressions is issued both ways under predicates).
template <bool SAME>
__global__ void __launch_bounds__(256)
field_rho_kernel(Geom g, FieldWeights w, int per, const double* __restrict__ prof, const double* __restrict__ Bx,
                 const double* __restrict__ By, const double* __restrict__ Bz, double* __restrict__ rho) {
    __shared__ double fac[FIELD_PLANES][5];   // rho_b, c5, c6/2hx, c6/2hy, c6/2hz of the block's planes
    const int tid = threadIdx.x;
    const int k0 = blockIdx.y * per, k1 = min(g.nz - 1, k0 + per - 1);
    if (tid <= k1 - k0) {
        const double* q = prof + 8 * (k0 + tid);
        fac[tid][0] = q[3];
        fac[tid][1] = q[5];
        for (int a = 0; a < 3; ++a) fac[tid][2 + a] = q[6] * w.hi[a];
    }
    __syncthreads();
    const size_t sz = size_t(g.nx) * size_t(g.ny);
    const size_t e = blockIdx.x * size_t(256) + tid;
    const bool node = e < sz;
    const int j = node ? int(unsigned(e) / unsigned(g.nx)) : 0;
    const int i = node ? int(unsigned(e) - unsigned(j) * unsigned(g.nx)) : 0;
    const ptrdiff_t sy = g.nx;
    const bool edge = node && (i == 0 || i == g.nx - 1 || j == 0 || j == g.ny - 1);
    const int edges = __any_sync(0xffffffffu, edge);
    if (!node) return;
    auto val = [&](size_t q, int) { return Bz[q]; };
    size_t o = e + sz * size_t(k0);
    double lo = k0 > 0 ? Bz[o - sz] : 0.0, c = Bz[o];
    for (int k = k0; k <= k1; ++k, o += sz) {
        const double up = k < g.nz - 1 ? Bz[o + sz] : 0.0;
        double dx, dy, dz;
        if (edges || k == 0 || k == g.nz - 1) {
            dx = num1(val, o, 1, i, g.nx);
            dy = num1(val, o, sy, j, g.ny);
            dz = num1(val, o, (ptrdiff_t)sz, k, g.nz);
        } else {
            dx = Bz[o + 1] - Bz[o - 1];
            dy = Bz[o + sy] - Bz[o - sy];
            dz = up - lo;
        }
        const double* q = fac[k - k0];
        double v = fma(c, fma(q[1], c, q[4] * dz), q[0]);
        if constexpr (SAME) {
            v = fma(q[2], fma(By[o], dy, Bx[o] * dx), v);
        } else {
            v = fma(q[3], By[o] * dy, v);
            v = fma(q[2], Bx[o] * dx, v);
        }
        rho[o] = v;
        lo = c;
        c = up;
    }
}

}  // namespace

void launch_fields(const Geom& g, double alpha, const double* prof, const double* P, double* Bx, double* By,
                   double* Bz, double* p, double* rho, int bz_mode, cudaStream_t st) {
    FieldWeights w;
    w.hi[0] = 1.0 / (2.0 * g.hx);
    w.hi[1] = 1.0 / (2.0 * g.hy);
    w.hi[2] = 1.0 / (2.0 * g.hz);
    w.h2[0] = 1.0 / (g.hx * g.hx);
    w.h2[1] = 1.0 / (g.hy * g.hy);
    w.m2[0] = 1.0 / (4.0 * g.hx * g.hx);
    w.m2[1] = 1.0 / (4.0 * g.hy * g.hy);
    w.ax = alpha / (2.0 * g.hy);
    w.ay = alpha / (2.0 * g.hx);
    w.mxz = 1.0 / (4.0 * g.hx * g.hz);
    w.myz = 1.0 / (4.0 * g.hy * g.hz);
    FieldGrid fg;
    fg.tx = (g.nx - 2 + 31) / 32;
    fg.ty = (g.ny - 2 + 7) / 8;
    // chunks of 4 .. 16 planes, about eight blocks per SM where the level has them
    const long long tiles = (long long)fg.tx * fg.ty;
    fg.per = int(std::min<long long>(FIELD_PLANES, std::max<long long>(4, (tiles * (g.nz - 2) + 152 * 8 - 1) / (152 * 8))));
    const long long faces = 2LL * g.nx * g.ny + 2LL * (g.nz - 2) * g.nx + 2LL * (g.nz - 2) * (g.ny - 2);
    fg.faces = int(std::min<long long>((faces + 255) / 256, 152 * 16));
    const long long blocks = fg.faces + tiles * ((g.nz - 2 + fg.per - 1) / fg.per);
    if (blocks > 0x7fffffffLL) throw Error(MHS_ERR_INVALID_ARG, "field recovery: grid too large");
    field_b_kernel<<<unsigned(blocks), 256, 0, st>>>(g, w, fg, prof, P, Bx, By, Bz, p, bz_mode);
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
    if (!rho) return;
    const long long pl = ((long long)g.nx * g.ny + 255) / 256;
    const int per = int(std::min<long long>(FIELD_PLANES, std::max<long long>(2, pl * g.nz / (152 * 8))));
    const auto rho_kernel = w.hi[0] == w.hi[1] ? field_rho_kernel<true> : field_rho_kernel<false>;
    rho_kernel<<<dim3(unsigned(pl), (g.nz + per - 1) / per), 256, 0, st>>>(g, w, per, prof, Bx, By, Bz, rho);
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

}  // namespace mhs
