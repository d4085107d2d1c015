// Per-block bodies of the double-float kernels of mixed-precision defect
// correction (kernels_df.cu), with explicit block index b and grid
// dimensions gd, so that grouped launches over many instances run the same
// code with each instance's own block decomposition (see mg_bodies.cuh).
//
// The iterate of the finest level is carried as an unevaluated sum of two
// FP32 words, P = hi + lo (|lo| <= ulp(hi)/2, about 48 significant bits), and
// the outer residual r = f - A P is evaluated with error-free
// transformations instead of FP64 instructions:
//   - TwoSum (Knuth, TAOCP vol. 2, 4.2.2): s + e = a + b exactly;
//   - Fast2Sum (Dekker 1971): the same when |a| >= |b|;
//   - TwoProd with a fused multiply-add: p + e = a * b exactly.
// Intrinsics with explicit rounding (__fadd_rn, ...) keep the compiler from
// contracting or reassociating the transformations.
#pragma once

#include "device_util.cuh"
#include "launch_rules.h"
#include "mhs_internal.h"

namespace mhs {

constexpr int DF_BX = 32, DF_BY = 8;

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}

__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
    p = __fmul_rn(a, b);
    e = __fmaf_rn(a, b, -p);
}

// r = f - A (hi + lo) at one interior node from its stencil values:
// centre C, x neighbours E W, y neighbours N S, z neighbours U D of the high
// and the low words.
template <bool D3, bool FZ = false>
__device__ __forceinline__ float df_stencil(const PlaneCoefDF& c, float hE, float hW, float hN, float hS, float hU,
                                           float hD, float hC, float lE, float lW, float lN, float lS, float lU,
                                           float lD, float lC, float fh, float fl) {
    // neighbour pair sums of the high words, exactly as (sum, error)
    float s1, e1, s2, e2, s3 = 0.f, e3 = 0.f;
    two_sum(hE, hW, s1, e1);
    two_sum(hN, hS, s2, e2);
    if (D3) two_sum(hU, hD, s3, e3);
    const float ch = hC;
    // leading products, exactly as (product, error)
    float px, qx, py, qy, pz = 0.f, qz = 0.f, pd, qd;
    two_prod(c.cxh, s1, px, qx);
    two_prod(c.cyh, s2, py, qy);
    if (D3) two_prod(c.czh, s3, pz, qz);
    two_prod(c.dh, ch, pd, qd);
    // second-order terms (each ~2^-24 of its leading product): plain FP32
    float t = qx + qy + qd;
    t = __fmaf_rn(c.cxh, e1, t);
    t = __fmaf_rn(c.cxl, s1, t);
    t = __fmaf_rn(c.cyh, e2, t);
    t = __fmaf_rn(c.cyl, s2, t);
    t = __fmaf_rn(c.dl, ch, t);
    if (D3) {
        t += qz;
        t = __fmaf_rn(c.czh, e3, t);
        t = __fmaf_rn(c.czl, s3, t);
    }
    // A applied to the low words (about 2^-24 of the total): plain FP32
    float al = c.cxh * (lE + lW) + c.cyh * (lN + lS) + c.dh * lC;
    if (D3) al += c.czh * (lU + lD);
    t += al;
    // exact sum of the leading products, which cancel down to the residual
    float s, e, err;
    two_sum(px, py, s, err);
    if (D3) {
        two_sum(s, pz, s, e);
        err += e;
    }
    two_sum(s, pd, s, e);
    err += e;
    // r = (fh - s) + (fl - err - t); FZ: f = 0, where the sums are exact
    if (FZ) return -s - (err + t);
    float a, b;
    two_sum(fh, -s, a, b);
    return a + (b + (fl - (err + t)));
}

// outer residual rounded to FP32 (r32) with this block's sum of r^2 in
// partial[b.x + gd.x (b.y + gd.y b.z)]; every thread of the block calls it.
// 3D: block b.z takes a contiguous chunk of planes and each thread marches up
// its column, the column's own and vertical-neighbour words kept in
// registers (10 loads per node instead of 14).
template <bool D3>
__device__ __forceinline__ void df_residual_body(const Geom& g, const PlaneCoefDF* __restrict__ cdf,
                                                 const float* __restrict__ hi, const float* __restrict__ lo,
                                                 const float* __restrict__ fh, const float* __restrict__ fl,
                                                 float* __restrict__ r32, double* __restrict__ partial, dim3 b,
                                                 dim3 gd) {
    const int i = 1 + b.x * blockDim.x + threadIdx.x;
    const int j = 1 + b.y * blockDim.y + threadIdx.y;
    float acc = 0.f;
    if (i <= g.nx - 2 && j <= g.ny - 2) {
        const ptrdiff_t sy = g.px, sz = (ptrdiff_t)g.plane;
        if (D3) {
            const int nzi = g.nz - 2, chunk = (nzi + int(gd.z) - 1) / int(gd.z);
            const int k0 = 1 + int(b.z) * chunk, k1 = min(g.nz - 2, k0 + chunk - 1);
            if (k0 <= k1) {
                // one plane ahead: the next plane's loads are issued before the
                // current plane's double-float arithmetic, so their latency overlaps it
                size_t o = at(g, i, j, k0);
                float hD = hi[o - sz], hC = hi[o], lD = lo[o - sz], lC = lo[o];
                float hE = hi[o + 1], hW = hi[o - 1], hN = hi[o + sy], hS = hi[o - sy], hU = hi[o + sz];
                float lE = lo[o + 1], lW = lo[o - 1], lN = lo[o + sy], lS = lo[o - sy], lU = lo[o + sz];
                float fa = fh ? fh[o] : 0.f, fb = fl ? fl[o] : 0.f;
                for (int k = k0; k <= k1; ++k, o += sz) {
                    float nhE = 0.f, nhW = 0.f, nhN = 0.f, nhS = 0.f, nhU = 0.f;
                    float nlE = 0.f, nlW = 0.f, nlN = 0.f, nlS = 0.f, nlU = 0.f, nfa = 0.f, nfb = 0.f;
                    if (k < k1) {
                        const size_t p = o + sz;
                        nhE = hi[p + 1], nhW = hi[p - 1], nhN = hi[p + sy], nhS = hi[p - sy], nhU = hi[p + sz];
                        nlE = lo[p + 1], nlW = lo[p - 1], nlN = lo[p + sy], nlS = lo[p - sy], nlU = lo[p + sz];
                        nfa = fh ? fh[p] : 0.f;
                        nfb = fl ? fl[p] : 0.f;
                    }
                    const float r = df_stencil<true>(cdf[k], hE, hW, hN, hS, hU, hD, hC, lE, lW, lN, lS, lU, lD, lC,
                                                     fa, fb);
                    r32[o] = r;
                    acc = __fmaf_rn(r, r, acc);
                    hD = hC;
                    hC = hU;
                    lD = lC;
                    lC = lU;
                    hE = nhE, hW = nhW, hN = nhN, hS = nhS, hU = nhU;
                    lE = nlE, lW = nlW, lN = nlN, lS = nlS, lU = nlU;
                    fa = nfa, fb = nfb;
                }
            }
        } else {
            const size_t o = at(g, i, j, 0);
            const float r = df_stencil<false>(cdf[0], hi[o + 1], hi[o - 1], hi[o + sy], hi[o - sy], 0.f, 0.f, hi[o],
                                              lo[o + 1], lo[o - 1], lo[o + sy], lo[o - sy], 0.f, 0.f, lo[o],
                                              fh ? fh[o] : 0.f, fl ? fl[o] : 0.f);
            r32[o] = r;
            acc = __fmaf_rn(r, r, acc);
        }
    }
    const double s = block_sum(double(acc));
    if (threadIdx.x == 0 && threadIdx.y == 0) partial[b.x + gd.x * (b.y + gd.y * b.z)] = s;
}

// (hi, lo) + e at one node, renormalised: TwoSum of the high word and e, the
// low word folded into the error, Fast2Sum
__device__ __forceinline__ void df_corrected(float& h, float& l, float e) {
    float s, t;
    two_sum(h, e, s, t);
    t = __fadd_rn(t, l);
    fast_two_sum(s, t, h, l);
}

// The outer residual of wide 3D levels (use_df_quads), alone or together
// with the correction before it (STEP: (hi, lo) + e into (ho, ln), faces
// copied, and the residual of that).  A block marches up a chunk of planes of
// 32 quads (four consecutive x nodes) by eight rows: a warp per row, and two
// warps for the rows below and above the tile, which only provide values.
// Every quad is loaded as 16-byte vectors two planes ahead and corrected once
// (rim rows by both tiles); z neighbours stay in registers, x neighbours
// come by shuffle (past the tile's ends one scalar each), y neighbours
// through shared memory, double-buffered, one barrier per plane.  r32 is
// written as whole quads (0 off the interior).  FZ: f = 0.  Measured at 257^3:
// 78 us for the residual (98 with a thread per node), 101 us with the
// correction (98 + 65 us as two launches); 146 instructions per node at 65 %
// of the issue slots.  Narrower levels keep a thread per node: a warp's 32
// quads would be mostly empty.  Norm partials:
// the residuals of a thread's quad over its planes in FP32, then block_sum
// (the rim warps, the last ones, add zeros, so every form sums in the same
// order).  Every thread of the block (32 x DQ_ROWS) calls it.
constexpr int DQ_X = 32, DQ_Y = 8, DQ_ROWS = DQ_Y + 2;

__host__ __device__ inline bool use_df_quads(const Geom& g) { return g.nz > 1 && (g.nx - 2) / 4 + 1 >= 24; }

struct DfQuad {
    float h[4], l[4];
};
struct DfRaw {   // a quad as loaded: the pair and the correction; the scalar beside the tile likewise
    float4 h, l, e;
    float sh, sl, se;
};

template <bool STEP, bool FZ>
__device__ __forceinline__ void df_march_body(const Geom& g, const PlaneCoefDF* __restrict__ cdf,
                                              const float* __restrict__ e, const float* __restrict__ hi,
                                              const float* __restrict__ lo, float* __restrict__ ho,
                                              float* __restrict__ ln, const float* __restrict__ fh,
                                              const float* __restrict__ fl, float* __restrict__ r32,
                                              double* __restrict__ partial, dim3 b, dim3 gd) {
    __shared__ float4 sh[2][DQ_ROWS][DQ_X], sl[2][DQ_ROWS][DQ_X];
    const int lane = threadIdx.x, w = threadIdx.y;
    const int j0 = int(b.y) * DQ_Y;                                  // row below the tile
    const int slot = w < DQ_Y ? w + 1 : w == DQ_Y ? 0 : DQ_ROWS - 1;   // row of the tile and its rim
    const int j = j0 + slot, x = 4 * (int(b.x) * DQ_X + lane);
    const bool there = j <= g.ny - 1 && x < g.px;
    const bool inrow = j >= 1 && j <= g.ny - 2;
    const bool own = w < DQ_Y && there, inner = own && inrow;
    const bool keep = STEP && there && (w < DQ_Y || j == 0 || j == g.ny - 1);   // rows this block writes
    // the node past the tile's end that lane 0 (west) or lane 31 (east) needs
    const int sx = lane == 0 ? x - 1 : x + 4;
    const bool side = j <= g.ny - 1 && (lane == 0 ? x > 0 : lane == DQ_X - 1 && sx <= g.nx - 1);
    const bool sface = keep && side && lane != 0 && sx == g.nx - 1;   // that node is the x = nx - 1 face: copied too
    const bool sinner = side && sx >= 1 && sx <= g.nx - 2;
    const int sd = sx - x;
    const size_t sz = g.plane;
    const int nzi = g.nz - 2, chunk = (nzi + int(gd.z) - 1) / int(gd.z);
    const int k0 = 1 + int(b.z) * chunk, k1 = min(g.nz - 2, k0 + chunk - 1);
    float acc = 0.f;
    if (k0 <= k1) {
        DfRaw raw{};
        auto load = [&](size_t o, int k) {   // plane k, element o
            if (!there || k > g.nz - 1) return;
            const bool up = STEP && inrow && k >= 1 && k <= g.nz - 2;
            raw.h = *reinterpret_cast<const float4*>(hi + o);
            raw.l = *reinterpret_cast<const float4*>(lo + o);
            raw.e = up ? *reinterpret_cast<const float4*>(e + o) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (side) {
                raw.sh = hi[o + sd];
                raw.sl = lo[o + sd];
                raw.se = up && sinner ? e[o + sd] : 0.f;
            }
        };
        // the corrected words (on the x faces e = 0, which leaves a normalised pair as it is)
        auto corrected = [&](DfQuad& v, float2& s) {
            v = DfQuad{{raw.h.x, raw.h.y, raw.h.z, raw.h.w}, {raw.l.x, raw.l.y, raw.l.z, raw.l.w}};
            s = make_float2(raw.sh, raw.sl);
            if (STEP) {
                df_corrected(v.h[0], v.l[0], raw.e.x);
                df_corrected(v.h[1], v.l[1], raw.e.y);
                df_corrected(v.h[2], v.l[2], raw.e.z);
                df_corrected(v.h[3], v.l[3], raw.e.w);
                df_corrected(s.x, s.y, raw.se);
            }
        };
        auto put = [&](size_t o, const DfQuad& v, float2 s) {
            if (!keep) return;
            *reinterpret_cast<float4*>(ho + o) = make_float4(v.h[0], v.h[1], v.h[2], v.h[3]);
            *reinterpret_cast<float4*>(ln + o) = make_float4(v.l[0], v.l[1], v.l[2], v.l[3]);
            if (sface) {
                ho[o + sd] = s.x;
                ln[o + sd] = s.y;
            }
        };
        size_t o = there ? at(g, x, j, k0) : 0;
        DfQuad D{}, C{}, U{};
        float2 sc = make_float2(0.f, 0.f), sn = sc;
        load(o - sz, k0 - 1);
        corrected(D, sc);
        if (STEP && k0 == 1) put(o - sz, D, sc);   // the face below
        load(o, k0);
        corrected(C, sc);
        load(o + sz, k0 + 1);
        for (int k = k0; k <= k1; ++k, o += sz) {
            const int u = k & 1;
            sh[u][slot][lane] = make_float4(C.h[0], C.h[1], C.h[2], C.h[3]);
            sl[u][slot][lane] = make_float4(C.l[0], C.l[1], C.l[2], C.l[3]);
            if (STEP) put(o, C, sc);
            corrected(U, sn);
            if (k < k1) load(o + 2 * sz, k + 2);
            float4 fa = make_float4(0.f, 0.f, 0.f, 0.f), fb = fa;
            if (!FZ && inner) {
                fa = *reinterpret_cast<const float4*>(fh + o);
                fb = *reinterpret_cast<const float4*>(fl + o);
            }
            float hw = __shfl_up_sync(0xffffffffu, C.h[3], 1), lw = __shfl_up_sync(0xffffffffu, C.l[3], 1);
            float he = __shfl_down_sync(0xffffffffu, C.h[0], 1), le = __shfl_down_sync(0xffffffffu, C.l[0], 1);
            if (lane == 0) hw = sc.x, lw = sc.y;
            if (lane == DQ_X - 1) he = sc.x, le = sc.y;
            // the buffers alternate: a plane's is written again after the next plane's barrier
            __syncthreads();
            if (inner) {
                const float4 Nh = sh[u][slot + 1][lane], Nl = sl[u][slot + 1][lane];
                const float4 Sh = sh[u][slot - 1][lane], Sl = sl[u][slot - 1][lane];
                const float nh[4] = {Nh.x, Nh.y, Nh.z, Nh.w}, nl[4] = {Nl.x, Nl.y, Nl.z, Nl.w};
                const float qh[4] = {Sh.x, Sh.y, Sh.z, Sh.w}, ql[4] = {Sl.x, Sl.y, Sl.z, Sl.w};
                const float ah[4] = {fa.x, fa.y, fa.z, fa.w}, al[4] = {fb.x, fb.y, fb.z, fb.w};
                const PlaneCoefDF c = cdf[k];
                float res[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float r = df_stencil<true, FZ>(
                        c, q < 3 ? C.h[q < 3 ? q + 1 : 3] : he, q ? C.h[q ? q - 1 : 0] : hw, nh[q], qh[q], U.h[q], D.h[q],
                        C.h[q], q < 3 ? C.l[q < 3 ? q + 1 : 3] : le, q ? C.l[q ? q - 1 : 0] : lw, nl[q], ql[q], U.l[q],
                        D.l[q], C.l[q], ah[q], al[q]);
                    res[q] = x + q >= 1 && x + q <= g.nx - 2 ? r : 0.f;
                    acc = __fmaf_rn(res[q], res[q], acc);
                }
                *reinterpret_cast<float4*>(r32 + o) = make_float4(res[0], res[1], res[2], res[3]);
            }
            D = C;
            C = U;
            sc = sn;
        }
        if (STEP && k1 == g.nz - 2) put(o, C, sc);   // the face above
    }
    const double s = block_sum(double(acc));
    if (lane == 0 && w == 0) partial[b.x + gd.x * (b.y + gd.y * b.z)] = s;
}

// blocks of df_march_body: tiles of the quads with interior nodes by eight
// rows, and chunks of planes; at most max_blocks partials
inline dim3 df_march_grid(const Geom& g, int max_blocks) {
    const int gx = ((g.nx - 2) / 4 + 1 + DQ_X - 1) / DQ_X, gy = (g.ny - 2 + DQ_Y - 1) / DQ_Y;
    return dim3(gx, gy, df_march_chunks((long long)gx * gy, g.nz - 2, max_blocks));
}

// (hi, lo) += e
__device__ __forceinline__ void df_correct_body(const Geom& g, int d3, const float* __restrict__ e,
                                                float* __restrict__ hi, float* __restrict__ lo, dim3 b, dim3 gd) {
    const int i = 1 + b.x * blockDim.x + threadIdx.x;
    const int j = 1 + b.y * blockDim.y + threadIdx.y;
    if (i > g.nx - 2 || j > g.ny - 2) return;
    for (int k = d3 ? 1 + b.z : 0; k <= (d3 ? g.nz - 2 : 0); k += gd.z) {
        const size_t o = at(g, i, j, k);
        float h = hi[o], l = lo[o];
        df_corrected(h, l, e[o]);
        hi[o] = h;
        lo[o] = l;
    }
}

// split a double into hi = fl32(x), lo = fl32(x - hi) at interior nodes (zero when f is absent)
__device__ __forceinline__ void df_split_body(const Geom& g, int d3, const double* __restrict__ f,
                                              float* __restrict__ hi, float* __restrict__ lo, dim3 b, dim3 gd) {
    const int i = 1 + b.x * blockDim.x + threadIdx.x;
    const int j = 1 + b.y * blockDim.y + threadIdx.y;
    if (i > g.nx - 2 || j > g.ny - 2) return;
    for (int k = d3 ? 1 + b.z : 0; k <= (d3 ? g.nz - 2 : 0); k += gd.z) {
        const size_t o = at(g, i, j, k);
        const double x = f ? f[o] : 0.0;
        const float h = float(x);
        hi[o] = h;
        lo[o] = float(x - double(h));
    }
}

// a float's double by integer operations (the FP64 pipe, which conversions
// use, is the bound of df_to_double): exponent rebiased, fraction shifted;
// zeros, subnormals, infinities and NaN take the conversion
__device__ __forceinline__ double df_widen(float f) {
    const unsigned u = __float_as_uint(f), a = u & 0x7fffffffu;
    if (a - 0x00800000u < 0x7f000000u)
        return __hiloint2double(int((u & 0x80000000u) | ((a >> 3) + 0x38000000u)), int(u << 29));
    return a == 0 ? __hiloint2double(int(u), 0) : double(f);
}
__device__ __forceinline__ double df_double(float hi, float lo) { return df_widen(hi) + df_widen(lo); }

// P = hi + lo over the whole array (grid-stride over gd.x blocks)
__device__ __forceinline__ void df_to_double_body(size_t n, const float* __restrict__ hi,
                                                  const float* __restrict__ lo, double* __restrict__ P, dim3 b,
                                                  dim3 gd) {
    for (size_t o = b.x * size_t(blockDim.x) + threadIdx.x; o < n; o += size_t(gd.x) * blockDim.x)
        P[o] = df_double(hi[o], lo[o]);
}

__device__ __forceinline__ void df_copy_plane_body(const Geom& g2, const float* __restrict__ hi2,
                                                   const float* __restrict__ lo2, const Geom& g3,
                                                   float* __restrict__ hi3, float* __restrict__ lo3, dim3 b) {
    const int i = b.x * blockDim.x + threadIdx.x;
    const int j = b.y * blockDim.y + threadIdx.y;
    if (i >= g2.nx || j >= g2.ny) return;
    hi3[at(g3, i, j, 0)] = hi2[at(g2, i, j, 0)];
    lo3[at(g3, i, j, 0)] = lo2[at(g2, i, j, 0)];
}

inline dim3 df_grid(const Geom& g, int d3, int max_blocks) {
    const int gx = (g.nx - 2 + DF_BX - 1) / DF_BX;
    const int gy = (g.ny - 2 + DF_BY - 1) / DF_BY;
    int gz = d3 ? g.nz - 2 : 1;
    if (d3 && max_blocks > 0) {
        const int cap = max_blocks / (gx * gy);
        gz = gz > cap ? (cap > 0 ? cap : 1) : gz;
    }
    if (gz > 65535) gz = 65535;
    return dim3(gx, gy, gz);
}
// norm partials: a few blocks per SM, each covering several planes (see residual_grid)
inline dim3 df_residual_grid(const Geom& g, int d3, int max_blocks) {
    if (d3 && use_df_quads(g)) return df_march_grid(g, max_blocks);
    return df_grid(g, d3, max_blocks < 152 * 8 ? max_blocks : 152 * 8);
}
inline dim3 df_plane_grid(const Geom& g2) { return dim3((g2.nx + DF_BX - 1) / DF_BX, (g2.ny + DF_BY - 1) / DF_BY); }
constexpr int DF_TO_DOUBLE_THREADS = 256;

}  // namespace mhs
