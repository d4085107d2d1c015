// Double-float outer loop of mixed-precision defect correction: the kernels
// over the bodies of df_bodies.cuh, and their launchers.
//
// On GB300 the FP64 pipe runs at about 1/70 of the FP32 rate, so the ~70 FP32
// instructions per node of the double-float residual cost far less than the
// ~10 FP64 ones they replace.  The residual is exact up to about 1e-14 of
// |A||P|, far below what the 1e-10 stopping test needs; it is then rounded
// to FP32, the right-hand side of the FP32 V-cycles.
#include <algorithm>

#include "check.cuh"
#include "device_util.cuh"
#include "df_bodies.cuh"
#include "mhs_internal.h"

namespace mhs {

namespace {

template <bool D3>
__global__ void df_residual_kernel(Geom g, const PlaneCoefDF* __restrict__ cdf, const float* __restrict__ hi,
                                   const float* __restrict__ lo, const float* __restrict__ fh,
                                   const float* __restrict__ fl, float* __restrict__ r32, double* partial,
                                   CheckArgs ck) {
    df_residual_body<D3>(g, cdf, hi, lo, fh, fl, r32, partial, blockIdx, gridDim);
    check_last_block(ck, partial);
}

__global__ void df_correct_kernel(Geom g, const float* __restrict__ e, float* __restrict__ hi,
                                  float* __restrict__ lo) {
    df_correct_body(g, 1, e, hi, lo, blockIdx, gridDim);
}

template <bool FZ>
__global__ void __launch_bounds__(32 * DQ_ROWS, 2)
df_march_kernel(Geom g, const PlaneCoefDF* __restrict__ cdf, const float* __restrict__ hi, const float* __restrict__ lo,
                const float* __restrict__ fh, const float* __restrict__ fl, float* __restrict__ r32, double* partial,
                CheckArgs ck) {
    df_march_body<false, FZ>(g, cdf, nullptr, hi, lo, nullptr, nullptr, fh, fl, r32, partial, blockIdx, gridDim);
    check_last_block(ck, partial);
}

// One step of defect correction in one pass: the current pair plus e into
// the other pair, and the residual of the result with its norm partials
// (df_march_body).  Apart they read 20 and wrote 12 bytes per node in two
// launches, here 12 and 12; a thread per node also spent half its
// instructions on addresses, which a thread per quad shares.
template <bool FZ>
__global__ void __launch_bounds__(32 * DQ_ROWS, 2)
df_step3_kernel(Geom g, const PlaneCoefDF* __restrict__ cdf, const float* __restrict__ e, DFPair pr,
                const float* __restrict__ fh, const float* __restrict__ fl, float* __restrict__ r32, double* partial,
                CheckArgs ck) {
    const bool flip = *pr.flip != 0;
    df_march_body<true, FZ>(g, cdf, e, flip ? pr.hi[1] : pr.hi[0], flip ? pr.lo[1] : pr.lo[0], flip ? pr.hi[0] : pr.hi[1],
                        flip ? pr.lo[0] : pr.lo[1], fh, fl, r32, partial, blockIdx, gridDim);
    check_last_block(ck, partial);
}

// The same on the lower-boundary plane: every thread corrects its node and
// the four neighbours it reads.
__global__ void __launch_bounds__(DF_BX * DF_BY)
df_step2_kernel(Geom g, const PlaneCoefDF* __restrict__ cdf, const float* __restrict__ e, DFPair pr,
                const float* __restrict__ fh, const float* __restrict__ fl, float* __restrict__ r32, double* partial,
                CheckArgs ck) {
    const bool flip = *pr.flip != 0;
    const float* __restrict__ hi = flip ? pr.hi[1] : pr.hi[0];
    const float* __restrict__ lo = flip ? pr.lo[1] : pr.lo[0];
    float* __restrict__ ho = flip ? pr.hi[0] : pr.hi[1];
    float* __restrict__ ln = flip ? pr.lo[0] : pr.lo[1];
    const int i = 1 + blockIdx.x * blockDim.x + threadIdx.x;
    const int j = 1 + blockIdx.y * blockDim.y + threadIdx.y;
    float acc = 0.f;
    if (i <= g.nx - 2 && j <= g.ny - 2) {
        auto node = [&](int x, int y) {
            const size_t o = at(g, x, y, 0);
            const bool in = x >= 1 && x <= g.nx - 2 && y >= 1 && y <= g.ny - 2;
            float2 v = make_float2(hi[o], lo[o]);
            if (in) df_corrected(v.x, v.y, e[o]);
            if (!in) {   // a face: copied by its inner neighbours
                ho[o] = v.x;
                ln[o] = v.y;
            }
            return v;
        };
        const size_t o = at(g, i, j, 0);
        const float2 C = node(i, j), E = node(i + 1, j), W = node(i - 1, j), N = node(i, j + 1), S = node(i, j - 1);
        // the plane's corners neighbour no inner node
        if ((i == 1 || i == g.nx - 2) && (j == 1 || j == g.ny - 2))
            for (int x = i == 1 ? 0 : g.nx - 1; x <= (i == g.nx - 2 ? g.nx - 1 : 0); x += g.nx - 1)
                for (int y = j == 1 ? 0 : g.ny - 1; y <= (j == g.ny - 2 ? g.ny - 1 : 0); y += g.ny - 1) (void)node(x, y);
        ho[o] = C.x;
        ln[o] = C.y;
        const float r = df_stencil<false>(cdf[0], E.x, W.x, N.x, S.x, 0.f, 0.f, C.x, E.y, W.y, N.y, S.y, 0.f, 0.f, C.y,
                                          fh ? fh[o] : 0.f, fl ? fl[o] : 0.f);
        r32[o] = r;
        acc = __fmaf_rn(r, r, acc);
    }
    const double s = block_sum(double(acc));
    if (threadIdx.x == 0 && threadIdx.y == 0) partial[blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)] = s;
    check_last_block(ck, partial);
}

__global__ void df_split_kernel(Geom g, int d3, const double* __restrict__ f, float* __restrict__ hi,
                                float* __restrict__ lo) {
    df_split_body(g, d3, f, hi, lo, blockIdx, gridDim);
}

// P = hi + lo, four nodes per thread (the arrays' lengths are multiples of four)
__global__ void __launch_bounds__(DF_TO_DOUBLE_THREADS) df_to_double_kernel(size_t n, DFPair pr, double* __restrict__ P) {
    const bool flip = *pr.flip != 0;
    const float4* __restrict__ hi = reinterpret_cast<const float4*>(flip ? pr.hi[1] : pr.hi[0]);
    const float4* __restrict__ lo = reinterpret_cast<const float4*>(flip ? pr.lo[1] : pr.lo[0]);
    double2* __restrict__ out = reinterpret_cast<double2*>(P);
    for (size_t o = blockIdx.x * size_t(blockDim.x) + threadIdx.x; o < n / 4; o += size_t(gridDim.x) * blockDim.x) {
        const float4 h = hi[o], l = lo[o];
        out[2 * o] = make_double2(df_double(h.x, l.x), df_double(h.y, l.y));
        out[2 * o + 1] = make_double2(df_double(h.z, l.z), df_double(h.w, l.w));
    }
}

__global__ void df_coef_kernel(int nz, const PlaneCoef<double>* __restrict__ c, PlaneCoefDF* __restrict__ out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nz) return;
    auto split = [](double x, float& h, float& l) {
        h = float(x);
        l = float(x - double(h));
    };
    PlaneCoefDF d;
    split(c[k].cx, d.cxh, d.cxl);
    split(c[k].cy, d.cyh, d.cyl);
    split(c[k].cz, d.czh, d.czl);
    split(c[k].d, d.dh, d.dl);
    out[k] = d;
}

__global__ void df_copy_plane_kernel(Geom g2, DFPair p2, Geom g3, float* __restrict__ hi3, float* __restrict__ lo3) {
    const bool flip = *p2.flip != 0;
    df_copy_plane_body(g2, flip ? p2.hi[1] : p2.hi[0], flip ? p2.lo[1] : p2.lo[0], g3, hi3, lo3, blockIdx);
}

}  // namespace

void launch_df_coef(const Geom& g, const PlaneCoef<double>* coef, PlaneCoefDF* cdf, cudaStream_t st) {
    df_coef_kernel<<<(g.nz + 127) / 128, 128, 0, st>>>(g.nz, coef, cdf);
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

void launch_df_split(const Geom& g, int dim, const double* f, float* hi, float* lo, cudaStream_t st) {
    const int d3 = dim == 3;
    df_split_kernel<<<df_grid(g, d3, 0), dim3(DF_BX, DF_BY), 0, st>>>(g, d3, f, hi, lo);
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

int launch_df_residual(const Geom& g, int dim, const PlaneCoefDF* cdf, const float* hi, const float* lo,
                       const float* fh, const float* fl, float* r32, double* partial, int max_blocks, cudaStream_t st,
                       const CheckArgs& ck) {
    const int d3 = dim == 3;
    const dim3 grid = df_residual_grid(g, d3, max_blocks);
    if (d3 && use_df_quads(g))
        (fh && fl ? df_march_kernel<false> : df_march_kernel<true>)<<<grid, dim3(DQ_X, DQ_ROWS), 0, st>>>(g, cdf, hi, lo, fh, fl, r32, partial, ck);
    else if (d3)
        df_residual_kernel<true><<<grid, dim3(DF_BX, DF_BY), 0, st>>>(g, cdf, hi, lo, fh, fl, r32, partial, ck);
    else df_residual_kernel<false><<<grid, dim3(DF_BX, DF_BY), 0, st>>>(g, cdf, hi, lo, fh, fl, r32, partial, ck);
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
    return int(grid.x * grid.y * grid.z);
}

bool df_step_available(const Geom& g, int dim) { return dim == 2 || use_df_quads(g); }

int launch_df_step(const Geom& g, int dim, const PlaneCoefDF* cdf, const float* e, const DFPair& p, const float* fh,
                   const float* fl, float* r32, double* partial, int max_blocks, cudaStream_t st, const CheckArgs& ck) {
    const dim3 grid = df_residual_grid(g, dim == 3, max_blocks);
    if (dim == 3)
        (fh && fl ? df_step3_kernel<false> : df_step3_kernel<true>)<<<grid, dim3(DQ_X, DQ_ROWS), 0, st>>>(
            g, cdf, e, p, fh, fl, r32, partial, ck);
    else df_step2_kernel<<<grid, dim3(DF_BX, DF_BY), 0, st>>>(g, cdf, e, p, fh, fl, r32, partial, ck);
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
    return int(grid.x * grid.y * grid.z);
}

void launch_df_correct(const Geom& g, const float* e, float* hi, float* lo, cudaStream_t st) {
    df_correct_kernel<<<df_grid(g, 1, 0), dim3(DF_BX, DF_BY), 0, st>>>(g, e, hi, lo);
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

void launch_df_to_double(const Geom& g, const DFPair& p, double* P, cudaStream_t st) {
    const size_t quads = g.n / 4;
    const int blocks = int(std::min<size_t>(152 * 16, (quads + DF_TO_DOUBLE_THREADS - 1) / DF_TO_DOUBLE_THREADS));
    df_to_double_kernel<<<blocks, DF_TO_DOUBLE_THREADS, 0, st>>>(g.n, p, P);
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

void launch_df_copy_plane(const Geom& g2, const DFPair& p2, const Geom& g3, float* hi3, float* lo3, cudaStream_t st) {
    df_copy_plane_kernel<<<df_plane_grid(g2), dim3(DF_BX, DF_BY), 0, st>>>(g2, p2, g3, hi3, lo3);
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

}  // namespace mhs
