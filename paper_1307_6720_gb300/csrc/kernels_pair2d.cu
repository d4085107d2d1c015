// Two red-black sweeps of a lower-boundary level in one launch (out of place),
// with the interpolation of the coarse-grid correction before them where asked.
//
// The colour passes of these levels (129^2 to 513^2 nodes) are launches of two
// to three microseconds for well under one of work, eight of them per cycle.
// A block loads a tile of 16 x 16 results with a rim of four nodes (four
// colour passes spread an unknown value by four), adds the interpolated
// correction, keeps f/d and runs the four passes in shared memory.  288
// threads: one pair of x neighbours of the 24 x 24 nodes each, of which either
// colour updates one, so every pass is one update per thread (the FP64 pipe
// charges whole warps).  Every node's operations are those of prolong_body and
// colour_body in their order: the result equals the separate launches bit for
// bit.  Faces are copied, so the output array is complete.
//
// 129^2, FP64: 4.9 us with the interpolation and 4.1 us without, in place of
// four colour passes of 2.4 us each and 2.9 us of prolong_kernel (FP32: 3.3 and
// 2.8 us); the cycle's arithmetic is the chain of four passes, the FP64 latency
// of one update each.
#include "device_util.cuh"
#include "mhs_internal.h"

namespace mhs {

namespace {

constexpr int LT = 16, LR = 4, LW = LT + 2 * LR, LP = LW / 2;

template <typename T, bool PROLONG>
__global__ void __launch_bounds__(LW * LP)
lower_pair_kernel(Geom g, const PlaneCoef<T>* __restrict__ coef, const T* __restrict__ uin, const T* __restrict__ f,
                  T* __restrict__ uout, Geom gc, const T* __restrict__ uc) {
    __shared__ T s[LW][LW + 1];
    const int row = threadIdx.x / LP, lx = 2 * (threadIdx.x - row * LP);
    const int y = int(blockIdx.y) * LT - LR + row, x = int(blockIdx.x) * LT - LR + lx;
    const PlaneCoef<T>& c = coef[0];
    const T inv_d = c.inv_d, ay = -c.ay, ax = -c.ax;
    const bool yin = y >= 1 && y <= g.ny - 2;
    T v[2], fs[2];
    bool in[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int xq = x + q;
        const bool there = xq >= 0 && xq <= g.nx - 1 && y >= 0 && y <= g.ny - 1;
        in[q] = yin && xq >= 1 && xq <= g.nx - 2;
        const size_t o = there ? at(g, xq, y, 0) : 0;
        v[q] = there ? uin[o] : T(0);
        fs[q] = in[q] ? f[o] * inv_d : T(0);
        if (PROLONG && in[q]) {
            const T* k = uc + at(gc, xq >> 1, y >> 1, 0);
            const int py = gc.px;
            if (xq & 1) {
                const T e = k[0] + k[1];
                v[q] = y & 1 ? fma(T(0.25), e + (k[py] + k[py + 1]), v[q]) : fma(T(0.5), e, v[q]);
            } else {
                v[q] = y & 1 ? fma(T(0.5), k[0] + k[py], v[q]) : v[q] + k[0];
            }
        }
        s[row][lx + q] = v[q];
    }
    // the tile's outermost nodes have no neighbours here and stay as they are
    const bool upd0 = in[0] && row >= 1 && row <= LW - 2 && lx >= 1;
    const bool upd1 = in[1] && row >= 1 && row <= LW - 2 && lx + 1 <= LW - 2;
#pragma unroll
    for (int pass = 0; pass < 4; ++pass) {
        __syncthreads();
        // the tile starts at an even node, so colour 0 (x + y even) of a row is at offset row & 1
        const int q = (row + pass) & 1, i = lx + q;
        if (q ? upd1 : upd0) {
            T w = q ? fs[1] : fs[0];
            w = fma(ay, s[row + 1][i] + s[row - 1][i], w);
            s[row][i] = fma(ax, s[row][i + 1] + s[row][i - 1], w);
        }
    }
    __syncthreads();
    if (row >= LR && row < LR + LT && y <= g.ny - 1 && lx >= LR && lx < LR + LT) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (x + q <= g.nx - 1) uout[at(g, x + q, y, 0)] = s[row][lx + q];
    }
}

}  // namespace

template <typename T>
void launch_lower_pair(const Geom& g, const PlaneCoef<T>* coef, const T* u, const T* f, T* out, const Geom* gc,
                       const T* uc, cudaStream_t st) {
    const dim3 grid((g.nx + LT - 1) / LT, (g.ny + LT - 1) / LT);
    if (gc) lower_pair_kernel<T, true><<<grid, LW * LP, 0, st>>>(g, coef, u, f, out, *gc, uc);
    else lower_pair_kernel<T, false><<<grid, LW * LP, 0, st>>>(g, coef, u, f, out, Geom{}, nullptr);
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}
template void launch_lower_pair<double>(const Geom&, const PlaneCoef<double>*, const double*, const double*, double*,
                                        const Geom*, const double*, cudaStream_t);
template void launch_lower_pair<float>(const Geom&, const PlaneCoef<float>*, const float*, const float*, float*,
                                       const Geom*, const float*, cudaStream_t);

}  // namespace mhs
