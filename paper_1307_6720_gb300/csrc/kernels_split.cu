// FP64 sine transforms of long lines on the tensor cores, by exact splitting.
//
// The FP64 pipe (two lanes per clock and SM) is the bound of the fast
// transforms: 26 FP64 instructions per element at 257 nodes.  Here a line is a
// dense product with the folded sine matrices (half the side: the sums of
// mirrored elements give the odd results, the differences the even ones) in
// fixed point, formed from exact small integer products (Ozaki, Ogita, Oishi
// and Rump, Numer. Algorithms 59, 2012):
//
// - the folded elements become integers of up to 2^55 relative to their line's
//   largest exponent, x = sum_i a_i 256^(6-i), seven digits in [-128, 127] (the
//   first up to 128); likewise the matrix entries, scaled by 2^55;
// - digits are exact in FP16, a product of two is at most 2^14, and a sum of up
//   to 7 x 128 of them stays below 2^24, so FP32 accumulation is exact; the
//   products with i + j = d share the accumulator of order d, d <= 7 (34
//   products of digit matrices; those left out lie below 2^-59 of the line's
//   largest element each);
// - the eight integers of a result are put together in 64 bits, rounded once
//   and written as a double, all by integer instructions (conversions between
//   64-bit integers and doubles run at the FP64 pipe's rate: 650 us a pass);
//   what is left to the FP64 pipe is the folding and the scaling of the last pass.
//
// mma.sync (m16n8k16) rather than tcgen05: the eight accumulators of a result
// meet in one thread and the digits are made in the fragments' layout.  Two
// warps share the digits of 16 lines of one parity in shared memory (29 KB at
// 256 cells), each forms half of their results, two column tiles at a time, so
// that three blocks (12 warps) fit an SM; the matrices' digits stream from L2
// in fragment order, one tile ahead.  Four tiles per warp with two warps' worth
// of registers and lines of its own ran at two warps per scheduler: 550 us.
//
// One pass over 255^3, in place of 733 us of the fast transform: 374 us to 420 us
// (strided stores), tensor pipe 67 % busy; the rest is the digits and putting
// results together (2.7 other instructions per product).  Over one plane of
// 255^2, where the results are spread over blocks: 17.5 us, was 27 us.
//
// Against the exact solution of the discrete equations, one direct step
// (four transforms in each problem), fast transforms -> these, 2-norm:
// 129^3 lower boundary 2.4e-15 -> 0.8e-15, volume 1.89e-14 -> 1.84e-14 (the
// tridiagonal solves'); 257 x 129 x 17 3.3e-15 -> 1.0e-15 and 4.7e-15 -> 2.4e-15;
// 257 x 257 x 33 6.0e-15 -> 1.4e-15 and 8.7e-15 -> 4.9e-15, its residual
// 4.5e-14 -> 2.6e-15.  Lines with an infinity or NaN become NaN.
#include <cuda_fp16.h>

#include <cmath>
#include <vector>

#include "device_util.cuh"
#include "dst_body.cuh"
#include "group.h"
#include "mhs_internal.h"
#include "solver.h"

namespace mhs {

namespace {

constexpr int DIG = 7;               // digits
constexpr int ORDERS = 8;            // of products of digits that are kept
constexpr int STEP = DIG * 128 + 4;   // words of a k step's digits of 16 lines (four more than they fill: lanes on other banks)
constexpr int SW = 4;                // warps of a block, two to 16 lines
constexpr int TILES = 2;             // column tiles of 8 results that a warp forms at a time
constexpr long long BIAS = 0x80808080808080LL;   // 128 in every digit

__device__ __forceinline__ void mma16816(float (&d)[4], const uint4& a, const uint2& b) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y));
}

// biased exponent (subnormals as exponent 1)
__device__ __forceinline__ int expo(double x) {
    const int e = (__double2hiint(x) >> 20) & 0x7ff;
    return e ? e : 1;
}

// x 2^(1077 - emax) rounded to an integer (|.| <= 2^55 for exponents up to emax)
__device__ __forceinline__ long long fixed(double x, int emax) {
    const unsigned hi = unsigned(__double2hiint(x)), ex = (hi >> 20) & 0x7ffu;
    const unsigned long long m =
        static_cast<unsigned long long>(__double_as_longlong(x) & 0xfffffffffffffLL) | (ex ? 0x10000000000000ull : 0ull);
    const int sh = emax - int(ex ? ex : 1u);
    const long long q = static_cast<long long>(sh > 60 ? 0ull : ((m << 2) + ((1ull << sh) >> 1)) >> sh);
    return (hi >> 31) ? -q : q;
}

// v 2^k as a double, rounded to nearest (ties away)
__device__ __forceinline__ double widened(long long v, int k) {
    const unsigned long long m0 = v < 0 ? 0ull - static_cast<unsigned long long>(v) : static_cast<unsigned long long>(v);
    if (m0 == 0) return 0.0;
    const int lz = __clzll(static_cast<long long>(m0));
    const unsigned long long m = (m0 << lz) >> 1;                 // leading bit 62
    const unsigned long long r = (m + (1ull << 9)) >> 10;         // 53 bits, or 2^53 after a carry
    const int e = 1023 + k + 63 - lz;                              // exponent field of the leading bit
    if (e < 1 || e > 2045) return scalbn(double(v), k);           // near the ends of the range
    const unsigned long long bits = (static_cast<unsigned long long>(e - 1) << 52) + r;   // the leading bit (and a carry) add to it
    return __longlong_as_double(static_cast<long long>(bits | (v < 0 ? 0x8000000000000000ull : 0ull)));
}

// Digits of the two folded elements f of row r at k, k + 1, relative to 2^(e - 1077)
__device__ __forceinline__ void put_digits(unsigned* A, int r, int k, double f0, double f1, int e) {
    const unsigned long long q0 = static_cast<unsigned long long>(fixed(f0, e) + BIAS);
    const unsigned long long q1 = static_cast<unsigned long long>(fixed(f1, e) + BIAS);
    const __half2 off = __halves2half2(__ushort_as_half(0xe480), __ushort_as_half(0xe480));   // -1152
    const int ks = k >> 4, kk = k & 15;
    unsigned* word = A + ks * STEP + (((r & 7) * 4 + ((kk & 7) >> 1)) << 2) + (r >> 3) + 2 * (kk >> 3);
#pragma unroll
    for (int s = 0; s < DIG; ++s) {
        const int b = DIG - 1 - s;   // byte of digit s
        const unsigned u0 = b < 4 ? unsigned(q0) : unsigned(q0 >> 32);
        const unsigned u1 = b < 4 ? unsigned(q1) : unsigned(q1 >> 32);
        // 1024 + byte, twice (the first digit may be 128: nine bits)
        const unsigned h = s == 0 ? __byte_perm(u0, u1, 0x7632) | 0x64006400u
                                  : __byte_perm(__byte_perm(u0, u1, (b & 3) | ((4 + (b & 3)) << 4)), 0x64646464u, 0x4140);
        const __half2 d = __hadd2(*reinterpret_cast<const __half2*>(&h), off);
        word[s * 128] = *reinterpret_cast<const unsigned*>(&d);
    }
}

// largest exponent of a line held by L lanes
template <int L>
__device__ __forceinline__ int line_max(int e) {
    if constexpr (L == 32) return int(__reduce_max_sync(0xffffffffu, unsigned(e)));
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    return e;
}

// The digit products of 16 rows with TILES column tiles; bt: the first tile's
// digits [tile][k step][digit][lane], at this lane, loaded one tile ahead
template <int KS>
__device__ __forceinline__ void products(const unsigned* A, const uint2* __restrict__ bt, int lane,
                                         float (&acc)[TILES][ORDERS][4]) {
    static_assert(DIG * 16LL * KS * 128 * 128 < 1LL << 24, "sums of digit products must be exact in FP32");
#pragma unroll
    for (int n = 0; n < TILES; ++n)
#pragma unroll
        for (int d = 0; d < ORDERS; ++d)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[n][d][c] = 0.f;
    auto load_b = [&](uint2(&v)[DIG], int ks, int n) {
#pragma unroll
        for (int s = 0; s < DIG; ++s) v[s] = __ldg(bt + ((n * KS + ks) * DIG + s) * 32);
    };
    uint2 bn[DIG];
    load_b(bn, 0, 0);
#pragma unroll 1
    for (int ks = 0; ks < KS; ++ks) {
        uint4 av[DIG];
#pragma unroll
        for (int s = 0; s < DIG; ++s) av[s] = *reinterpret_cast<const uint4*>(A + ks * STEP + s * 128 + 4 * lane);
#pragma unroll
        for (int n = 0; n < TILES; ++n) {
            uint2 bv[DIG];
#pragma unroll
            for (int s = 0; s < DIG; ++s) bv[s] = bn[s];
            if (n + 1 < TILES) load_b(bn, ks, n + 1);
            else if (ks + 1 < KS) load_b(bn, ks + 1, 0);
#pragma unroll
            for (int i = 0; i < DIG; ++i)
#pragma unroll
                for (int j = 0; j < DIG && i + j < ORDERS; ++j) mma16816(acc[n][i + j], av[i], bv[j]);
        }
    }
}

// result c of a tile's accumulators, of a row with exponent e
__device__ __forceinline__ double joined(const float (&acc)[ORDERS][4], int c, int e) {
    auto in = [&](int d) { return static_cast<long long>(__float2int_rn(acc[d][c])); };
    const long long top = (in(0) << 24) + (in(1) << 16) + (in(2) << 8) + in(3);
    const long long low = (in(4) << 16) + (in(5) << 8) + in(6) + (in(7) >> 8);
    // 256^7 2^-55 times 2^(e - 1077) of the elements: 2^(e - 1076)
    const double v = widened((top << 16) + ((low + 128) >> 8), e - 1076);
    return e == 2047 ? __longlong_as_double(0x7ff8000000000000LL) : v;
}

// lines of N - 1 elements, N = 32 KS; tab: the matrices' digits in fragment
// order [parity][column tile][k step][digit][lane]
template <int KS>
__global__ void __launch_bounds__(32 * SW, 3) dst_split_kernel(DstArgs<double> a, const uint2* __restrict__ tab) {
    constexpr int Ko = 16 * KS, N = 2 * Ko;
    constexpr int NG = Ko / 16 / TILES;              // groups of tiles of a warp
    constexpr int EP = Ko >= 64 ? Ko / 32 : 2;       // folded elements of a lane
    constexpr int LL = Ko / EP, RW = 32 / LL;        // lanes of a line, lines of a warp
    extern __shared__ __align__(16) unsigned char split_smem[];
    __shared__ int s_e[SW / 2][16];
    const int lane = threadIdx.x & 31, half = (threadIdx.x >> 5) & 1, w = threadIdx.x >> 6;
    unsigned* A = reinterpret_cast<unsigned*>(split_smem) + w * (KS * STEP);
    const long long total = (long long)a.lines * a.planes, first = ((long long)blockIdx.x * (SW / 2) + w) * 16;
    const int g = lane >> 2, t4 = lane & 3, li = lane % LL;
    // the two lines whose results this thread holds
    long long base[2];
    bool live[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const long long gl = first + g + 8 * h;
        live[h] = gl < total;
        const long long pl = live[h] ? gl / a.lines : 0, l = live[h] ? gl - pl * a.lines : 0;
        base[h] = pl * a.out_plane + l * a.out_line;
    }
    // all results, or (few lines, gridDim.y = 2 NG) one group of each warp
    const bool one = gridDim.y > 1;
    const int par0 = one ? blockIdx.y & 1 : 0, par1 = one ? par0 : 1;
    const int ng0 = one ? (blockIdx.y >> 1) * 2 + half : half * NG, ng1 = one ? ng0 + 1 : ng0 + NG;
    for (int par = par0; par <= par1; ++par) {
        // digits of the folded lines, each line loaded while the one before is worked on
        auto load_line = [&](int r, double(&lo)[EP], double(&hi)[EP]) {
            const long long gl = first + r;
            const bool on = gl < total;
            const long long pl = on ? gl / a.lines : 0;
            const double* x = a.in + pl * a.in_plane + (on ? gl - pl * a.lines : 0) * a.in_line;
#pragma unroll
            for (int u = 0; u < EP; ++u) {
                const int i = li * EP + u, j = N - 2 - i;
                lo[u] = on ? x[i] : 0.0;
                // (the middle element is its own mirror: it counts once, in the sums)
                hi[u] = !on ? 0.0 : j != i ? x[j] : par ? lo[u] : 0.0;
            }
        };
        double lo[EP], hi[EP];
        const int r0 = 8 * half + lane / LL, r1 = 8 * half + 8;
        load_line(r0, lo, hi);
#pragma unroll 1
        for (int r = r0; r < r1; r += RW) {
            double f[EP];
            int e = 1;
#pragma unroll
            for (int u = 0; u < EP; ++u) {
                f[u] = par ? lo[u] - hi[u] : lo[u] + hi[u];
                e = max(e, expo(f[u]));
            }
            if (r + RW < r1) load_line(r + RW, lo, hi);
            e = line_max<LL>(e);
            if (li == 0) s_e[w][r] = e;
#pragma unroll
            for (int u = 0; u < EP; u += 2) put_digits(A, r, li * EP + u, f[u], f[u + 1], e);
        }
        __syncthreads();
        for (int ng = ng0; ng < ng1; ++ng) {
            float acc[TILES][ORDERS][4];
            products<KS>(A, tab + (size_t(par) * (Ko / 8) + ng * TILES) * KS * DIG * 32 + lane, lane, acc);
#pragma unroll
            for (int n = 0; n < TILES; ++n)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int h = c >> 1, col = (ng * TILES + n) * 8 + 2 * t4 + (c & 1), m = 2 * col + par;
                    if (!live[h] || m > N - 2) continue;
                    const double v = joined(acc[n], c, s_e[w][g + 8 * h]);
                    double* o = a.out + base[h] + (long long)m * a.out_elem;
                    *o = a.scale == 1.0 && !a.accumulate ? v : dst_result(a.scale, v, a.accumulate != 0, a.accumulate ? *o : 0.0);
                }
        }
        __syncthreads();
    }
}

// Both transforms of a plane of 63 x 63 values (64 cells; the coarse-grid solves
// of 129^3 and 257^3 FP64 cycles): along the lines, then across.  Block (par, plane) forms the lines' odd (par = 0) or even
// results and takes them across by itself, so nothing passes between blocks.
// Eight warps: two to 16 lines of a parity, each for half of their results
// (one group of tiles); the second transforms read the first ones' results
// from shared memory.  63 planes in 126 blocks: 13.5 us, of which the chain of
// loads, digits, products and sums of one block is all; the fast transforms on
// clusters of two blocks took 30 us, 67 % of it FP64 pipe.  A 65^3 level's solve
// 75 -> 42 us, its residual 7e-15 -> 1.6e-15.
constexpr int SP_CELLS = 64, SP_KS = 2, SP_T = 256;

__device__ __forceinline__ void split_plane_body(const PlaneArgs<double>& a, const uint2* __restrict__ tab, int par,
                                                 int plane) {
    constexpr int KS = SP_KS, Ko = 16 * KS, N = SP_CELLS, LD = N + 1;
    __shared__ __align__(16) unsigned s_A[4][KS * STEP];
    __shared__ double s_x[Ko][LD];   // results of the first transforms [mode][line]
    __shared__ int s_e[4][16];
    const int lane = threadIdx.x & 31, half = (threadIdx.x >> 5) & 1, w = threadIdx.x >> 6;
    const int g = lane >> 2, t4 = lane & 3, li = lane & 15, sub = lane >> 4;
    unsigned* A = s_A[w];
    // the digits of rows r, r + 2, .. of 8 half .. 8 half + 7, two rows at a time, of lines x(r)
    auto digits = [&](auto&& line, int p) {
        double lo[4][2], hi[4][2];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const double* x = line(8 * half + 2 * q + sub);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int i = 2 * li + u, j = N - 2 - i;
                lo[q][u] = x ? x[i] : 0.0;
                hi[q][u] = !x ? 0.0 : j != i ? x[j] : p ? lo[q][u] : 0.0;
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = 8 * half + 2 * q + sub;
            const double f0 = p ? lo[q][0] - hi[q][0] : lo[q][0] + hi[q][0];
            const double f1 = p ? lo[q][1] - hi[q][1] : lo[q][1] + hi[q][1];
            const int e = line_max<16>(max(max(1, expo(f0)), expo(f1)));
            if (li == 0) s_e[w][r] = e;
            put_digits(A, r, 2 * li, f0, f1, e);
        }
    };
    auto form = [&](int p, float(&acc)[TILES][ORDERS][4]) {
        products<KS>(A, tab + (size_t(p) * (Ko / 8) + half * TILES) * KS * DIG * 32 + lane, lane, acc);
    };
    float acc[TILES][ORDERS][4];
    const double* in = a.in + plane * a.in_plane;
    digits([&](int r) { return 16 * w + r < a.A ? in + (16 * w + r) * a.in_line : nullptr; }, par);
    __syncthreads();
    form(par, acc);
#pragma unroll
    for (int n = 0; n < TILES; ++n)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int row = g + 8 * (c >> 1), col = (half * TILES + n) * 8 + 2 * t4 + (c & 1);
            s_x[col][16 * w + row] = joined(acc[n], c, s_e[w][row]);
        }
    __syncthreads();
    // 32 lines of both parities: warps 0 .. 3 the first 16, 4 .. 7 the others
    const int p2 = w & 1, l0 = 16 * (w >> 1);
    digits([&](int r) { return &s_x[l0 + r][0]; }, p2);
    __syncthreads();
    form(p2, acc);
#pragma unroll
    for (int n = 0; n < TILES; ++n)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int row = g + 8 * (c >> 1), m = 2 * (l0 + row) + par;
            const int col = (half * TILES + n) * 8 + 2 * t4 + (c & 1), q = 2 * col + p2;
            if (m > N - 2 || q > N - 2) continue;
            const double v = joined(acc[n], c, s_e[w][row]);
            double* o = a.out + plane * a.out_plane + m * a.out_line + q;
            *o = a.scale == 1.0 && !a.accumulate ? v : dst_result(a.scale, v, a.accumulate != 0, a.accumulate ? *o : 0.0);
        }
}

__global__ void __launch_bounds__(SP_T) split_plane_kernel(PlaneArgs<double> a, const uint2* __restrict__ tab) {
    split_plane_body(a, tab, int(blockIdx.x), int(blockIdx.y));
}

__global__ void __launch_bounds__(SP_T) g_split_plane_kernel(const GSepItem<double>* items, int n, int fmg_step, int gate) {
    int lb;
    const GSepItem<double>* it = glocate(items, n, gate, fmg_step, lb);
    if (!it) return;
    split_plane_body(it->st.plane, static_cast<const uint2*>(it->st.digits), lb % it->gx, lb / it->gx);
}

template <int KS>
void launch_split(const DstArgs<double>& a, const void* tab, cudaStream_t st) {
    constexpr int smem = SW / 2 * KS * STEP * 4;
    allow_smem(dst_split_kernel<KS>, smem);
    const long long total = (long long)a.lines * a.planes;
    const unsigned blocks = unsigned((total + 8 * SW - 1) / (8 * SW));
    // up to a block per SM (4864 lines): a group of results per block, their lines' digits made by each
    // (255 lines: 17.5 us; the same in eight blocks 130 us)
    const dim3 grid(blocks, blocks <= 152 ? 2 * KS / TILES : 1);
    dst_split_kernel<KS><<<grid, 32 * SW, smem, st>>>(a, static_cast<const uint2*>(tab));
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

}  // namespace

// coarse FP64 levels: planes of 64 x 64 cells (one parity's digits of a whole plane in one block); the dense plane
// transforms serve smaller ones
bool split_planes(const Geom& g) { return g.nx - 1 == SP_CELLS && g.ny - 1 == SP_CELLS; }

// direct corrections, where both axes are of such lengths.  512 cells: 7 x 256 digit products of up to 2^14 pass 2^24, so
// FP32 sums of them would not be exact (and the digits of a parity, 58 KB for 16 lines, would leave one block per SM); 64:
// direct corrections keep the fast transforms (their error, 2.3e-15 to 3.5e-15 at 65 x 65 x 33, is the tridiagonal solves')
bool split_length(int N) { return N == 128 || N == 256; }

// sin(pi q / N) 2^55 as an integer
static long long sine55(long long q, int N) {
    return llrintl(sinl(3.14159265358979323846264338327950288L * (long double)q / (long double)N) * 36028797018963968.0L);
}

// digits of the folded sine matrices of N cells in fragment order (B of
// m16n8k16: lane (g, t) holds rows 2t, 2t + 1 and 2t + 8, 2t + 9 of column g)
void* make_split_table(int N, size_t* bytes) {
    const int Ko = N / 2, KS = Ko / 16;
    std::vector<uint2> tab(size_t(2) * (Ko / 8) * KS * DIG * 32);
    std::vector<long long> sines(2 * N);
    for (int q = 0; q <= N / 2; ++q) {   // one quarter of the period holds them all
        const long long v = sine55(q, N);
        sines[q] = sines[N - q] = v;
        sines[N + q] = -v;
        sines[(2 * N - q) % (2 * N)] = -v;
    }
    sines[0] = sines[N] = 0;
    auto digits = [&](int par, int i, int p) -> unsigned long long {   // of element i of result p, biased
        const int m = 2 * p + 1 + par;                                  // mode
        if (m > N - 1 || (par && i >= Ko - 1)) return BIAS;             // padding: zero
        return static_cast<unsigned long long>(sines[size_t(m) * (i + 1) % (2 * N)] + BIAS);
    };
    unsigned short half_of[257];   // a digit (biased by 128; the first may be 128) as FP16
    for (int q = 0; q <= 256; ++q) half_of[q] = __half_as_ushort(__float2half(float(q - 128)));
    for (int par = 0; par < 2; ++par)
        for (int nt = 0; nt < Ko / 8; ++nt)
            for (int ks = 0; ks < KS; ++ks)
                for (int l = 0; l < 32; ++l) {
                    const int g = l >> 2, t = l & 3;
                    unsigned long long d[4];
                    for (int r = 0; r < 4; ++r) d[r] = digits(par, ks * 16 + 2 * t + (r & 1) + 8 * (r >> 1), nt * 8 + g);
                    for (int s = 0; s < DIG; ++s) {
                        const int sh = 8 * (DIG - 1 - s);
                        auto digit = [&](int r) { return unsigned(half_of[s ? (d[r] >> sh) & 255 : d[r] >> sh]); };
                        auto pack = [&](int r) { return digit(r) | (digit(r + 1) << 16); };
                        tab[(((size_t(par) * (Ko / 8) + nt) * KS + ks) * DIG + s) * 32 + l] = make_uint2(pack(0), pack(2));
                    }
                }
    void* p = nullptr;
    MHS_CUDA(cudaMalloc(&p, tab.size() * sizeof(uint2)));
    MHS_CUDA(cudaMemcpy(p, tab.data(), tab.size() * sizeof(uint2), cudaMemcpyHostToDevice));
    *bytes = tab.size() * sizeof(uint2);
    return p;
}

void launch_dst_split(const DstArgs<double>& a, const void* tab, cudaStream_t st) {
    if (a.L == SP_CELLS) launch_split<2>(a, tab, st);
    else if (a.L == 128) launch_split<4>(a, tab, st);
    else launch_split<8>(a, tab, st);
}

SepStage<double> split_plane_stage(const PlaneArgs<double>& p, const void* digits, int planes) {
    SepStage<double> s;
    s.kind = SEP_SPLIT_PLANE;
    s.plane = p;
    s.digits = digits;
    s.threads = SP_T;
    s.grid = dim3(2, planes);
    return s;
}

void launch_split_plane(const SepStage<double>& s, cudaStream_t st) {
    split_plane_kernel<<<s.grid, s.threads, 0, st>>>(s.plane, static_cast<const uint2*>(s.digits));
}

void glaunch_split_plane(const GSepTable<double>& t, int fmg_step, int gate, cudaStream_t st) {
    g_split_plane_kernel<<<t.blocks, t.threads, 0, st>>>(t.items, t.n, fmg_step, gate);
}

}  // namespace mhs
