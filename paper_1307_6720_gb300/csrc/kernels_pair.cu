// Two red-black sweeps of an FP32 level in one pass (out of place).
//
// V(2,2)-cycles smooth in pairs of sweeps.  Colour by colour a pair moves u
// four times and f four times through the memory system; here a block marches
// up the planes once, every plane loaded once and stored once, with four
// updates in flight: at step m, plane m arrives, then red 1 of plane m-1,
// black 1 of plane m-2, red 2 of plane m-3 and black 2 of plane m-4, which
// is stored.  Each update needs the opposite colour of its own plane as the
// previous step left it and the two planes beside it as this step's earlier
// updates left them, so one block barrier per step orders everything.
//
// A thread owns a quad of four consecutive x nodes in two adjacent rows and
// keeps the planes of its column in registers: z neighbours, the row beside
// and the x neighbours inside the quad cost nothing; the x neighbour past the
// quad is a warp shuffle, the y neighbour past the two rows comes from the
// neighbouring warp through shared memory (two values per row and update,
// double-buffered).  Registers are indexed by plane modulo six, the march
// unrolled six times, so no plane is ever moved.  Planes of u and f arrive by
// TMA (132 x 2 NW boxes, one thread, two steps ahead, three-slot rings).
//
// Four updates spread an unknown value by four nodes: a tile of 32 quads x
// 2 NW rows stores its quads 1 .. 30 and all rows but four at either end
// (nothing is lost at the faces of the box, whose values are fixed), and a
// chunk of planes starts and ends four planes outside.  Faces are copied, so
// the output array is complete.  Every update forms the colour passes'
// operations in their order: the result equals four colour passes bit for
// bit.
//
// Measured: 513 x 513 x 257 243 us per pair (twice 307 us as fused single
// sweeps), 257^3 85 us (twice 65), 129^3 17 us; its traffic at 513 x 513 x 257
// takes 119 us.  In scalar FP32 instructions 256, 95 and 19 us (240 per thread
// and step of eight nodes).  47 % of the issue slots at 129^3; the stalls are
// shared memory, dependent instructions and the barrier in equal parts; a
// quarter of the rows and a fifth of the quads (513 nodes: 5 tiles) are halo.
//
// TMA rules as in kernels_tma.cu: boxes start at x a multiple of four floats,
// slots are 128-byte aligned, every mbarrier wait is bounded.
#include <cuda.h>

#include "device_util.cuh"
#include "launch_rules.h"
#include "mhs_internal.h"
#include "tma_util.cuh"

namespace mhs {

namespace {

constexpr int QUADS = PAIR_QUADS;  // quads of a tile (lanes)
constexpr int PBW = 4 * QUADS + 4; // floats per box row: the tile and the quad east of it
constexpr int NS = 3;              // ring slots (half the unrolled steps, so slots and phases are constants)
constexpr int MAX_CHUNK = PAIR_CHUNK;

template <int NW>
struct PairShape {
    static constexpr int H = 2 * NW;               // tile rows
    static constexpr int SLOT = H * PBW;           // floats of a staged plane
    static constexpr int PUB = H * 32;             // published pairs of one update
    static constexpr unsigned BOX_BYTES = SLOT * 4;
    static constexpr size_t PUB_OFF = size_t(2 * NS) * SLOT * 4;             // published values [2][4][H][32] float2
    static constexpr size_t EAST_OFF = PUB_OFF + size_t(2) * 4 * PUB * 8;    // east face values [6][H]
    static constexpr size_t COEF_OFF = EAST_OFF + (size_t(6) * H * 4 + 15) / 16 * 16;   // per-plane factors
    static constexpr size_t BAR_OFF = COEF_OFF + size_t(MAX_CHUNK + 16) * 16;
    static constexpr size_t BYTES = BAR_OFF + NS * 8 + 128;
    static_assert(SLOT * 4 % 128 == 0, "TMA slots must stay 128-byte aligned");
};

// What a thread knows of its place.  nx = 4m + 1, so of a quad's nodes only
// the first can lie on a face (x = 0 or nx-1); nodes past x = nx-1 are never
// read by others and may hold anything.
struct PairTile {
    int lo, hi;             // published entries of the rows below and above the thread's two
    int own;                // published entry of its first row
    bool rk[2];             // the row is interior (the same for a warp)
    bool k0;                // the quad's first node is off the x faces
    bool east;              // the tile's last quad ends next to the x = nx-1 face (the same for a block)
    bool last;              // this thread owns that quad
};

// Planes in registers: [slot][row][p] holds the quad's nodes p and p + 2, the
// pair that one colour updates, so that every operation of an update is one
// packed FP32 instruction and a published pair is a register pair.
typedef float2 PairRegs[6][2][2];

// The values outside the thread that an update of colour COL of the plane in
// register slot S reads: per row the pair the neighbouring row published and
// the x neighbour outside the quad (west of node 0 or east of node 3).  All
// were final when the step began, so they are fetched ahead of the updates.
struct PairOuter {
    float2 y[2];
    float x[2];
};
template <int NW, int S, int COL>
__device__ __forceinline__ void pair_gather(PairOuter& o, const PairRegs& U, const PairTile& t, const float2* pub,
                                            const float* east) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        o.y[r] = pub[r == 0 ? t.lo : t.hi];
        if (((r + S + COL) & 1) == 0) {
            o.x[r] = __shfl_up_sync(0xffffffffu, U[S][r][1].y, 1);
        } else {
            o.x[r] = __shfl_down_sync(0xffffffffu, U[S][r][0].x, 1);
            if (t.east && t.last) o.x[r] = east[S * 2 * NW + r];
        }
    }
}

// colour COL (0 red, 1 black) of the plane in register slot S; the new values
// are published to `out` unless this is the plane's last update.
// c = (1/d, -az, -ay, -ax); F holds f/d.
template <int S, int COL, bool LAST>
__device__ __forceinline__ void pair_update(PairRegs& U, const PairRegs& F, const PairTile& t, const float4 c,
                                            const PairOuter& o, float2* out) {
    constexpr int UP = (S + 1) % 6, DN = (S + 5) % 6;
    const float2 cz = make_float2(c.y, c.y), cy = make_float2(c.z, c.z), cx = make_float2(c.w, c.w);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int s = (r + S + COL) & 1;   // the colour's nodes: s and s + 2
        if (t.rk[r]) {
            // x neighbours: (west, node 1) and (1, 3) of nodes (0, 2); (0, 2) and (node 2, east) of (1, 3)
            const float2 ew = s == 0 ? __fadd2_rn(U[S][r][1], make_float2(o.x[r], U[S][r][1].x))
                                     : __fadd2_rn(make_float2(U[S][r][0].y, o.x[r]), U[S][r][0]);
            float2 v = __ffma2_rn(cz, __fadd2_rn(U[UP][r][s], U[DN][r][s]), F[S][r][s]);
            v = __ffma2_rn(cy, __fadd2_rn(o.y[r], U[S][1 - r][s]), v);
            v = __ffma2_rn(cx, ew, v);
            if (s == 0) v.x = t.k0 ? v.x : U[S][r][0].x;
            U[S][r][s] = v;
        }
        // a face row publishes its fixed values
        if (!LAST) out[t.own + r * 32] = U[S][r][s];
    }
}

template <int NW>
__global__ void __launch_bounds__(32 * NW, 1)
    rb_pair_kernel(const __grid_constant__ CUtensorMap tm_u, const __grid_constant__ CUtensorMap tm_f, Geom g,
                   const PlaneCoef<float>* __restrict__ coef, float* __restrict__ uout, int kchunk,
                   int* __restrict__ err) {
    using S_ = PairShape<NW>;
    constexpr int H = S_::H;
    extern __shared__ unsigned char pair_smem[];
    unsigned char* base = pair_smem + ((128u - (smem_addr(pair_smem) & 127u)) & 127u);
    float* s_u = reinterpret_cast<float*>(base);
    float* s_f = s_u + NS * S_::SLOT;
    float2* s_pub = reinterpret_cast<float2*>(base + S_::PUB_OFF);
    float* s_east = reinterpret_cast<float*>(base + S_::EAST_OFF);
    float4* s_c = reinterpret_cast<float4*>(base + S_::COEF_OFF);
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(base + S_::BAR_OFF);

    const int tid = threadIdx.x, lane = tid & 31, row = 2 * (tid >> 5);
    const int q0 = blockIdx.x * (QUADS - 2), y0 = blockIdx.y * (H - 8);
    const int ka = blockIdx.z * kchunk, kb = min(g.nz - 1, ka + kchunk - 1);   // planes stored
    // kchunk is even, so p0 is, and a plane's parity is that of its register slot
    const int p0 = max(0, ka - 4), mend = kb + 4, plast = min(mend, g.nz - 1);
    const int plo = max(1, p0), phi = g.nz - 2;   // planes updated
    const int x = 4 * (q0 + lane), j0 = y0 + row;
    // what the tile stores: its valid quads and rows, faces included
    const int nqi = (g.nx - 2) / 4 + 1;   // quads that hold interior nodes
    const bool xlast = q0 + QUADS >= nqi, ylast = y0 + H >= g.ny;
    const bool xok = (lane >= 1 || q0 == 0) && (lane <= 30 || xlast) && x < g.px;
    bool yok[2];
    PairTile t;
    t.own = row * 32 + lane;
    t.lo = max(row - 1, 0) * 32 + lane;
    t.hi = min(row + 2, H - 1) * 32 + lane;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        t.rk[r] = j0 + r >= 1 && j0 + r <= g.ny - 2;
        yok[r] = xok && (row + r >= 4 || y0 == 0) && (row + r < H - 4 || ylast) && j0 + r <= g.ny - 1;
    }
    t.k0 = x != 0 && x != g.nx - 1;
    t.east = xlast && 4 * (q0 + QUADS) == g.nx - 1;
    t.last = lane == 31;

    for (int k = tid; k <= plast - p0; k += 32 * NW) {
        const PlaneCoef<float> c = coef[p0 + k];
        s_c[k] = make_float4(c.inv_d, -c.az, -c.ay, -c.ax);
    }
    // stage p: plane p of u and plane p - 1 of f (where they exist), slots by
    // plane modulo NS, completing on mbarrier p % NS; thread 0 issues and waits
    auto issue = [&](int p) {
        if (p > mend) return;
        const int q = (p - p0) % NS;
        const bool lu = p <= plast, lf = p - 1 >= plo && p - 1 <= phi;
        mbar_arrive_expect_tx(&bar[q], (lu ? S_::BOX_BYTES : 0) + (lf ? S_::BOX_BYTES : 0));
        if (lu) tma_load_plane(s_u + q * S_::SLOT, &tm_u, 4 * q0, y0, p, &bar[q]);
        if (lf) tma_load_plane(s_f + (q == 0 ? NS - 1 : q - 1) * S_::SLOT, &tm_f, 4 * q0, y0, p - 1, &bar[q]);
    };
    bool failed = false;   // (thread 0) a wait ran out: no more loads; the march ends on whatever arrived
    auto wait = [&](int p, int q, int phase) {
        if (failed || p > mend || mbar_wait(&bar[q], phase)) return;
        failed = true;
        atomicExch(err, 1);
        // the one later stage in flight
        const int n = q == NS - 1 ? 0 : q + 1;
        if (p + 1 <= mend) (void)mbar_wait(&bar[n], n == 0 ? phase ^ 1 : phase);
    };
    if (tid == 0) {
        for (int q = 0; q < NS; ++q) mbar_init(&bar[q], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        issue(p0);
        issue(p0 + 1);
        wait(p0, 0, 0);
    }
    __syncthreads();

    PairRegs U = {}, F = {};
    float* out = uout + (size_t(x) + size_t(g.px) * size_t(j0) + g.plane * size_t(ka));   // plane ka of the quad
    const float* su = s_u + row * PBW + 4 * lane;
    const float* sf = s_f + row * PBW + 4 * lane;
    float* se = s_east + row;
    const float4* cp = s_c;   // factors of the plane of step 0
    bool done = false;

// one step of the march at plane m, register slot S = (m - p0) % 6
#define MHS_PAIR_STEP(S)                                                                                              \
    {                                                                                                                 \
        const int m = mm + S;                                                                                         \
        const float2* pin = s_pub + ((S + 1) & 1) * 4 * S_::PUB; /* published by the previous step */                 \
        float2* pout = s_pub + (S & 1) * 4 * S_::PUB;                                                                 \
        /* stage m + 2 refills the slots of u plane m - 1 and f plane m - 2, read in the last step */                 \
        if (tid == 0 && !failed) issue(m + 2);                                                                        \
        PairOuter o0, o1, o2, o3;                                                                                     \
        pair_gather<NW, (S + 5) % 6, 0>(o0, U, t, pin, se);                                                           \
        pair_gather<NW, (S + 4) % 6, 1>(o1, U, t, pin + S_::PUB, se);                                                 \
        if (m <= plast) {                                                                                             \
            const float* a = su + (S % NS) * S_::SLOT;                                                                \
            _Pragma("unroll") for (int r = 0; r < 2; ++r) {                                                           \
                const float4 v = *reinterpret_cast<const float4*>(a + r * PBW);                                       \
                U[S][r][0] = make_float2(v.x, v.z), U[S][r][1] = make_float2(v.y, v.w);                                 \
                const int b = (r + S + 1) & 1; /* the row's black pair */                                          \
                pout[t.own + r * 32] = U[S][r][b];                                                                    \
                if (t.east && t.last) se[S * H + r] = a[r * PBW + 4];                                                 \
            }                                                                                                         \
        }                                                                                                             \
        if (m - 1 >= plo && m - 1 <= phi) {                                                                           \
            constexpr int Z = (S + 5) % 6;                                                                            \
            const float* a = sf + (Z % NS) * S_::SLOT;                                                                \
            const float4 c = cp[S - 1];                                                                               \
            _Pragma("unroll") for (int r = 0; r < 2; ++r) {                                                           \
                const float4 v = *reinterpret_cast<const float4*>(a + r * PBW);                                       \
                F[Z][r][0] = __fmul2_rn(make_float2(v.x, v.z), make_float2(c.x, c.x));                                \
                F[Z][r][1] = __fmul2_rn(make_float2(v.y, v.w), make_float2(c.x, c.x));                                \
            }                                                                                                         \
            pair_update<Z, 0, false>(U, F, t, c, o0, pout + S_::PUB);                                             \
        }                                                                                                             \
        pair_gather<NW, (S + 3) % 6, 0>(o2, U, t, pin + 2 * S_::PUB, se);                                             \
        if (m - 2 >= plo && m - 2 <= phi)                                                                             \
            pair_update<(S + 4) % 6, 1, false>(U, F, t, cp[S - 2], o1, pout + 2 * S_::PUB);                       \
        pair_gather<NW, (S + 2) % 6, 1>(o3, U, t, pin + 3 * S_::PUB, se);                                             \
        if (m - 3 >= plo && m - 3 <= phi)                                                                             \
            pair_update<(S + 3) % 6, 0, false>(U, F, t, cp[S - 3], o2, pout + 3 * S_::PUB);                       \
        if (m - 4 >= plo && m - 4 <= phi)                                                                             \
            pair_update<(S + 2) % 6, 1, true>(U, F, t, cp[S - 4], o3, nullptr);                                   \
        if (m - 4 >= ka) {                                                                                            \
            constexpr int Z = (S + 2) % 6;                                                                            \
            _Pragma("unroll") for (int r = 0; r < 2; ++r) {                                                           \
                if (yok[r]) {                                                                                         \
                    float* o = out + size_t(r) * g.px;                                                                \
                    *reinterpret_cast<float4*>(o) =                                                                   \
                        make_float4(U[Z][r][0].x, U[Z][r][1].x, U[Z][r][0].y, U[Z][r][1].y);                          \
                    if (t.east && t.last) o[4] = se[Z * H + r];                                                       \
                }                                                                                                     \
            }                                                                                                         \
            out += g.plane;                                                                                           \
        }                                                                                                             \
        if (m >= mend) {                                                                                              \
            done = true;                                                                                              \
            break;                                                                                                    \
        }                                                                                                             \
        if (tid == 0) wait(m + 1, (S + 1) % NS, ((S + 1) / NS) & 1);                                                  \
        __syncthreads();                                                                                              \
    }

    for (int mm = p0; !done; mm += 6, cp += 6) {
        do {
            MHS_PAIR_STEP(0)
            MHS_PAIR_STEP(1)
            MHS_PAIR_STEP(2)
            MHS_PAIR_STEP(3)
            MHS_PAIR_STEP(4)
            MHS_PAIR_STEP(5)
        } while (false);
    }
#undef MHS_PAIR_STEP
}

template <int NW>
void launch_pair(const Geom& g, const CUtensorMap& tm_u, const CUtensorMap& tm_f, const PlaneCoef<float>* coef,
                 float* uout, int* err, cudaStream_t st) {
    using S = PairShape<NW>;
    allow_smem(rb_pair_kernel<NW>, S::BYTES);
    static_assert(S::H == PAIR_ROWS, "the rows that the rule counts with");
    const PairShapeOf p = pair_shape(g.nx, g.ny, g.nz);
    const int kchunk = p.chunk;
    const dim3 grid(p.gx, p.gy, (g.nz + kchunk - 1) / kchunk);
    rb_pair_kernel<NW><<<grid, 32 * NW, S::BYTES, st>>>(tm_u, tm_f, g, coef, uout, kchunk, err);
    count_launches(1);
    MHS_CUDA(cudaGetLastError());
}

constexpr int PAIR_WARPS = 16;

}  // namespace

void make_pair_map(CUtensorMap* map, const Geom& g, const float* base) {
    make_box_map(map, g, base, PBW, PairShape<PAIR_WARPS>::H);
}

bool pair_level(const Geom& g) { return pair_pays(g.nx, g.ny, g.nz); }

void launch_pair_sweep(const Geom& g, const CUtensorMap& tm_u, const CUtensorMap& tm_f,
                       const PlaneCoef<float>* coef, float* uout, int* err, cudaStream_t st) {
    launch_pair<PAIR_WARPS>(g, tm_u, tm_f, coef, uout, err, st);
}

}  // namespace mhs
