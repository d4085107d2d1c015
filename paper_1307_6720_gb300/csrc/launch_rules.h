// Rules of launch shapes and of the choice between forms of an operation that
// depend on sizes alone: plain host functions without CUDA types, so that
// tests can go through them for any size without a GPU.
#pragma once

#include <algorithm>

namespace mhs {

constexpr int RULE_SMS = 152;

// Results of either parity per block of the plane transforms (plane_body) of
// lines with ko odd results, before the limit of shared memory: as many as
// leave a block per SM, not below `least`, and never so many that half of them
// would do, as a block forms all it has room for, wanted or not (17 x 17 x 257
// nodes with sixteen for eight results: 20 us a pass in FP64, with eight 13 us;
// 9 x 9 x 513 41 and 19 us for both).  Grouped launches have blocks enough of
// other instances: eight (1024 FP32 solves of 33^3 42.7 -> 40.0 ms, 256 in FP64
// 16.4 -> 13.3 ms; with sixteen, 64 FP64 solves of 65 x 65 x 33 7.75 instead
// of 7.63 ms).
inline int plane_results(int ko, int planes, int least, bool grouped) {
    int sp = grouped ? 8 : 16;
    while (sp / 2 >= ko && sp > least) sp /= 2;
    while (!grouped && sp > least && (long long)((ko + sp - 1) / sp) * planes < RULE_SMS) sp /= 2;
    return sp;
}

// Whether a level of cx x cy cells (powers of two, at most 128) and `planes`
// planes takes the dense plane transforms or the fast ones, by device time of
// its transforms (us, fast / dense; two launches on 3D levels).
//
// A dense plane is O(n) per node but one launch of few steps; the fast ones are
// a chain of short steps that a wave of planes shares.  So dense loses
// - in FP64, whose pipe it fills, with 32 cells from about a wave of planes:
//   33 x 33 nodes 63 planes 29.7 / 25.8, 127 planes 38.6 / 41.7, 511 planes
//   108 / 136; 33 x 17 nodes 127 planes 28.9 / 27.3, 255 planes 35.4 / 43.6;
//   33 x 9 nodes 127 planes 26.4 / 21.6, 191 planes 27.3 / 32.4.  17 x 17 nodes
//   stay ahead (127 planes 26.2 / 17.5, 2047 planes 167 / 128), 65 x 33 lose at
//   any count (one plane: 25.7 / 13.7);
// - in FP32 where the short side is far below a warp's 32 lanes, which the long
//   side's matrix then feeds badly: 129 x 9 nodes 31 planes 14.5 / 14.3, 39 planes
//   15.0 / 16.1; 129 x 17 nodes 127 planes 25.4 / 24.3, 191 planes 29.4 / 32.7;
//   65 x 9 nodes 191 planes 15.9 / 14.6, 255 planes 15.9 / 16.2; 65 x 17 nodes
//   511 planes 28.4 / 27.4, 1023 planes 44.4 / 46.4;
// - with 128 x 128 cells in FP32 by the count of waves, of four blocks a plane,
//   20 us each and pass, against two, 37 us each: 31 planes (one wave) 47.5 / 35.9,
//   63 planes 77.9 / 84.1, 95 planes 151 / 124, 127 planes 152 / 163, 191 planes
//   226 / 240, 255 planes 300 / 285;
// - on single FP32 planes of 128 cells, in one cluster either way: 129 x 33 nodes
//   11.8 / 13.3, 129 x 129 17.4 / 17.9; 65 x 65 12.2 / 10.8.
inline bool dense_planes_faster(bool fp64, int dim, int cx, int cy, int planes) {
    const int big = std::max(cx, cy), small = std::min(cx, cy);
    if (dim == 2) return big <= 64;
    if (fp64)
        return big <= 16 || (big == 32 && planes <= RULE_SMS && (long long)(cx - 1) * (cy - 1) * planes <= 100000);
    if (big <= 32) return true;
    if (small == 128) {
        const int dense = (4 * planes + RULE_SMS - 1) / RULE_SMS, fast = (2 * planes + RULE_SMS - 1) / RULE_SMS;
        return dense == 1 || dense * 20 <= fast * 37;
    }
    if (small > 16) return true;
    if (big == 64) return planes <= (small == 16 ? 512 : 192);
    return planes <= (small == 16 ? RULE_SMS : 32);
}

// Chunks of the nzi inner planes of the double-float march (df_march_body) over
// `tiles` tiles: the count with the least waves of resident blocks (two per
// SM) times planes, three of them start-up; at most max_blocks blocks (0: any)
// unless the tiles alone are more.  Chunks of four planes or more, and two of
// levels of five to seven planes (a direct mixed solve of 129 x 129 x 9: 205 us in
// one chunk, 196 in two; as two launches per step 198).  Shorter chunks fill the
// chip better on shallow levels by themselves (190 us with single planes) but groups
// keep the decomposition, which orders the sums, and have blocks enough: 32 of
// them 3.70 ms, in two chunks 3.75, in single planes 4.08; 16 of 129 x 33 x 33
// 1.89 and, in single planes, 2.10 ms.
inline int df_march_chunks(long long tiles, int nzi, int max_blocks) {
    const long long resident = 2 * RULE_SMS;
    long long best = 0;
    int chunks = 1;
    for (int n = 1; n <= std::max(nzi > 4 ? 2 : 1, nzi / 4); ++n) {
        const int per = (nzi + n - 1) / n, m = (nzi + per - 1) / per;
        if (n > 1 && max_blocks > 0 && tiles * m > max_blocks) break;
        const long long cost = (tiles * m + resident - 1) / resident * (per + 3);
        if (n == 1 || cost < best) {
            best = cost;
            chunks = m;
        }
    }
    return chunks;
}

// Tiles of the pairs of sweeps (kernels_pair.cu): 32 quads of nodes, of which 30
// inside a row are stored, by 32 rows, of which all but four at either end are.
constexpr int PAIR_QUADS = 32, PAIR_ROWS = 32, PAIR_CHUNK = 256;   // (most planes of a chunk)
struct PairShapeOf {
    int gx, gy, chunk;   // tiles, planes of a chunk (even)
    long long steps;     // of the march: waves of one block per SM, times planes and start-up
};
// Chunks of an even count of planes; a chunk runs eight planes more than it
// stores and starts up for about two: the count of chunks with the least steps.
inline PairShapeOf pair_shape(int nx, int ny, int nz) {
    PairShapeOf s{};
    const int quads = (nx - 2) / 4 + 1;
    s.gx = quads <= PAIR_QUADS ? 1 : (quads - PAIR_QUADS + PAIR_QUADS - 3) / (PAIR_QUADS - 2) + 1;
    s.gy = ny <= PAIR_ROWS ? 1 : (ny - PAIR_ROWS + PAIR_ROWS - 9) / (PAIR_ROWS - 8) + 1;
    const long long tiles = (long long)s.gx * s.gy;
    for (int c = std::max(1, (nz + PAIR_CHUNK - 1) / PAIR_CHUNK); c <= std::max(1, nz / 4) + 1; ++c) {
        const int kc = std::min(PAIR_CHUNK, ((nz + c - 1) / c + 1) / 2 * 2), n = (nz + kc - 1) / kc;
        const long long steps = (tiles * n + RULE_SMS - 1) / RULE_SMS * (kc + 10);
        if (!s.chunk || steps < s.steps) {
            s.steps = steps;
            s.chunk = kc;
        }
    }
    return s;
}

// Levels whose pairs of sweeps run as one pass: those where its march takes less
// time than four colour passes, or up to 2.5 us more.  nx = 4m + 1: see PairTile.  A
// step takes 1.04 us; the colour passes, up to four million nodes, 7.45 us more than
// the march's start and 5.57 us per million nodes, rows counted in whole warps of 64
// nodes (fitted to whole mixed solves of 82 boxes of 0.9 to 4 million nodes: within
// 2.5 us but on three of the longest).  Four passes against one, us more (+) or less
// (-) for the one: 129^3 -1.4, 113^3 -2.1, 97 x 97 x 193 -4.1, 193 x 193 x 97 -5.1; 129 x
// 129 x 65 +1.4, 65 x 65 x 513 +4.1, 33 x 33 x 1025 +6.9, 17 x 33 x 2049 +9.6 (17 of 128
// columns of its tiles used), 33 x 33 x 4097 +22.  The passes are ahead while u and f stay
// in cache, of which the one pass needs a quarter of the traffic: from four million
// nodes, where they run in their vector form, it wins on every box (257 x 129 x 129 -8.2,
// 33 x 129 x 1025 -36), and beside other solves it wins earlier (an uneven group with 129
// x 129 x 65 members 11.16 ms, with passes for these 11.43; eight solves of 257 x 257 x 33
// 4.72 and 5.43 ms), hence the 2.5 us.  Levels of less than 800,000 nodes keep the
// passes (65^3 mixed solves 1.04 ms with them, 1.15 ms with pairs).
inline bool pair_pays(int nx, int ny, int nz) {
    const long long rows = (long long)(ny - 2) * (nz - 2), nodes = rows * (nx - 2);
    if ((nx & 3) != 1 || nodes < 800000) return false;
    const double padded = double((nx - 2 + 63) / 64 * 64) * double(rows);
    return nodes >= 4000000 || 1.04 * double(pair_shape(nx, ny, nz).steps) < 7.45 + 5.57e-6 * padded + 2.5;
}

}  // namespace mhs
