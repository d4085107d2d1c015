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
// unless the tiles alone are more.  Down to single planes, or a shallow level
// is marched by its few tiles (129 x 129 x 9 in one chunk of seven planes: 16
// blocks; a direct mixed solve 205 us, with single planes 190 us).
inline int df_march_chunks(long long tiles, int nzi, int max_blocks) {
    const long long resident = 2 * RULE_SMS;
    long long best = 0;
    int chunks = 1;
    for (int n = 1; n <= nzi; ++n) {
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

}  // namespace mhs
