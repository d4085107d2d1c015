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

}  // namespace mhs
