// launch_rules.h -- how launches split their work, as functions of sizes alone (plain host code, no
// CUDA).
#pragma once
#include <math.h>
#include <stdint.h>

#include <algorithm>

namespace dafmm {

constexpr int kSMs = 152;  // of a GB300

// Bounding boxes of a forest: blocks of 256 threads for each of the nroots problems, the largest of
// which has max_n particles.  The grid is the same for every problem, so that blocks for the largest
// one are empty blocks for all the others: about 0.5 ns each, against 2.2 ms for a problem of 1e6
// particles by one block.  2 sqrt(max_n / nroots) balances the two, up to 8 particles per thread
// and 4 blocks per SM.  One problem of 1e6 particles among 100,000 of 3, the whole build: 29.5 ms with
// as many blocks as the largest fills, 11.2 ms with one block each (and a slower build otherwise), 5.3
// ms with this rule; among 20,000: 8.1, 7.1 and 3.4 ms.
inline int bbox_blocks(int64_t nroots, int64_t max_n) {
    const int64_t fill = (max_n + 2047) / 2048;
    const int64_t room = (int64_t)(2.0 * sqrt((double)max_n / (double)std::max<int64_t>(nroots, 1)));
    return (int)std::max<int64_t>(1, std::min<int64_t>({fill, room, 4 * kSMs}));
}

// Near field of a uniform tree (FP32 and FP64): warps that share a leaf's sources.  Such a tree has 8^depth
// leaves: from 4096 on, one warp each gives an SM the 24 or 28 warps that it holds; 512 leaves and
// fewer do not fill the GPU, and take 8.  In FP32 the warps share segments of 128 sources, so that a tree of
// at most 128 particles has nothing to share: 8 warps only add their joining (2 particles, one
// leaf: 7.5 us with one warp, 10.2 with 8).
constexpr int kLeafWarps = 8;
inline int leaf_warps(int64_t nleaf, int64_t n, bool f64) {
    if (nleaf >= 16 * kSMs || (!f64 && n <= 128)) return 1;
    return kLeafWarps;
}

// M2L by rotation of a uniform level of nbox boxes: targets per warp.  Two from 512 boxes on (they share
// the table reads: N = 200,003, depth 4, p = 8: FP64 7.1 -> 6.8 ms, float-float 5.9 -> 4.6 ms; N = 1e4, p = 6: 0.81
// -> 0.78 ms), but in FP64 only while the level is about one wave: two targets need 96 registers, 16 warps
// per SM, and from 32768 boxes on the warps in flight count for more.  One target compiled for 32
// warps, finest level against two at 16: depth 5, p = 4, 6, 8, 10: 13.48, 21.49, 38.6, 68.6 -> 12.58, 20.27, 36.5, 65.3 ms;
// depth 6, p = 4, 6: 109.5, 174.5 -> 102.9, 166.1 ms (one target at 24 warps, packed tables: 12.43, 20.15, 37.2,
// 68.1; 103.5, 167.5).  Float-float (72 registers either way) keeps two.
inline int rot_targets(int64_t nbox, bool harm, bool f64) {
    return harm && nbox >= 512 && !(f64 && nbox >= 32768) ? 2 : 1;
}
// ... and warps that share the displacements of the same targets: up to 8 while there are fewer than 16
// warps per SM
inline int rot_share(int64_t nbox, int targets) {
    int k = 1;
    while (k < 8 && nbox / targets * k < 16 * kSMs) k *= 2;
    return k;
}

// FP32 near field of an adaptive tree: blocks that share the passes (32 targets each) of a leaf, one
// while the leaves alone fill the 24 warps that an SM holds, otherwise as many as the GPU has room
// for, up to the passes of the largest leaf and 8.  A lone warp on a large leaf is bound by the latency
// of its pairs: one leaf of 1000 particles 0.69 ms with one target per lane, 0.99 with two, 0.13 with
// two and 8 blocks; 500 particles 0.190, 0.260, 0.038; 200 problems of 1000 particles, one leaf each, p = 6:
// the evaluation 0.855, 1.054, 0.241.  A pass does not depend on the others: the results are the same.
inline int leaf_a_split(int64_t nleaves, int max_leaf) {
    const int64_t passes = ((int64_t)max_leaf + 31) / 32, room = 24 * kSMs / std::max<int64_t>(nleaves, 1);
    return (int)std::max<int64_t>(1, std::min<int64_t>({passes, room, 8}));
}

}  // namespace dafmm
