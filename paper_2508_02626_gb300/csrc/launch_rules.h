// launch_rules.h -- how launches split their work, as functions of sizes alone (plain host code, no
// CUDA).
#pragma once
#include <math.h>
#include <stdint.h>

#include <algorithm>

namespace dafmm {

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
    return (int)std::max<int64_t>(1, std::min<int64_t>({fill, room, 608}));
}

}  // namespace dafmm
