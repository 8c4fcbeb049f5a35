// C entries to the launch rules, for tests/test_launch_rules.py
#include "launch_rules.h"

extern "C" int bbox_blocks(long long nroots, long long max_n) { return dafmm::bbox_blocks(nroots, max_n); }
extern "C" int leaf_a_split(long long nleaves, int max_leaf) { return dafmm::leaf_a_split(nleaves, max_leaf); }
extern "C" int leaf_warps(long long nleaf, long long n, int f64) { return dafmm::leaf_warps(nleaf, n, f64 != 0); }
extern "C" int rot_targets(long long nbox, int harm, int f64) { return dafmm::rot_targets(nbox, harm != 0, f64 != 0); }
extern "C" int rot_share(long long nbox, int targets) { return dafmm::rot_share(nbox, targets); }
