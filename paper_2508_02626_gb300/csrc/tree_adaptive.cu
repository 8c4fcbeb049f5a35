// tree_adaptive.cu -- adaptive octree on the GPU (Sec. 3.5: a box with more than s particles
// is subdivided) and its interaction lists (Cheng, Greengard and Rokhlin 1999):
//   colleagues : same-level adjacent boxes, kept in a 27-slot table indexed by relative
//                position (slot 13 = the box itself), -1 where no box exists;
//   V (M2L)    : children of the parent's colleagues that are not adjacent -- looked up on
//                the fly from the colleague table by the evaluation kernels;
//   U (P2P)    : for a leaf, every leaf adjacent to it, and itself;
//   W (M2P)    : for a leaf b, descendants of its colleagues that are not adjacent to b but
//                whose parent is;
//   X (P2L)    : for a box b, the leaves c coarser than b that are adjacent to parent(b) and
//                not adjacent to b (exactly the boxes whose W list holds b).
// Particles are sorted by 63-bit Morton keys of their 21-bit integer coordinates, so every
// box is a contiguous particle range.  A forest holds several independent trees (one root
// box each, level 0): the particles are grouped by tree and sorted inside each tree, and no
// list ever crosses trees, since every relation is derived from the parent's colleagues.
#include <cuda_runtime.h>

#include "check.cuh"
#include "internal.h"
#include "launch_rules.h"
#include "tree_adaptive.h"
#include "tree_common.cuh"

namespace dafmm {

__device__ inline int quantize_a(double x, double x0, double scale) {
    double f = floor(__dmul_rn(__dsub_rn(x, x0), scale));
    const double top = (double)((1 << kQBits) - 1);
    if (!(f >= 0.0)) return 0;
    if (f > top) return (1 << kQBits) - 1;
    return (int)f;
}

__device__ inline uint64_t spread3(uint32_t v) {
    uint64_t x = v & 0x1fffffu;
    x = (x | x << 32) & 0x1f00000000ffffull;
    x = (x | x << 16) & 0x1f0000ff0000ffull;
    x = (x | x << 8) & 0x100f00f00f00f00full;
    x = (x | x << 4) & 0x10c30c30c30c30c3ull;
    x = (x | x << 2) & 0x1249249249249249ull;
    return x;
}

// tree of particle i: the last r with offs[r] <= i
__device__ inline int tree_of(const int* offs, int nroots, int i) {
    int lo = 0, hi = nroots - 1;
    while (lo < hi) {
        const int m = (lo + hi + 1) >> 1;
        if (offs[m] <= i) lo = m;
        else hi = m - 1;
    }
    return lo;
}

__global__ void k_morton_keys(const double* __restrict__ xyz, int64_t n, const int* __restrict__ offs, int nroots,
                              const double* __restrict__ rootdom, uint64_t* keys, int* vals) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int r = nroots > 1 ? tree_of(offs, nroots, (int)i) : 0;
    const double* d = rootdom + 4 * r;
    const double scale = ldexp(1.0, kQBits) / d[3];
    const uint32_t a = quantize_a(xyz[3 * i], d[0], scale);
    const uint32_t b = quantize_a(xyz[3 * i + 1], d[1], scale);
    const uint32_t c = quantize_a(xyz[3 * i + 2], d[2], scale);
    keys[i] = spread3(a) | (spread3(b) << 1) | (spread3(c) << 2);
    vals[i] = (int)i;
}

cudaError_t launch_morton_keys(const double* xyz, int64_t n, const int* offs, int nroots, const double* rootdom,
                               uint64_t* keys, int* vals, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_morton_keys<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(xyz, n, offs, nroots, rootdom, keys, vals);
    return cudaGetLastError();
}

__global__ void k_tree_keys(const int* __restrict__ perm, int64_t n, const int* __restrict__ offs, int nroots,
                            uint64_t* tkeys, int* pos) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= n) return;
    tkeys[t] = (uint64_t)tree_of(offs, nroots, perm[t]);
    pos[t] = (int)t;
}

cudaError_t launch_tree_keys(const int* perm, int64_t n, const int* offs, int nroots, uint64_t* tkeys, int* pos,
                             cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_tree_keys<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(perm, n, offs, nroots, tkeys, pos);
    return cudaGetLastError();
}

__global__ void k_apply_order(const int* __restrict__ pos, int64_t n, const int* __restrict__ perm_in,
                              const uint64_t* __restrict__ keys_in, int* perm_out, uint64_t* keys_out) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int j = pos[t];
    perm_out[t] = perm_in[j];
    keys_out[t] = keys_in[j];
}

cudaError_t launch_apply_order(const int* pos, int64_t n, const int* perm_in, const uint64_t* keys_in, int* perm_out,
                               uint64_t* keys_out, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_apply_order<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pos, n, perm_in, keys_in, perm_out, keys_out);
    return cudaGetLastError();
}

// order-preserving map of a double to an unsigned integer (for atomic min/max)
__device__ inline unsigned long long ordered_bits(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

__global__ void __launch_bounds__(256) k_bbox_roots(const double* __restrict__ xyz, const int* __restrict__ offs,
                                                    unsigned long long* bb) {
    // blocks (r, 0 ..) of problem r stride over its particles: one block per problem took 2.2 ms on
    // a problem of 1e6 particles beside small ones, many blocks 20 us
    const int r = blockIdx.x;
    const int b = offs[r], e = offs[r + 1];
    if (b + (int64_t)blockIdx.y * blockDim.x >= e) return;
    unsigned long long mn[3] = {~0ull, ~0ull, ~0ull}, mx[3] = {0ull, 0ull, 0ull};
    for (int64_t i = b + (int64_t)blockIdx.y * blockDim.x + threadIdx.x; i < e; i += gridDim.y * blockDim.x)
        for (int d = 0; d < 3; ++d) {
            const unsigned long long u = ordered_bits(xyz[3 * i + d]);
            mn[d] = u < mn[d] ? u : mn[d];
            mx[d] = u > mx[d] ? u : mx[d];
        }
    for (int d = 0; d < 3; ++d) {
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long a = __shfl_xor_sync(0xffffffffu, mn[d], o);
            const unsigned long long c = __shfl_xor_sync(0xffffffffu, mx[d], o);
            mn[d] = a < mn[d] ? a : mn[d];
            mx[d] = c > mx[d] ? c : mx[d];
        }
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&bb[6 * r + d], mn[d]);
            atomicMax(&bb[6 * r + 3 + d], mx[d]);
        }
    }
}

__global__ void k_bbox_init(unsigned long long* bb, int nroots) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < 6 * nroots) bb[i] = (i % 6) < 3 ? ~0ull : 0ull;
}

cudaError_t launch_bbox_roots(const double* xyz, const int* offs, int nroots, int max_n, unsigned long long* bb,
                              cudaStream_t s) {
    if (nroots == 0) return cudaSuccess;
    k_bbox_init<<<(6 * nroots + 255) / 256, 256, 0, s>>>(bb, nroots);
    k_bbox_roots<<<dim3(nroots, bbox_blocks(nroots, max_n)), 256, 0, s>>>(xyz, offs, bb);
    return cudaGetLastError();
}

__global__ void k_box_geometry(const int* __restrict__ root, const int* __restrict__ level,
                               const int* __restrict__ ijk, const double* __restrict__ rootdom, int nbox,
                               double4* geom) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbox) return;
    const double* d = rootdom + 4 * root[b];
    const double h = ldexp(d[3], -level[b]);
    geom[b] = make_double4(d[0] + ((double)ijk[3 * (size_t)b] + 0.5) * h, d[1] + ((double)ijk[3 * (size_t)b + 1] + 0.5) * h,
                           d[2] + ((double)ijk[3 * (size_t)b + 2] + 0.5) * h, h);
}

cudaError_t launch_box_geometry(const int* root, const int* level, const int* ijk, const double* rootdom, int nbox,
                                double4* geom, cudaStream_t s) {
    if (nbox == 0) return cudaSuccess;
    k_box_geometry<<<(nbox + 255) / 256, 256, 0, s>>>(root, level, ijk, rootdom, nbox, geom);
    return cudaGetLastError();
}

// first sorted position in [b, e) whose level-(l+1) digit is >= c
__device__ inline int first_digit_ge(const uint64_t* keys, int b, int e, int shift, int c) {
    while (b < e) {
        const int m = (b + e) >> 1;
        if ((int)((keys[m] >> shift) & 7u) < c) b = m + 1;
        else e = m;
    }
    return b;
}

// Children of the boxes of level l: eight lanes per box, lane c searching the end of child c's
// particles (one thread per box ran the eight searches, some 20 dependent loads each, one after
// another).  [s, e): child c's particles, empty when the box does not split.
__device__ inline void child_range(const AdaptiveBuild& ab, int b, int level, bool split, int c, int& s, int& e) {
    const int pb = ab.pbeg[b], pe = ab.pend[b];
    e = split ? first_digit_ge(ab.keys, pb, pe, 3 * (kQBits - level - 1), c + 1) : pb;
    s = __shfl_up_sync(0xffffffffu, e, 1, 8);
    if (c == 0) s = pb;
}

// per box of level l: number of non-empty children when it splits
__global__ void k_split_count(AdaptiveBuild ab, int lb, int le, int level, int max_leaf, int max_depth, int* nch) {
    const int c = threadIdx.x & 7, own = lb + (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 3);
    const int b = min(own, le - 1);
    int s, e;
    child_range(ab, b, level, ab.pend[b] - ab.pbeg[b] > max_leaf && level < max_depth, c, s, e);
    const unsigned any = __ballot_sync(0xffffffffu, e > s);
    if (c == 0 && own < le) nch[b - lb] = __popc((any >> (threadIdx.x & 24)) & 0xffu);
}

__global__ void k_split_fill(AdaptiveBuild ab, int lb, int le, int level, const int* offs, int first_new) {
    const int c = threadIdx.x & 7, own = lb + (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 3);
    const int b = min(own, le - 1);
    const int k0 = offs[b - lb], k1 = offs[b - lb + 1];
    int s, e;
    child_range(ab, b, level, k1 > k0, c, s, e);
    const unsigned any = (__ballot_sync(0xffffffffu, e > s) >> (threadIdx.x & 24)) & 0xffu;
    if (own >= le) return;
    int k = -1;
    if (e > s) {
        k = first_new + k0 + __popc(any & ((1u << c) - 1u));
        if (DAFMM_IN(k, ab.cap, kChkSplitChild)) {
            ab.root[k] = ab.root[b];
            ab.level[k] = level + 1;
            ab.ijk[3 * (size_t)k] = 2 * ab.ijk[3 * (size_t)b] + (c & 1);
            ab.ijk[3 * (size_t)k + 1] = 2 * ab.ijk[3 * (size_t)b + 1] + ((c >> 1) & 1);
            ab.ijk[3 * (size_t)k + 2] = 2 * ab.ijk[3 * (size_t)b + 2] + ((c >> 2) & 1);
            ab.parent[k] = b;
            ab.pbeg[k] = s;
            ab.pend[k] = e;
        } else {
            k = -1;
        }
    }
    ab.child[8 * (size_t)b + c] = k;
}

__global__ void k_leaf_children_init(int* child, int b0, int b1) {
    const int b = b0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (b < b1)
        for (int c = 0; c < 8; ++c) child[8 * (size_t)b + c] = -1;
}

cudaError_t launch_split(AdaptiveBuild ab, int lb, int le, int level, int max_leaf, int max_depth, int* nch,
                         cudaStream_t s) {
    const int n = le - lb;
    if (n == 0) return cudaSuccess;
    k_split_count<<<(n + 15) / 16, 128, 0, s>>>(ab, lb, le, level, max_leaf, max_depth, nch);
    return cudaGetLastError();
}

cudaError_t launch_split_fill(AdaptiveBuild ab, int lb, int le, int level, const int* offs, int first_new,
                              cudaStream_t s) {
    const int n = le - lb;
    if (n == 0) return cudaSuccess;
    k_split_fill<<<(n + 15) / 16, 128, 0, s>>>(ab, lb, le, level, offs, first_new);
    return cudaGetLastError();
}

cudaError_t launch_children_init(int* child, int b0, int b1, cudaStream_t s) {
    if (b1 <= b0) return cudaSuccess;
    k_leaf_children_init<<<(b1 - b0 + 127) / 128, 128, 0, s>>>(child, b0, b1);
    return cudaGetLastError();
}

// Exclusive scans of n ints (out[n] = total), in tiles of 2048 per block: the tiles' sums first,
// then every block adds the sums of the tiles before its own and scans it.  One block walking the
// whole array, each thread a chunk of its own, took about 20 us at any size.
constexpr int kScanTile = 2048;

__device__ inline int block_sum_256(int v, int* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    int t = 0;
    for (int w = 0; w < 8; ++w) t += sh[w];
    __syncthreads();
    return t;
}

__global__ void __launch_bounds__(256) k_tile_sums(ScanJobs jobs, int n, int* __restrict__ sums, int ntile) {
    __shared__ int sh[8];
    const int* in = jobs.in[blockIdx.y];
    const int base = blockIdx.x * kScanTile;
    int v = 0;
    for (int i = base + threadIdx.x; i < min(base + kScanTile, n); i += 256) v += in[i];
    v = block_sum_256(v, sh);
    if (threadIdx.x == 0) sums[blockIdx.y * ntile + blockIdx.x] = v;
}

__global__ void __launch_bounds__(256) k_tile_scan(ScanJobs jobs, int n, const int* __restrict__ sums, int ntile) {
    __shared__ int sh[8];
    const int* in = jobs.in[blockIdx.y];
    int* out = jobs.out[blockIdx.y];
    const int base = blockIdx.x * kScanTile;
    int before = 0;
    for (int t = threadIdx.x; t < (int)blockIdx.x; t += 256) before += sums[blockIdx.y * ntile + t];
    int run = block_sum_256(before, sh);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int i0 = base; i0 < min(base + kScanTile, n); i0 += 256) {
        const int i = i0 + threadIdx.x;
        const int v = i < n ? in[i] : 0;
        int incl = v;
        for (int d = 1; d < 32; d <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += u;
        }
        if (lane == 31) sh[w] = incl;
        __syncthreads();
        int pre = 0, tot = 0;
        for (int k = 0; k < 8; ++k) {
            pre += k < w ? sh[k] : 0;
            tot += sh[k];
        }
        __syncthreads();
        if (i < n) out[i] = run + pre + incl - v;
        run += tot;
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = run;
}

size_t scan_temp_ints(int64_t n) { return 3 * (size_t)(n / kScanTile + 2); }

cudaError_t launch_scans(const ScanJobs& jobs, int njobs, int n, int* temp, cudaStream_t s) {
    const int ntile = n > 0 ? (n + kScanTile - 1) / kScanTile : 1;
    const dim3 grd(ntile, njobs);
    if (ntile > 1) k_tile_sums<<<grd, 256, 0, s>>>(jobs, n, temp, ntile);
    k_tile_scan<<<grd, 256, 0, s>>>(jobs, n, temp, ntile);
    return cudaGetLastError();
}

cudaError_t launch_scan(const int* in, int* out, int n, int* temp, cudaStream_t s) {
    ScanJobs j;
    j.in[0] = in;
    j.out[0] = out;
    return launch_scans(j, 1, n, temp, s);
}

// ---- colleagues ---------------------------------------------------------------------------
__device__ inline bool same_level_adjacent(const int* ijk, int a, int b) {
    for (int d = 0; d < 3; ++d) {
        const int df = ijk[3 * (size_t)a + d] - ijk[3 * (size_t)b + d];
        if (df < -1 || df > 1) return false;
    }
    return true;
}

// closed cubes of two boxes (any levels) intersect
__device__ inline bool touch(const AdaptiveBuild& ab, int a, int b) {
    const int la = ab.level[a], lb = ab.level[b];
    const int L = la > lb ? la : lb;
    for (int d = 0; d < 3; ++d) {
        // (levels up to 20: everything below 2^21)
        const int alo = ab.ijk[3 * (size_t)a + d] << (L - la), ahi = (ab.ijk[3 * (size_t)a + d] + 1) << (L - la);
        const int blo = ab.ijk[3 * (size_t)b + d] << (L - lb), bhi = (ab.ijk[3 * (size_t)b + d] + 1) << (L - lb);
        if (alo > bhi || blo > ahi) return false;
    }
    return true;
}

// Colleague k of box b, at relative position (dx, dy, dz): one thread each.  Its parent is the
// colleague of b's parent at offset floor((i_b + d) / 2) - floor(i_b / 2), its octant the parity.
// (One thread per box tested all children of the parent's colleagues.)  A block takes whole boxes:
// 27 times the boxes of a level may not fit an int.
constexpr int kColleagueBoxes = 9;

__global__ void k_colleagues(AdaptiveBuild ab, int lb, int le) {
    const int b = lb + blockIdx.x * kColleagueBoxes + threadIdx.x / 27, k = threadIdx.x % 27;
    if (b >= le) return;
    int c = k == 13 ? b : -1;
    const int P = ab.parent[b];
    if (P >= 0 && k != 13) {
        const int nx = (ab.ijk[3 * (size_t)b] & 1) + k / 9 - 1, ny = (ab.ijk[3 * (size_t)b + 1] & 1) + (k / 3) % 3 - 1,
                  nz = (ab.ijk[3 * (size_t)b + 2] & 1) + k % 3 - 1;  // in [-1, 2]: parent offset n >> 1, parity n & 1
        const int Q = ab.colleague[27 * (size_t)P + ((nx >> 1) + 1) * 9 + ((ny >> 1) + 1) * 3 + ((nz >> 1) + 1)];
        if (Q >= 0) c = ab.child[8 * (size_t)Q + ((nx & 1) | ((ny & 1) << 1) | ((nz & 1) << 2))];
    }
    ab.colleague[27 * (size_t)b + k] = c;
}

cudaError_t launch_colleagues(AdaptiveBuild ab, int lb, int le, cudaStream_t s) {
    if (le <= lb) return cudaSuccess;
    k_colleagues<<<(le - lb + kColleagueBoxes - 1) / kColleagueBoxes, 27 * kColleagueBoxes, 0, s>>>(ab, lb, le);
    return cudaGetLastError();
}

// ---- U, W (leaves) and X (all boxes) lists: count pass, then fill pass --------------------
constexpr int kStack = 256;

__device__ inline bool box_is_leaf(const AdaptiveBuild& ab, int b) {
    const int4 c0 = reinterpret_cast<const int4*>(ab.child)[2 * (size_t)b], c1 = reinterpret_cast<const int4*>(ab.child)[2 * (size_t)b + 1];
    return (c0.x & c0.y & c0.z & c0.w & c1.x & c1.y & c1.z & c1.w) < 0;  // (absent children are -1)
}

// U and W entries of leaf b among the colleague c and its descendants: c itself when it is a leaf,
// otherwise a traversal: adjacent leaves (U), boxes that are not adjacent but whose parent is (W).
// Written to ou / ow when FILL.
template <bool FILL>
__device__ void uw_colleague(const AdaptiveBuild& ab, int b, int c, int& cu, int& cw, int* ou, int* ow, int* err,
                             int cap_u, int cap_w) {
    if (box_is_leaf(ab, c)) {
        if (FILL && DAFMM_IN(cu, cap_u, kChkListFill)) ou[cu] = c;
        ++cu;
        return;
    }
    int stack[kStack];
    int sp = 0;
    for (int j = 0; j < 8; ++j)
        if (ab.child[8 * (size_t)c + j] >= 0) stack[sp++] = ab.child[8 * (size_t)c + j];
    while (sp > 0) {
        const int x = stack[--sp];
        if (touch(ab, x, b)) {
            if (box_is_leaf(ab, x)) {
                if (FILL && DAFMM_IN(cu, cap_u, kChkListFill)) ou[cu] = x;
                ++cu;
            } else {
                for (int j = 0; j < 8; ++j)
                    if (ab.child[8 * (size_t)x + j] >= 0) {
                        if (sp < kStack) stack[sp++] = ab.child[8 * (size_t)x + j];
                        else atomicExch(err, 41);
                    }
            }
        } else {
            if (FILL && DAFMM_IN(cw, cap_w, kChkListFill)) ow[cw] = x;
            ++cw;
        }
    }
}

__device__ inline int warp_scan_excl(int v, int lane, int& total) {
    int incl = v;
    for (int d = 1; d < 32; d <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += u;
    }
    total = __shfl_sync(0xffffffffu, incl, 31);
    return incl - v;
}

// The lists of box b by one warp, lane k on the colleagues at position k (one thread per box
// walked the 27 colleagues, their descendants and the ancestors' colleagues in series: 220 us at
// 32 thousand boxes, 63 us now).  Order of the entries, as a serial walk gives it: U: b, then the
// colleagues' parts by position, then the coarser leaves adjacent to b by ancestor and position;
// W: the colleagues' parts; X (all boxes): the leaf colleagues of the ancestors that are adjacent
// to parent(b) but not to b, by ancestor and position.
template <bool FILL>
__device__ void box_lists(const AdaptiveBuild& ab, int b, int lane, int& nu, int& nw, int& nx, int* ou, int* ow,
                          int* ox, int* err, int cap_u, int cap_w, int cap_x) {
    const bool leaf = box_is_leaf(ab, b);
    nu = nw = nx = 0;
    if (leaf) {
        const int c = lane < 27 && lane != 13 ? ab.colleague[27 * (size_t)b + lane] : -1;
        int cu = 0, cw = 0;
        if (c >= 0) uw_colleague<false>(ab, b, c, cu, cw, nullptr, nullptr, err, 0, 0);
        __syncwarp();
        int tu, tw;
        const int pu = 1 + warp_scan_excl(cu, lane, tu), pw = warp_scan_excl(cw, lane, tw);
        if (FILL) {
            if (lane == 0 && DAFMM_IN(0, cap_u, kChkListFill)) ou[0] = b;
            if (c >= 0) {
                cu = cw = 0;
                uw_colleague<true>(ab, b, c, cu, cw, ou + pu, ow + pw, err, cap_u - pu, cap_w - pw);
            }
            __syncwarp();
        }
        nu = 1 + tu;
        nw = tw;
    }
    const int P = ab.parent[b];
    for (int a = P; a >= 0; a = ab.parent[a]) {
        const int c = lane < 27 && lane != 13 ? ab.colleague[27 * (size_t)a + lane] : -1;
        const bool cl = c >= 0 && box_is_leaf(ab, c);
        const bool near = cl && touch(ab, c, b);
        const unsigned below = (1u << lane) - 1u;
        const unsigned mu = __ballot_sync(0xffffffffu, leaf && near);
        if (FILL && (mu >> lane & 1u) && DAFMM_IN(nu + __popc(mu & below), cap_u, kChkListFill))
            ou[nu + __popc(mu & below)] = c;
        nu += __popc(mu);
        const unsigned mx = __ballot_sync(0xffffffffu, cl && !near && touch(ab, c, P));
        if (FILL && (mx >> lane & 1u) && DAFMM_IN(nx + __popc(mx & below), cap_x, kChkListFill))
            ox[nx + __popc(mx & below)] = c;
        nx += __popc(mx);
    }
}

// V of box b (counted only): children of the parent's colleagues that are not adjacent to b
__device__ int v_count(const AdaptiveBuild& ab, int b, int lane) {
    const int P = ab.parent[b];
    if (P < 0) return 0;
    const int Q = lane < 27 && lane != 13 ? ab.colleague[27 * (size_t)P + lane] : -1;
    int cv = 0;
    for (int c = 0; c < 8 && Q >= 0; ++c) {
        const int ch = ab.child[8 * (size_t)Q + c];
        if (ch >= 0 && !same_level_adjacent(ab.ijk, ch, b)) ++cv;
    }
    __syncwarp();
    return __reduce_add_sync(0xffffffffu, cv);
}

constexpr int kListBoxes = 4;  // boxes (warps) per block

__global__ void k_list_count(AdaptiveBuild ab, int nbox, int* cu, int* cw, int* cx, unsigned long long* nv,
                             int* err) {
    const int b = blockIdx.x * kListBoxes + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    __shared__ unsigned long long sv;
    if (threadIdx.x == 0) sv = 0;
    __syncthreads();
    if (b < nbox) {
        int nu, nw, nx;
        box_lists<false>(ab, b, lane, nu, nw, nx, nullptr, nullptr, nullptr, err, 0, 0, 0);
        const int v = v_count(ab, b, lane);
        if (lane == 0) {
            cu[b] = nu;
            cw[b] = nw;
            cx[b] = nx;
            if (v) atomicAdd(&sv, (unsigned long long)v);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && sv) atomicAdd(nv, sv);
}

__global__ void k_list_fill(AdaptiveBuild ab, int nbox, const int* pu, const int* pw, const int* px, int* iu, int* iw,
                            int* ix, int* err) {
    const int b = blockIdx.x * kListBoxes + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= nbox) return;
    int nu, nw, nx;
    box_lists<true>(ab, b, lane, nu, nw, nx, iu + pu[b], iw + pw[b], ix + px[b], err, pu[b + 1] - pu[b],
                    pw[b + 1] - pw[b], px[b + 1] - px[b]);
}

cudaError_t launch_list_count(AdaptiveBuild ab, int nbox, int* cu, int* cw, int* cx, unsigned long long* nv, int* err,
                              cudaStream_t s) {
    if (nbox == 0) return cudaSuccess;
    k_list_count<<<(nbox + kListBoxes - 1) / kListBoxes, 32 * kListBoxes, 0, s>>>(ab, nbox, cu, cw, cx, nv, err);
    return cudaGetLastError();
}

cudaError_t launch_list_fill(AdaptiveBuild ab, int nbox, const int* pu, const int* pw, const int* px, int* iu, int* iw,
                             int* ix, int* err, cudaStream_t s) {
    if (nbox == 0) return cudaSuccess;
    k_list_fill<<<(nbox + kListBoxes - 1) / kListBoxes, 32 * kListBoxes, 0, s>>>(ab, nbox, pu, pw, px, iu, iw, ix, err);
    return cudaGetLastError();
}

// ---- gather of the sorted particles: FP64 SoA and FP32 offsets in each particle's own leaf ----
__global__ void k_gather_adaptive(const double* __restrict__ xyz, const double* __restrict__ q,
                                  const int* __restrict__ perm, AdaptiveBuild ab, const int* __restrict__ leaves,
                                  int nleaves, const double4* __restrict__ geom, const int* __restrict__ xq0,
                                  double* x, double* y, double* z, double* qs, float4* xq, float4* xl, int64_t n,
                                  int64_t nrec) {
    const int li = blockIdx.x;
    if (li >= nleaves) return;
    const int b = leaves[li];
    if (!DAFMM_IN(b, ab.nbox, kChkBoxIndex) || !DAFMM_RANGE(ab.pbeg[b], ab.pend[b], n, kChkBoxRange)) return;
    const double4 g = geom[b];
    const double ih = 1.0 / g.w;
    const double cx = g.x, cy = g.y, cz = g.z;
    for (int t = ab.pbeg[b] + threadIdx.x; t < ab.pend[b]; t += blockDim.x) {
        const int i = perm[t];
        if (!DAFMM_IN(i, n, kChkPerm)) continue;
        const double px = xyz[3 * (size_t)i], py = xyz[3 * (size_t)i + 1], pz = xyz[3 * (size_t)i + 2], pq = q[i];
        x[t] = px; y[t] = py; z[t] = pz; qs[t] = pq;
        const double ox = (px - cx) * ih, oy = (py - cy) * ih, oz = (pz - cz) * ih;
        const float hx = (float)ox, hy = (float)oy, hz = (float)oz;
        const int r = xq0[b] + (t - ab.pbeg[b]);
        if (!DAFMM_IN(r, nrec, kChkRecord)) continue;
        xq_store(xq, r, hx, hy, hz, (float)pq);
        xq_store(xl, r, (float)(ox - (double)hx), (float)(oy - (double)hy), (float)(oz - (double)hz),
                 (float)(pq - (double)(float)pq));
    }
}

__global__ void k_leaf_pairs(const int* __restrict__ leaves, int nl, const int* __restrict__ pbeg,
                             const int* __restrict__ pend, int* cnt) {
    const int li = blockIdx.x * blockDim.x + threadIdx.x;
    if (li < nl) {
        const int b = leaves[li];
        cnt[li] = (pend[b] - pbeg[b] + 1) >> 1;
    }
}

__global__ void k_leaf_xq0(const int* __restrict__ leaves, int nl, const int* __restrict__ off, int* xq0) {
    const int li = blockIdx.x * blockDim.x + threadIdx.x;
    if (li < nl) xq0[leaves[li]] = 2 * off[li];
}

cudaError_t launch_leaf_records(const int* leaves, int nl, const int* pbeg, const int* pend, int* cnt, int* off,
                                int* temp, int* xq0, cudaStream_t s) {
    if (nl == 0) return cudaSuccess;
    k_leaf_pairs<<<(nl + 255) / 256, 256, 0, s>>>(leaves, nl, pbeg, pend, cnt);
    cudaError_t e = launch_scan(cnt, off, nl, temp, s);
    if (e != cudaSuccess) return e;
    k_leaf_xq0<<<(nl + 255) / 256, 256, 0, s>>>(leaves, nl, off, xq0);
    return cudaGetLastError();
}

cudaError_t launch_gather_adaptive(const double* xyz, const double* q, const int* perm, AdaptiveBuild ab,
                                   const int* leaves, int nleaves, const double4* geom, const int* xq0, double* x,
                                   double* y, double* z, double* qs, float4* xq, size_t xq_n4, int64_t n, cudaStream_t s) {
    // the zero fill supplies the padding record of leaves with an odd particle count (both
    // halves: the records and their remainders)
    cudaError_t e = cudaMemsetAsync(xq, 0, 2 * xq_n4 * sizeof(float4), s);
    if (e != cudaSuccess || nleaves == 0) return e;
    k_gather_adaptive<<<nleaves, 128, 0, s>>>(xyz, q, perm, ab, leaves, nleaves, geom, xq0, x, y, z, qs, xq,
                                              xq + xq_n4, n, (int64_t)xq_n4);
    return cudaGetLastError();
}

// ---- leaves and M2L target groups --------------------------------------------------------------
__global__ void k_leaf_flags(const int* __restrict__ child, int nbox, int* flags) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbox) return;
    bool leaf = true;
    for (int j = 0; j < 8; ++j) leaf = leaf && child[8 * (size_t)b + j] < 0;
    flags[b] = leaf ? 1 : 0;
}

__global__ void k_scatter_flagged(const int* __restrict__ flags, const int* __restrict__ offs, int nbox, int* out,
                                  int* rest) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbox) return;
    if (flags[b]) out[offs[b]] = b;
    else rest[b - offs[b]] = b;
}

__global__ void k_parent_starts(LevelStarts ls, int nlev, const int* __restrict__ offs, int* out) {
    const int l = threadIdx.x;
    if (l <= nlev) out[l] = ls.v[l] - offs[ls.v[l]];
}

cudaError_t launch_parent_starts(const LevelStarts& ls, int nlev, const int* offs, int* out, cudaStream_t s) {
    k_parent_starts<<<1, 32, 0, s>>>(ls, nlev, offs, out);
    return cudaGetLastError();
}

// group key (level, octant) of the boxes of levels >= 2; other boxes sort last
__global__ void k_group_keys(const int* __restrict__ level, const int* __restrict__ ijk, int nbox, uint64_t* keys,
                             int* vals) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbox) return;
    const int l = level[b];
    const int oct = (ijk[3 * (size_t)b] & 1) | ((ijk[3 * (size_t)b + 1] & 1) << 1) | ((ijk[3 * (size_t)b + 2] & 1) << 2);
    keys[b] = l >= 2 ? (uint64_t)(l * 8 + oct) : 0xffu;
    vals[b] = b;
}

__global__ void k_group_ptr(const uint64_t* __restrict__ keys, int n, int ngroups, int* ptr) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g > ngroups) return;
    int lo = 0, hi = n;
    while (lo < hi) {
        const int m = (lo + hi) >> 1;
        if (keys[m] < (uint64_t)g) lo = m + 1;
        else hi = m;
    }
    ptr[g] = lo;
}

cudaError_t launch_leaf_flags(const int* child, int nbox, int* flags, cudaStream_t s) {
    if (nbox == 0) return cudaSuccess;
    k_leaf_flags<<<(nbox + 255) / 256, 256, 0, s>>>(child, nbox, flags);
    return cudaGetLastError();
}

cudaError_t launch_scatter_flagged(const int* flags, const int* offs, int nbox, int* out, int* rest, cudaStream_t s) {
    if (nbox == 0) return cudaSuccess;
    k_scatter_flagged<<<(nbox + 255) / 256, 256, 0, s>>>(flags, offs, nbox, out, rest);
    return cudaGetLastError();
}

cudaError_t launch_group_keys(const int* level, const int* ijk, int nbox, uint64_t* keys, int* vals, cudaStream_t s) {
    if (nbox == 0) return cudaSuccess;
    k_group_keys<<<(nbox + 255) / 256, 256, 0, s>>>(level, ijk, nbox, keys, vals);
    return cudaGetLastError();
}

cudaError_t launch_group_ptr(const uint64_t* keys, int n, int ngroups, int* ptr, cudaStream_t s) {
    k_group_ptr<<<(ngroups + 1 + 255) / 256, 256, 0, s>>>(keys, n, ngroups, ptr);
    return cudaGetLastError();
}

}  // namespace dafmm
