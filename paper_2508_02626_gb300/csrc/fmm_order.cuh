// fmm_order.cuh -- the FMM kernels of one expansion order (DAFMM_P), instantiated by fmm_p*.cu.
//
// Every expansion is stored in box-scaled variables (a box of width h becomes width 1):
//   multipole M~_a = M_a / h^|a|,  local L~_b = L_b h^|b|,
// so P2M/L2P/M2P use offsets divided by h, M2M and L2L are level-independent tables, and
// M2L is L~ = (1/h) K^_v M~ with K^_v depending only on the integer box displacement v.
//
// Kernels (paper operator -> kernel):
//   P2M  (Eq. 2)  k_p2m       one warp per leaf; each lane runs the generated straight-line
//                             P2M of one particle, a padded shared-memory transpose sums the
//                             32 lanes per coefficient
//   M2M  (Eq. 4)  k_m2m       8 parents per block; the 8 octant maps are one table with sign
//                             flips (Sec. 3.3)
//   M2L  (Eq. 5)  k_kgen      K^_v for all 316 displacements, FP64 numerical DA products of the
//                             generated transfer map (one block per v)
//                 k_m2l       L~_t = (1/h) sum_v K^_v M~_{t-v} over the 189 displacements of
//                             the target's octant (SIMT, FP64 or FP32)
//                 k_m2l_rot   the same by rotation (Sec. 3.4), FP64 and float-float: one or two
//                             targets per warp (the FP32 and MIXED M2L: tc_ops.cu, tc_gather.cu)
//   L2L  (Eq. 7)  k_l2l       32 parents and 16 rows per block, 8 child tables by sign flips
//   L2P + P2P     k_leaf      one block per target leaf (8 warps in trees of few leaves, else one):
//                 k_leaf64    pairwise sum over the 27 neighbour leaves and the generated L2P of the
//                             leaf's local expansion
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "da_common.cuh"
#include "check.cuh"
#include "ff.cuh"
#include "internal.h"
#include "launch_rules.h"
#include "tree_adaptive.h"
#include "tree_common.cuh"

#define DAFMM_CAT_(a, b) a##b
#define DAFMM_CAT(a, b) DAFMM_CAT_(a, b)
#define DAFMM_STR_(a) #a
#define DAFMM_STR(a) DAFMM_STR_(a)
#include DAFMM_STR(DAFMM_CAT(generated/da_ops_p, DAFMM_P).cuh)
#include DAFMM_STR(DAFMM_CAT(generated/da_tables_p, DAFMM_P).h)

#define GEN(name) DAFMM_CAT(name, DAFMM_CAT(_o, DAFMM_P))
#define GENT(name, suffix) DAFMM_CAT(GEN(name), suffix)

namespace dafmm {
namespace DAFMM_CAT(ord_, DAFMM_P) {

constexpr int P = DAFMM_P;
constexpr int NC = ncoef_of(P);
constexpr int NCP = ncp_of(P);

template <class T>
struct SmemSink {
    T* base;
    int lane;
    __device__ __forceinline__ void operator()(int k, T v) const { base[k * 33 + lane] = v; }
};

// Sums one coefficient per lane over the warp's 32 particles while the generated code emits
// the coefficients in increasing order: every 32 coefficients the [32][33] staging block is
// reduced row by row (lane j takes coefficient 32 c + j), so the staging needs 32 x 33
// values per warp instead of ncoef x 33.  The generated code passes k as a constant, so the
// flush tests fold away.
// NO: the number of coefficients the generated code emits (NC; the harmonic P2M: (p + 1)^2).
template <class T, int NJ, int NO = NC>
struct ChunkSink {
    T* buf;       // [32][33] per warp
    int lane;
    T (&acc)[NJ];  // acc[c] += coefficient 32 c + lane
    __device__ __forceinline__ void operator()(int k, T v) const {
        buf[(k & 31) * 33 + lane] = v;
        if ((k & 31) == 31 || k == NO - 1) {
            __syncwarp();
            if (lane <= (k & 31)) {
                T s = T(0);
#pragma unroll 8
                for (int l = 0; l < 32; ++l) s += buf[lane * 33 + l];
                acc[k >> 5] += s;
            }
            __syncwarp();
        }
    }
};

template <class T>
struct RowLoad {
    const double* row;
    __device__ __forceinline__ T operator()(int k) const { return (T)row[k]; }
};

// a row already converted to FP32 in shared memory (one conversion per coefficient per warp
// instead of one per coefficient per lane)
struct SmemRowF {
    const float* row;
    __device__ __forceinline__ float operator()(int k) const { return row[k]; }
};
// the same as float-float pairs
struct SmemRowFF {
    const ff* row;
    __device__ __forceinline__ ff operator()(int k) const { return row[k]; }
};

// the warp copies an FP64 row into `buf` as FP32
__device__ __forceinline__ void warp_row_to_f32(const double* __restrict__ row, float* buf, int lane) {
    __syncwarp();
    for (int k = lane; k < NC; k += 32) buf[k] = (float)row[k];
    __syncwarp();
}

// The steps that restore the coefficients of z exponent >= 2 of a harmonic expansion from its free
// ones by Laplace's equation (internal.h): V[i] = w1 V[i1] + w2 V[i2], those of z exponent c at
// [cst[c], cst[c + 1]).
struct HarmTab {
    static constexpr int N = NC - nharm_of(P) > 0 ? NC - nharm_of(P) : 1;
    int cst[P + 3];
    unsigned short i[N], i1[N], i2[N];
    float w1[N], w2[N], w1l[N], w2l[N];  // FP32, and its remainder (float-float)
    double d1[N], d2[N];
};
constexpr HarmTab make_harm_tab() {
    HarmTab t{};
    int k = 0;
    for (int c = 2; c <= P; ++c) {
        t.cst[c] = k;
        for (int n = c; n <= P; ++n)
            for (int b = 0; b <= n - c; ++b, ++k) {
                const int a = n - c - b;
                t.i[k] = (unsigned short)da_index(a, b, c);
                t.i1[k] = (unsigned short)da_index(a + 2, b, c - 2);
                t.i2[k] = (unsigned short)da_index(a, b + 2, c - 2);
                t.d1[k] = -(double)((a + 2) * (a + 1)) / (double)(c * (c - 1));
                t.d2[k] = -(double)((b + 2) * (b + 1)) / (double)(c * (c - 1));
                t.w1[k] = (float)t.d1[k];
                t.w2[k] = (float)t.d2[k];
                t.w1l[k] = (float)(t.d1[k] - (double)t.w1[k]);
                t.w2l[k] = (float)(t.d2[k] - (double)t.w2[k]);
            }
    }
    for (int c = P < 1 ? 2 : P + 1; c < P + 3; ++c) t.cst[c] = k;
    return t;
}
__device__ const HarmTab harm_tab = make_harm_tab();

__device__ __forceinline__ float harm_step(const float* V, int s) {
    return fmaf(harm_tab.w1[s], V[harm_tab.i1[s]], harm_tab.w2[s] * V[harm_tab.i2[s]]);
}
__device__ __forceinline__ double harm_step(const double* V, int s) {
    return fma(harm_tab.d1[s], V[harm_tab.i1[s]], harm_tab.d2[s] * V[harm_tab.i2[s]]);
}
__device__ __forceinline__ ff harm_step(const ff* V, int s) {
    return ff_add(ff_mul(ff(harm_tab.w1[s], harm_tab.w1l[s]), V[harm_tab.i1[s]]),
                  ff_mul(ff(harm_tab.w2[s], harm_tab.w2l[s]), V[harm_tab.i2[s]]));
}
// the warp restores V's coefficients of z exponent >= 2, exponent by exponent
template <class R>
__device__ __forceinline__ void harm_expand_warp(R* V, int lane) {
#pragma unroll 1
    for (int c = 2; c <= P; ++c) {
        for (int s = harm_tab.cst[c] + lane; s < harm_tab.cst[c + 1]; s += 32) V[harm_tab.i[s]] = harm_step(V, s);
        __syncwarp();
    }
}

// ---- P2M ---------------------------------------------------------------------------------
// the full FP64 row from a warp's free coefficients (acc[c]: coefficient 32 c + lane), by way of the
// staging block sm
template <class T, int NJ>
__device__ __forceinline__ void p2m_row(const T (&acc)[NJ], T* sm, double* __restrict__ row, int lane) {
    __syncwarp();
#pragma unroll
    for (int j = 0; j < NJ; ++j)
        if (lane + 32 * j < nharm_of(P)) sm[harm_full_index(lane + 32 * j)] = acc[j];
    __syncwarp();
    harm_expand_warp(sm, lane);
    for (int k = lane; k < NC; k += 32) row[k] = (double)sm[k];
}

// rows32: the multipole rows are FP32 (NCP floats per leaf) instead of FP64.  The FP32 kernel
// reads the particles' FP32 leaf-frame records, which hold exactly the values it would compute
// from the FP64 coordinates ((x - c) / h rounded once to FP32), without FP64 arithmetic.
// H: the harmonic basis -- the generated code emits only the (p + 1)^2 free coefficients
// (z exponent <= 1), which are summed and written at their layout positions; the others are
// not computed (the multipole's homogeneous parts are harmonic, Eq. 2, so they are implied).  FP64
// and float-float (always H) restore them here, once per leaf, by Laplace's equation: the rows are
// complete, with 0.4 times the arithmetic per particle at p = 8 (N = 200,003, depth 4: FP64 672 -> 315
// us, float-float 493 -> 138 us).
// f16 (H, FP32 rows): the row's F16 split as well, as tc_split_f16_multi makes it -- the warp
// holds the whole row, so its largest magnitude is one warp reduction away.
template <class T, bool H = false>
__global__ void k_p2m(TreeView tv, double* __restrict__ M, int rows32, F16Rows f16) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw) + threadIdx.y * (32 * 33);
    const int lane = threadIdx.x;
    const int leaf = blockIdx.x * blockDim.y + threadIdx.y;
    if (leaf >= tv.nleaf) return;
    int i0 = tv.leaf_start[leaf], i1 = tv.leaf_start[leaf + 1];
    if (!DAFMM_RANGE(i0, i1, tv.n, kChkLeafRange)) i0 = i1 = 0;
    int a, b, c;
    octmajor_decode(tv.depth, leaf, a, b, c);
    const double cx = tv.x0 + ((double)a + 0.5) * tv.h_leaf;
    const double cy = tv.y0 + ((double)b + 0.5) * tv.h_leaf;
    const double cz = tv.z0 + ((double)c + 0.5) * tv.h_leaf;
    const int r_own = xq_base(i0, leaf) - i0;  // FP32 record of sorted position i: i + r_own
    constexpr int NO = H ? nharm_of(P) : NC;
    constexpr int NJ = (NO + 31) / 32;
    T acc[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[j] = T(0);
    ChunkSink<T, NJ, NO> sink{sm, lane, acc};
    for (int base = i0; base < i1; base += 32) {
        const int i = base + lane;
        T x = T(0), y = T(0), z = T(0), q = T(0);
        if (i < i1) {
            if constexpr (sizeof(T) == 4) {
                const float4 r = xq_load(tv.xq, i + r_own);
                x = r.x;
                y = r.y;
                z = r.z;
                q = r.w;
            } else {
                x = (T)((tv.x[i] - cx) * tv.inv_h_leaf);
                y = (T)((tv.y[i] - cy) * tv.inv_h_leaf);
                z = (T)((tv.z[i] - cz) * tv.inv_h_leaf);
                q = (T)tv.q[i];
            }
        }
        if constexpr (H) gen::GEN(p2mh)<T>(x, y, z, q, sink);
        else gen::GEN(p2m)<T>(x, y, z, q, sink);
    }
    if (rows32) {
        float* Mf = reinterpret_cast<float*>(M) + (size_t)leaf * NCP;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const int k = lane + 32 * j;
            if (k < NO) Mf[H ? harm_full_index(k) : k] = (float)acc[j];
        }
        if constexpr (H && sizeof(T) == 4) {
            if (f16.hi) {
                float mx = 0.f;
#pragma unroll
                for (int j = 0; j < NJ; ++j)
                    if (lane + 32 * j < NO) mx = fmaxf(mx, fabsf((float)acc[j]));
                for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                int e = 0;
                if (mx > 0.f) frexpf(mx, &e);  // mx = f 2^e, f in [0.5, 1)
                e = e < -120 ? -120 : (e > 120 ? 120 : e);
                const float sc = ldexpf(1.f, -e);
                __half* hi = static_cast<__half*>(f16.hi) + (size_t)leaf * f16.rowlen;
                __half* lo = static_cast<__half*>(f16.lo) + (size_t)leaf * f16.rowlen;
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const int k = lane + 32 * j;
                    if (k >= f16.rowlen) break;
                    const float f = (k < NO ? (float)acc[j] : 0.f) * sc;
                    const __half h = __float2half_rn(f);
                    hi[k] = h;
                    lo[k] = __float2half_rn(f - __half2float(h));
                }
                if (lane == 0) f16.inv[leaf] = ldexpf(1.f, e);
            }
        }
        return;
    }
    if constexpr (H && sizeof(T) == 8) {
        p2m_row(acc, sm, M + (size_t)leaf * NCP, lane);
        return;
    }
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = lane + 32 * j;
        if (k < NO) M[(size_t)leaf * NCP + (H ? harm_full_index(k) : k)] = (double)acc[j];
    }
}

// ---- M2M / L2L ------------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ T tab_val(const ShiftTab& t, int e);
template <>
__device__ __forceinline__ double tab_val<double>(const ShiftTab& t, int e) { return t.val[e]; }
template <>
__device__ __forceinline__ float tab_val<float>(const ShiftTab& t, int e) { return t.valf[e]; }

constexpr int SH_ROWS = (NC + 7) / 8;  // output rows per warp (8 warps)

// Both shifts use the octant structure of Sec. 3.3: the entry (b, a) of the table of child
// octant c is the octant-0 entry times (-1)^popcount(par & c), par = parity pattern of the
// entry.  Summing over the 8 octants first -- the Hadamard transform
//   S_m[a] = sum_c (-1)^popcount(m & c) M_c[a]
// -- turns the 8 signed products per entry into one: parent M[b] = sum_e val_e S_{par_e}[col_e].
// For L2L the transform runs the other way: R_m[b] = sum_{e of parity m} val_e L[col_e], and
// child c receives sum_m (-1)^popcount(m & c) R_m[b].  Table entries are stored per row in
// parity order (tab.rp8).
template <class T>
__device__ __forceinline__ void hadamard8(T (&m)[8]) {
#pragma unroll
    for (int h = 1; h < 8; h <<= 1)
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (!(i & h)) {
                const T a = m[i], b = m[i | h];
                m[i] = a + b;
                m[i | h] = a - b;
            }
}

// The parents of one level's shift and where their rows lie.  Uniform trees: parent i of level
// lc - 1 in the order of its children's octant slabs.  Adaptive trees: box list[i]; only boxes
// with children are listed (at most one box in about eight has any, so a walk over all boxes
// left most lanes idle).
struct ShiftUniform {
    int lc, n;  // children's level, parents
    __device__ __forceinline__ int parent(int i) const {
        const int Pc = 1 << (lc - 1);
        return octmajor_index(lc - 1, i % Pc, (i / Pc) % Pc, i / (Pc * Pc));
    }
    __device__ __forceinline__ int child(int i, int c) const { return c * n + i; }
};
struct ShiftAdaptive {
    AdaptiveView av;
    const int* list;
    int n;
    __device__ __forceinline__ int parent(int i) const { return list[i]; }
    __device__ __forceinline__ int child(int i, int c) const {
        const int ch = av.child[8 * (size_t)list[i] + c];
        return ch >= 0 && DAFMM_IN(ch, av.nbox, kChkBoxIndex) ? ch : -1;
    }
};

// parents per thread block of the M2M kernel: 8.  The output rows of a parent are then spread
// over 32 threads (4 lanes in each of the 8 warps) and a level of 4096 parents over 512 blocks.
constexpr int kM2MParents = 8;
// rows of S: the coefficients staged per box, made odd (bank conflicts)
template <bool H>
constexpr int m2m_stride() {
    return (H ? nharm_of(P) : NC) | 1;
}
// the transformed children S [8][kM2MParents][stride], and (harmonic) the table's entries
template <class T, bool H>
constexpr size_t m2m_smem(int nnz) {
    return (size_t)8 * kM2MParents * m2m_stride<H>() * sizeof(T) + (H ? (size_t)nnz * (sizeof(T) + 2) : 0);
}

// M2M (Eq. 4) from the children into the parents of one level.  H: harmonic multipoles -- tab is
// the harmonic M2M table (rows and columns by free index), which reads and writes only the free
// coefficients.  Its entries are staged in shared memory, the parity and column of an entry as
// one offset into S: read from global memory they are a chain of dependent loads per entry.  The
// rows go to the lanes in order of decreasing length (tab.ord), so that the four rows a warp works
// on at a time end together.  Measured, all levels: clustered N = 4e6, p = 10, FP64: 2.86 -> 0.63
// ms (mostly the parents' list); uniform N = 1e6, p = 8: FP64 89 -> 78 us, FP32 40 -> 32 us.
template <class T, bool H, class Fam>
__global__ void __launch_bounds__(256) k_m2m(ShiftTab tab, const __grid_constant__ Fam fam, const double* Mc,
                                             double* Mp, int rows32) {
    constexpr int PP = kM2MParents, RS = 32 / PP, ST = m2m_stride<H>(), NO = H ? nharm_of(P) : NC;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* S = reinterpret_cast<T*>(smem_raw);
    T* tv = S + 8 * PP * ST;
    unsigned short* tx = reinterpret_cast<unsigned short*>(tv + (H ? tab.nnz : 0));
    if constexpr (H) {
        for (int e = threadIdx.x; e < tab.nnz; e += 256) {
            tv[e] = tab_val<T>(tab, e);
            tx[e] = (unsigned short)(tab.par[e] * (PP * ST) + tab.col[e]);
        }
    }
    const int i0 = blockIdx.x * PP;
    for (int e = threadIdx.x; e < PP * NO; e += 256) {
        const int r = e / NO, j = e - r * NO;
        const int k = H ? harm_full_index(j) : j;
        T m[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int ch = i0 + r < fam.n ? fam.child(i0 + r, c) : -1;
            const size_t at = (size_t)ch * NCP + k;
            m[c] = ch < 0 ? T(0) : rows32 ? (T)reinterpret_cast<const float*>(Mc)[at] : (T)Mc[at];
        }
        hadamard8(m);
#pragma unroll
        for (int q = 0; q < 8; ++q) S[(q * PP + r) * ST + j] = m[q];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int r = lane % PP, sub = lane / PP;
    if (i0 + r >= fam.n) return;
    const size_t ob = (size_t)fam.parent(i0 + r) * NCP;
    const T* Sr = S + r * ST;
    for (int jj = w * RS + sub; jj < NO; jj += 8 * RS) {
        const int j = tab.ord ? tab.ord[jj] : jj;
        T acc = T(0);
        if constexpr (H) {
#pragma unroll 4
            for (int e = tab.rowptr[j]; e < tab.rowptr[j + 1]; ++e) acc += tv[e] * Sr[tx[e]];
        } else {
            for (int e = tab.rowptr[j]; e < tab.rowptr[j + 1]; ++e)
                acc += tab_val<T>(tab, e) * Sr[tab.par[e] * (PP * ST) + tab.col[e]];
        }
        const size_t at = ob + (H ? harm_full_index(j) : j);
        if (rows32) reinterpret_cast<float*>(Mp)[at] = (float)acc;
        else Mp[at] = (double)acc;
    }
}

// L2L (Eq. 7): the children of one level's parents receive the parents' locals (added to what
// M2L and P2L wrote).  A block takes 32 parents (one per lane) and 16 rows of the table (one per
// warp), so that even a level of 64 parents spreads over ncoef / 16 blocks; the parents' columns
// and the rows' table entries are staged in shared memory, and the 8 children's results pass
// through it so that their rows are updated in whole 128-byte (FP64) segments.  The form before
// (8 warps walking all rows, entries read from global memory one dependent load after another,
// strided updates) took about 170 us per level whatever its size.  Measured, all levels: uniform
// N = 1e6, p = 8, FP64: 509 -> 125 us; clustered N = 4e6, p = 10, FP64: 4.35 -> 1.83 ms; 64-problem
// forest, p = 6, FP32: 235 -> 57 us.
constexpr int kL2LRows = 16;
template <class T>
constexpr size_t l2l_smem(int maxe) {
    return ((size_t)32 * (NCP + 1) + (size_t)8 * 32 * (kL2LRows + 1) + maxe) * sizeof(T) + (size_t)maxe * 2;
}

template <class T, class Fam>
__global__ void __launch_bounds__(32 * kL2LRows) k_l2l(ShiftTab tab, const __grid_constant__ Fam fam, int maxe,
                                                       const double* Lp, double* Lc) {
    constexpr int ST = NCP + 1, OR = kL2LRows + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* src = reinterpret_cast<T*>(smem_raw);  // [32][ST]
    T* out = src + 32 * ST;                   // [8][32][OR]
    T* tv = out + 8 * 32 * OR;                // the rows' entries
    unsigned short* tc = reinterpret_cast<unsigned short*>(tv + maxe);
    const int b0 = blockIdx.y * kL2LRows, nb = min(kL2LRows, NC - b0);
    const int i0 = blockIdx.x * 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int e0 = tab.rowptr[b0], e1 = tab.rowptr[b0 + nb];
    for (int e = e0 + (int)threadIdx.x; e < e1; e += 32 * kL2LRows) {
        tv[e - e0] = tab_val<T>(tab, e);
        tc[e - e0] = tab.col[e];
    }
    // row b reads columns a >= b componentwise only, which have indices >= b
    for (int r = w; r < 32; r += kL2LRows) {
        if (i0 + r >= fam.n) break;
        const double* row = Lp + (size_t)fam.parent(i0 + r) * NCP;
        for (int k = b0 + lane; k < NC; k += 32) src[r * ST + k] = (T)row[k];
    }
    __syncthreads();
    if (w < nb && i0 + lane < fam.n) {
        const T* srow = src + lane * ST;
        const int* rp = tab.rp8 + 8 * (b0 + w);
        T R[8];
        int nm = 0;  // parity classes with entries, class 0 aside
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            T s = T(0);
            const int ea = rp[m] - e0, ez = rp[m + 1] - e0;
#pragma unroll 4
            for (int e = ea; e < ez; ++e) s += tv[e] * srow[tc[e]];
            R[m] = s;
            nm += m > 0 && ez > ea;
        }
        if (nm > 0) {
            hadamard8(R);  // R[c] = what child octant c receives
        } else {
#pragma unroll
            for (int c = 1; c < 8; ++c) R[c] = R[0];  // (the top degree's rows: one entry)
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) out[(c * 32 + lane) * OR + w] = R[c];
    }
    __syncthreads();
    const int i = threadIdx.x % kL2LRows;
    if (i >= nb) return;
    for (int g = threadIdx.x / kL2LRows; g < 8 * 32; g += 32) {
        const int r = g & 31, c = g >> 5;
        if (i0 + r >= fam.n) continue;
        const int ch = fam.child(i0 + r, c);
        if (ch >= 0) Lc[(size_t)ch * NCP + b0 + i] += (double)out[g * OR + i];
    }
}

// ---- K generation (Eq. 5 as a matrix per displacement) -------------------------------------
// K^_v[b][a] = coefficient b of sqrt(R) (M2)^a, M2 = (v + u) R, R = 1/|v + u|^2, boxes of width 1.
__device__ void da_mul_block(const MulTab& mt, const double* A, const double* B, double* C) {
    for (int k = threadIdx.x; k < NC; k += blockDim.x) {
        double s = 0.0;
        for (int e = mt.rowptr[k]; e < mt.rowptr[k + 1]; ++e) {
            const ushort2 pr = mt.pairs[e];
            s = fma(A[pr.x], B[pr.y], s);
        }
        C[k] = s;
    }
    __syncthreads();
}

struct SmemStore {
    double* o;
    __device__ __forceinline__ void operator()(int k, double v) const { o[k] = v; }
};

// r0s (optional): block b computes the matrix of the displacement r0s[3 b .. 3 b + 2] (any
// real vector, e.g. along an axis) into slot b of K64, instead of an integer key's
__global__ void __launch_bounds__(256) k_kgen(MulTab mt, double* __restrict__ K64, float* __restrict__ K32,
                                              int key_only, const short* __restrict__ key_list,
                                              const double* __restrict__ r0s) {
    __shared__ double buf[8][NCP];
    const int key = key_only >= 0 ? key_only : (key_list ? key_list[blockIdx.x] : blockIdx.x);
    const int vx = key / 49 - 3, vy = (key / 7) % 7 - 3, vz = key % 7 - 3;
    const int amax = max(abs(vx), max(abs(vy), abs(vz)));
    if (!r0s && amax <= 1) return;  // adjacent boxes never interact through M2L
    double* sR = buf[0];
    double* m2[3] = {buf[1], buf[2], buf[3]};
    double* X = buf[4];
    double* XY = buf[5];
    double* Z0 = buf[6];
    double* Z1 = buf[7];
    const double v[3] = {r0s ? r0s[3 * blockIdx.x] : (double)vx, r0s ? r0s[3 * blockIdx.x + 1] : (double)vy,
                         r0s ? r0s[3 * blockIdx.x + 2] : (double)vz};
    const size_t slot = r0s ? blockIdx.x : (size_t)(key_only >= 0 ? 0 : key);
    const double rho = 1.0 / (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    if (threadIdx.x == 0) {
        gen::GEN(m2lmap_inv)<double>(v[0], v[1], v[2], rho, SmemStore{X});
        gen::GEN(m2lmap_isq)<double>(v[0], v[1], v[2], rho, SmemStore{sR});
    }
    __syncthreads();
    const double srho = sqrt(rho);
    for (int k = threadIdx.x; k < NC; k += blockDim.x) {
        X[k] *= rho;      // R
        sR[k] *= srho;    // sqrt(R)
    }
    __syncthreads();
    for (int k = threadIdx.x; k < NC; k += blockDim.x)
        for (int d = 0; d < 3; ++d) {
            const int km = mt.minus[d * NC + k];
            m2[d][k] = v[d] * X[k] + (km >= 0 ? X[km] : 0.0);
        }
    __syncthreads();
    // monomials (M2)^(a,b,c): X = M2x^a, XY = X M2y^b, Z = XY M2z^c
    for (int k = threadIdx.x; k < NC; k += blockDim.x) X[k] = (k == 0) ? 1.0 : 0.0;
    __syncthreads();
    double* Xn = XY;  // scratch while stepping X
    for (int a = 0; a <= P; ++a) {
        if (a > 0) {
            da_mul_block(mt, X, m2[0], Z0);
            for (int k = threadIdx.x; k < NC; k += blockDim.x) X[k] = Z0[k];
            __syncthreads();
        }
        for (int k = threadIdx.x; k < NC; k += blockDim.x) Xn[k] = X[k];
        __syncthreads();
        for (int b = 0; b <= P - a; ++b) {
            if (b > 0) {
                da_mul_block(mt, Xn, m2[1], Z0);
                for (int k = threadIdx.x; k < NC; k += blockDim.x) Xn[k] = Z0[k];
                __syncthreads();
            }
            double* Zc = Z0;
            double* Zn = Z1;
            for (int k = threadIdx.x; k < NC; k += blockDim.x) Zc[k] = Xn[k];
            __syncthreads();
            for (int c = 0; c <= P - a - b; ++c) {
                if (c > 0) {
                    da_mul_block(mt, Zc, m2[2], Zn);
                    double* t = Zc; Zc = Zn; Zn = t;
                }
                // column alpha = sqrt(R) * Z  -> K[key][beta][alpha]
                const int alpha = da_index(a, b, c);
                double* out = K64 + slot * NC * NCP;
                float* out32 = K32 ? K32 + slot * NC * NCP : nullptr;
                for (int k = threadIdx.x; k < NC; k += blockDim.x) {
                    double s = 0.0;
                    for (int e = mt.rowptr[k]; e < mt.rowptr[k + 1]; ++e) {
                        const ushort2 pr = mt.pairs[e];
                        s = fma(sR[pr.x], Zc[pr.y], s);
                    }
                    out[(size_t)k * NCP + alpha] = s;
                    if (out32) out32[(size_t)k * NCP + alpha] = (float)s;
                }
                __syncthreads();
            }
        }
    }
}

// ---- M2L (SIMT) ----------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ const T* ktab(const double* K64, const float* K32);
template <>
__device__ __forceinline__ const double* ktab<double>(const double* K64, const float*) { return K64; }
template <>
__device__ __forceinline__ const float* ktab<float>(const double*, const float* K32) { return K32; }

// targets: level l, octant blockIdx.y, 32 consecutive parent positions per block
template <class T, class Src>
__global__ void __launch_bounds__(256) k_m2l(const T* __restrict__ K, int l, const Src* __restrict__ M,
                                             double* __restrict__ L, double inv_h) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* src = reinterpret_cast<T*>(smem_raw);  // [32][NCP + 1]
    __shared__ int sidx[32];
    const int Pp = 1 << (l - 1);  // parents per axis
    const int nlin = Pp * Pp * Pp;
    const int oct = blockIdx.y;
    const int lin0 = blockIdx.x * 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ox = oct & 1, oy = (oct >> 1) & 1, oz = (oct >> 2) & 1;
    const int n_side = 1 << l;
    T acc[SH_ROWS];
#pragma unroll
    for (int j = 0; j < SH_ROWS; ++j) acc[j] = T(0);
    for (int vx = -3 + ox; vx <= 2 + ox; ++vx)
        for (int vy = -3 + oy; vy <= 2 + oy; ++vy)
            for (int vz = -3 + oz; vz <= 2 + oz; ++vz) {
                if (abs(vx) <= 1 && abs(vy) <= 1 && abs(vz) <= 1) continue;
                if (threadIdx.x < 32) {
                    const int lin = lin0 + threadIdx.x;
                    int s = -1;
                    if (lin < nlin) {
                        const int px = lin % Pp, py = (lin / Pp) % Pp, pz = lin / (Pp * Pp);
                        const int tx = 2 * px + ox, ty = 2 * py + oy, tz = 2 * pz + oz;
                        const int sx = tx - vx, sy = ty - vy, sz = tz - vz;
                        if (sx >= 0 && sy >= 0 && sz >= 0 && sx < n_side && sy < n_side && sz < n_side)
                            s = octmajor_index(l, sx, sy, sz);
                    }
                    sidx[threadIdx.x] = s;
                }
                __syncthreads();
                for (int e = threadIdx.x; e < 32 * NC; e += 256) {
                    const int r = e / NC, k = e - r * NC;
                    const int s = sidx[r];
                    src[r * (NCP + 1) + k] = s >= 0 ? (T)M[(size_t)s * NCP + k] : T(0);
                }
                __syncthreads();
                const int key = (vx + 3) * 49 + (vy + 3) * 7 + (vz + 3);
                const T* Kv = K + (size_t)key * NC * NCP;
                const T* srow = src + lane * (NCP + 1);
                const T* kw = Kv + (size_t)w * NCP;  // rows b = w + 8 j
#pragma unroll 1
                for (int a = 0; a < NC; ++a) {
                    const T sv = srow[a];
#pragma unroll
                    for (int j = 0; j < SH_ROWS; ++j)
                        if (w + 8 * j < NC) acc[j] = fma(kw[(size_t)(8 * j) * NCP + a], sv, acc[j]);
                }
                __syncthreads();
            }
    const int lin = lin0 + lane;
    if (lin < nlin) {
        const int t = oct * nlin + lin;
#pragma unroll
        for (int j = 0; j < SH_ROWS; ++j) {
            const int b = w + 8 * j;
            if (b < NC) L[(size_t)t * NCP + b] = (double)acc[j] * inv_h;
        }
    }
}

// ---- M2L by rotation (Sec. 3.4), FP64 -------------------------------------------------------
// K^_v = B_v A_|v| F_v: F_v rotates the source expansion so that v lies on the positive x axis
// (M^(u) = M(Q^T u), Q = Rz(phi) Rx(theta) with theta = atan2(vz, vy), phi = atan2(sqrt(vy^2 +
// vz^2), vx)), A_rho is Eq. 5 along the axis (displacement (rho, 0, 0)), and B_v rotates the
// result back (L(d) = L^(Q d)).  A linear substitution keeps every degree apart; a rotation
// about one axis moves only the other two variables, so it acts on the binary forms of fixed
// exponent of the untouched variable: the form of degree m in (p, q) is multiplied by the
// (m+1) x (m+1) matrix of p -> al p + be q, q -> ga p + de q.  The four substitutions (forward
// about x then z, back about z then x) are tabulated per displacement key; A_rho is sparse:
// column (a, b, c) reaches row (a', b', c') only when b' >= b, c' >= c and both differences are
// even (the axial map depends on y and z through y^2 + z^2 and odd powers of y, z alone).
constexpr int ROT_TSZ = (P + 1) * (P + 2) * (2 * P + 3) / 6;  // sum over m <= P of (m+1)^2

__host__ __device__ constexpr int rot_off(int m) { return m * (m + 1) * (2 * m + 1) / 6; }
// per key: the four substitution matrices (forward x-step, forward z-step, back z-step, back
// x-step), each packed over m = 0..P
__global__ void __launch_bounds__(128) k_rot_tables(double* __restrict__ T) {
    const int key = blockIdx.x;
    const double vx = key / 49 - 3, vy = (key / 7) % 7 - 3, vz = key % 7 - 3;
    const double ryz = sqrt(vy * vy + vz * vz), rho = sqrt(vx * vx + vy * vy + vz * vz);
    const double c1 = ryz > 0.0 ? vy / ryz : 1.0, s1 = ryz > 0.0 ? vz / ryz : 0.0;
    const double c2 = rho > 0.0 ? vx / rho : 1.0, s2 = rho > 0.0 ? ryz / rho : 0.0;
    // (al, be, ga, de) per substitution: old p = al p' + be q', old q = ga p' + de q'
    const double sub[4][4] = {{c1, -s1, s1, c1}, {c2, -s2, s2, c2}, {c2, s2, -s2, c2}, {c1, s1, -s1, c1}};
    for (int e = threadIdx.x; e < 4 * ROT_TSZ; e += blockDim.x) {
        const int w = e / ROT_TSZ, r = e - w * ROT_TSZ;
        int m = 0;
        while (rot_off(m + 1) <= r) ++m;
        const int i = (r - rot_off(m)) / (m + 1), j = (r - rot_off(m)) % (m + 1);
        const double al = sub[w][0], be = sub[w][1], ga = sub[w][2], de = sub[w][3];
        // coefficient of p^(m-i) q^i in (al p + be q)^(m-j) (ga p + de q)^j
        double acc = 0.0;
        for (int k = 0; k <= i; ++k) {  // k from the first factor, i - k from the second
            if (k > m - j || i - k > j) continue;
            double c_a = 1.0, c_b = 1.0;
            for (int t = 0; t < k; ++t) c_a = c_a * (m - j - t) / (t + 1);
            for (int t = 0; t < i - k; ++t) c_b = c_b * (j - t) / (t + 1);
            double pw = c_a * c_b;
            for (int t = 0; t < m - j - k; ++t) pw *= al;
            for (int t = 0; t < k; ++t) pw *= be;
            for (int t = 0; t < j - (i - k); ++t) pw *= ga;
            for (int t = 0; t < i - k; ++t) pw *= de;
            acc += pw;
        }
        T[(size_t)key * 4 * ROT_TSZ + e] = acc;
    }
}

// the axial matrices [nrho][NC][NCP] (dense, from k_kgen) -> their structural non-zeros
__global__ void k_axial_gather(const double* __restrict__ K, const int* __restrict__ rowptr,
                               const unsigned short* __restrict__ col, int nnz, double* __restrict__ val) {
    const int r = blockIdx.x;
    for (int b = threadIdx.x; b < NC; b += blockDim.x)
        for (int e = rowptr[b]; e < rowptr[b + 1]; ++e)
            val[(size_t)r * nnz + e] = K[((size_t)r * NC + b) * NCP + col[e]];
}

// the arithmetic of the rotation M2L: FP64, or float-float (the DAFMM_FF mode)
__device__ __forceinline__ double rot_add(double a, double b) { return a + b; }
__device__ __forceinline__ ff rot_add(ff a, ff b) { return ff_acc(a, b); }
template <class R>
__device__ __forceinline__ R rot_zero() { return R(0.0); }
__device__ __forceinline__ double rot_to_double(double a) { return a; }
__device__ __forceinline__ double rot_to_double(ff a) { return a.to_double(); }

// running sums of a rotation step's output.  FP64: a plain fma chain.  Float-float: a cascaded
// sum (as Ogita, Rump and Oishi's Sum2): each product's high part joins the high sum through
// TwoSum and its rounding error, with the product's low part, joins the low sum; the pair is
// renormalised once per output.  A renormalisation per term (ff_acc) would put about eight
// dependent FP32 operations between consecutive terms of a lane's chain instead of two adds.
struct RotAccD {
    double s = 0.0;
    __device__ __forceinline__ void madd(double a, double b) { s = fma(a, b, s); }
    __device__ __forceinline__ double get() const { return s; }
};
struct RotAccF {
    float hi = 0.f, lo = 0.f;
    // the product enters unnormalised: its rounded high part p through TwoSum, and p's exact
    // rounding error plus the cross terms (a.hi b.lo + a.lo b.hi) into the low sum (13 FP32
    // operations instead of 16 with a renormalised product; the low sum's rounding stays of
    // the order u^2 |a b|)
    __device__ __forceinline__ void madd(ff a, ff b) {
        const float p = mul_rn(a.hi, b.hi);
        const float e = fmaf(a.hi, b.hi, -p) + fmaf(a.hi, b.lo, mul_rn(a.lo, b.hi));
        const ff t = two_sum(hi, p);
        hi = t.hi;
        lo += t.lo + e;
    }
    __device__ __forceinline__ ff get() const { return fast_two_sum(hi, lo); }
};
template <class R>
struct RotAcc;
template <>
struct RotAcc<double> {
    using type = RotAccD;
};
template <>
struct RotAcc<ff> {
    using type = RotAccF;
};

// The tables of the rotation M2L in the order in which the kernel reads them.  Each of the five
// steps of a pair runs, per lane, a list of multiply-adds out[k] += tab * in[i] (a precomputed,
// load-balanced share of the step, whole outputs per lane, padded to a common length with tasks
// that read the zero at in[NC]; lanes with outputs of very different lengths would otherwise run
// every loop to the longest one).  Task t of lane l: the word idx[32 t + l] = input index | output
// index << 9 | last-of-output << 31, the same for every displacement, and its table value at
// val[32 t + l] -- per key the four substitutions' values one after another (forward x, forward
// z, back z, back x), the axial values per distinct length.  A warp's reads are then whole
// 128-byte lines; gathered from the packed matrices, 32 lanes read 32 scattered values and the L1
// held the kernel below the FP64 rate, and far below the FP32 rate in float-float.
struct RotStream {
    const unsigned* idx;  // x-step, z-step, axial: [lx + lz + la][32]
    int lx, lz, la;
    const int* krho;      // per key, the index of its length
};

template <bool ACC, int NV, class R>
__device__ __forceinline__ void rot_step(const unsigned* __restrict__ idx, int len, const R* __restrict__ val,
                                         R* const (&in)[NV], R* const (&out)[NV], int lane) {
    typename RotAcc<R>::type s[NV];
#pragma unroll 4
    for (int t = 0; t < len; ++t) {
        const unsigned w = idx[32 * t + lane];
        const R v = val[32 * t + lane];
        const int i = (int)(w & 511u), k = (int)((w >> 9) & 511u);
        if (DAFMM_IN(i, NC + 1, kChkRotTask)) {
#pragma unroll
            for (int u = 0; u < NV; ++u) s[u].madd(v, in[u][i]);
        }
        if (w >> 31) {
#pragma unroll
            for (int u = 0; u < NV; ++u) {
                if (DAFMM_IN(k, NC, kChkRotTask)) {
                    if (ACC) out[u][k] = rot_add(out[u][k], s[u].get());
                    else out[u][k] = s[u].get();
                }
                s[u] = typename RotAcc<R>::type();
            }
        }
    }
}

// the multipole rows: FP64, or (float-float) their FP32 high and low parts, split once per
// evaluation
struct RotRows {
    const double* M;
    const float *Mh, *Ml;
};
__device__ __forceinline__ void rot_load(double* X, const RotRows& m, size_t row, int lane) {
    for (int k = lane; k < NC; k += 32) X[k] = m.M[row + k];
}
__device__ __forceinline__ void rot_load(ff* X, const RotRows& m, size_t row, int lane) {
    for (int k = lane; k < NC; k += 32) X[k] = ff(m.Mh[row + k], m.Ml[row + k]);
}

// NV well-separated pairs of one displacement key for the warp: S[u] += B_v A_|v| F_v M_src[u]
// (X, Y: work vectors with X[NC] = Y[NC] = 0).  HARM: harmonic task lists (free outputs only),
// the vector restored before the last x-step
template <bool HARM, int NV, class R>
__device__ __forceinline__ void rot_pairs(const RotStream& rs, const R* __restrict__ val, const R* __restrict__ ax,
                                          const RotRows& m, const int (&src)[NV], R* const (&X)[NV],
                                          R* const (&Y)[NV], R* const (&S)[NV], int lane) {
    __syncwarp();
#pragma unroll
    for (int u = 0; u < NV; ++u) rot_load(X[u], m, (size_t)src[u] * NCP, lane);
    __syncwarp();
    const unsigned *iz = rs.idx + 32 * rs.lx, *ia = iz + 32 * rs.lz;
    rot_step<false, NV>(rs.idx, rs.lx, val, X, Y, lane);  // forward, about x
    __syncwarp();
    rot_step<false, NV>(iz, rs.lz, val + 32 * rs.lx, Y, X, lane);  // forward, about z
    __syncwarp();
    rot_step<false, NV>(ia, rs.la, ax, X, Y, lane);  // Eq. 5 on the axis
    __syncwarp();
    rot_step<false, NV>(iz, rs.lz, val + 32 * (rs.lx + rs.lz), Y, X, lane);  // back, about z
    __syncwarp();
    if constexpr (HARM) {  // the x-step reads every z exponent
#pragma unroll
        for (int u = 0; u < NV; ++u) harm_expand_warp(X[u], lane);
    }
    rot_step<true, NV>(rs.idx, rs.lx, val + 32 * (rs.lx + 2 * rs.lz), X, S, lane);  // back, about x, into the sums
}

// Where the targets of one octant lie and their sources.  Uniform trees: octant oct of level l.
// Adaptive trees: the group of one (level, octant); the source of displacement v is child sc of
// the parent's colleague at offset a (o - v = 2a + sc).
struct RotUniform {
    int l;
    double inv_h;
    __device__ __forceinline__ int target(int oct, int i) const {
        const int P3 = 1 << (3 * (l - 1));
        return i < P3 ? oct * P3 + i : -1;
    }
    __device__ __forceinline__ int source(int t, int oct, const int (&v)[3]) const {
        const int Pp = 1 << (l - 1), lin = t & ((1 << (3 * (l - 1))) - 1), n = 1 << l;
        const int x = 2 * (lin & (Pp - 1)) + (oct & 1) - v[0], y = 2 * ((lin >> (l - 1)) & (Pp - 1)) + ((oct >> 1) & 1) - v[1],
                  z = 2 * (lin >> (2 * (l - 1))) + ((oct >> 2) & 1) - v[2];
        return x >= 0 && y >= 0 && z >= 0 && x < n && y < n && z < n ? octmajor_index(l, x, y, z) : -1;
    }
    __device__ __forceinline__ double scale(int) const { return inv_h; }
};
struct RotAdaptive {
    AdaptiveView av;
    const int *tg, *grp_ptr;
    int grp0;
    __device__ __forceinline__ int target(int g, int i) const {
        const int g0 = grp_ptr[grp0 + g], g1 = grp_ptr[grp0 + g + 1];
        if (!DAFMM_RANGE(g0, g1, av.nbox, kChkListPtr) || i >= g1 - g0) return -1;
        const int t = tg[g0 + i];
        return DAFMM_IN(t, av.nbox, kChkBoxIndex) && DAFMM_IN(av.parent[t], av.nbox, kChkBoxIndex) ? t : -1;
    }
    __device__ __forceinline__ int source(int t, int g, const int (&v)[3]) const {
        const int dx = (g & 1) - v[0], dy = ((g >> 1) & 1) - v[1], dz = ((g >> 2) & 1) - v[2];
        const int Q = av.colleague[27 * (size_t)av.parent[t] + ((dx >> 1) + 1) * 9 + ((dy >> 1) + 1) * 3 + (dz >> 1) + 1];
        if (Q < 0 || !DAFMM_IN(Q, av.nbox, kChkBoxIndex)) return -1;
        const int sb = av.child[8 * (size_t)Q + ((dx & 1) | ((dy & 1) << 1) | ((dz & 1) << 2))];
        return sb >= 0 && DAFMM_IN(sb, av.nbox, kChkBoxIndex) ? sb : -1;
    }
    __device__ __forceinline__ double scale(int t) const { return 1.0 / av.geom[t].w; }  // (each tree has its own)
};

template <class R>
constexpr size_t rot_smem(int nt) {
    return (size_t)8 * nt * 3 * (NCP + 1) * sizeof(R);
}

// L~ = (1/h) sum_v B_v A_|v| F_v M~ for the targets of one octant (blockIdx.y).  A warp takes NT
// targets -- two pairs of one displacement share the table reads and give two chains -- and KS of
// a block's 8 warps share out the displacements of the same targets (every KS-th each, the sums
// joined in that order), so that a level of few boxes still fills the SMs.  The block's warps walk
// the displacements together (a barrier every fourth one), so that the tables of a key, read by
// one of them, serve the others from the L1.
// Measured against one warp per target reading the packed matrices: uniform N = 200,003, depth 4,
// p = 8: FP64 9.7 -> 7.1 ms, float-float 9.7 -> 5.9 ms; N = 1e4, depth 3, p = 6, FP64: 1.84 -> 0.81
// ms; Gaussian N = 100,003, p = 8, FP64 (all levels in one launch): 8.4 -> 2.8 ms.
// MINB: blocks per SM it is compiled for (rot_targets).
template <class R, bool HARM, int NT, int MINB, class Fam>
__global__ void __launch_bounds__(256, MINB)
    k_m2l_rot(RotStream rs, const R* __restrict__ val, const R* __restrict__ ax, const __grid_constant__ Fam fam, RotRows m,
              double* __restrict__ L, int KS) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sub = w % KS, oct = blockIdx.y;  // (adaptive: 8 (level - 2) + octant)
    if (fam.target(oct, (int)blockIdx.x * (8 / KS) * NT) < 0) return;  // beyond this group
    R* base = reinterpret_cast<R*>(smem_raw) + (size_t)w * NT * 3 * (NCP + 1);
    R *X[NT], *Y[NT], *S[NT];
    int t[NT];
#pragma unroll
    for (int u = 0; u < NT; ++u) {
        X[u] = base + u * 3 * (NCP + 1);
        Y[u] = X[u] + NCP + 1;
        S[u] = Y[u] + NCP + 1;
        t[u] = fam.target(oct, ((int)blockIdx.x * (8 / KS) + w / KS) * NT + u);
        for (int k = lane; k <= NCP; k += 32) {
            X[u][k] = rot_zero<R>();  // X[NC], Y[NC]: the zero that padding tasks read
            Y[u][k] = rot_zero<R>();
            S[u][k] = rot_zero<R>();
        }
    }
    const int ox = oct & 1, oy = (oct >> 1) & 1, oz = (oct >> 2) & 1;
    const size_t kstride = (size_t)64 * (rs.lx + rs.lz), astride = (size_t)32 * rs.la;
    int d = 0;
    for (int vx = -3 + ox; vx <= 2 + ox; ++vx)
        for (int vy = -3 + oy; vy <= 2 + oy; ++vy)
            for (int vz = -3 + oz; vz <= 2 + oz; ++vz) {
                if (abs(vx) <= 1 && abs(vy) <= 1 && abs(vz) <= 1) continue;
                const int mine = d++;
                if ((mine & 3) == 0) __syncthreads();
                if (mine % KS != sub) continue;
                const int v[3] = {vx, vy, vz};
                const int key = (vx + 3) * 49 + (vy + 3) * 7 + (vz + 3);
                const R *kv = val + key * kstride, *ka = ax + rs.krho[key] * astride;
                int src[NT], nv = 0;
#pragma unroll
                for (int u = 0; u < NT; ++u) {
                    src[u] = t[u] >= 0 ? fam.source(t[u], oct, v) : -1;
                    nv += src[u] >= 0;
                }
                if (nv == NT) {
                    rot_pairs<HARM, NT, R>(rs, kv, ka, m, src, X, Y, S, lane);
                } else if (nv > 0) {
                    const bool second = src[0] < 0;
                    const int s1[1] = {second ? src[NT - 1] : src[0]};
                    R *const x1[1] = {second ? X[NT - 1] : X[0]}, *const y1[1] = {second ? Y[NT - 1] : Y[0]},
                      *const z1[1] = {second ? S[NT - 1] : S[0]};
                    rot_pairs<HARM, 1, R>(rs, kv, ka, m, s1, x1, y1, z1, lane);
                }
            }
    __syncthreads();
    if (sub != 0) return;
#pragma unroll
    for (int u = 0; u < NT; ++u) {
        if (t[u] < 0) continue;
        const size_t step = (size_t)NT * 3 * (NCP + 1);
        for (int o = 1; o < KS; ++o)
            for (int k = lane; k < NC; k += 32) S[u][k] = rot_add(S[u][k], S[u][k + o * step]);
        __syncwarp();
        if constexpr (HARM) harm_expand_warp(S[u], lane);  // the sums' coefficients of z exponent >= 2
        const double sc = fam.scale(t[u]);
        for (int k = lane; k < NC; k += 32) L[(size_t)t[u] * NCP + k] = rot_to_double(S[u][k]) * sc;
    }
}

// the kernel's table order from the packed matrices: the substitutions' values of every key
// (tasks: x-step then z-step lists, x = offset | last << 31) ...
__global__ void k_rot_pack(const double* __restrict__ T, const uint2* __restrict__ tasks, int lx, int lz,
                           double* __restrict__ val) {
    const int key = blockIdx.x, nx = 32 * lx, nz = 32 * lz;
    const double* Tk = T + (size_t)key * 4 * ROT_TSZ;
    double* out = val + (size_t)key * 2 * (nx + nz);
    for (int e = threadIdx.x; e < nx + nz; e += blockDim.x) {
        const unsigned off = tasks[e].x & 0x7fffffffu;
        if (e < nx) {
            out[e] = Tk[off];
            out[nx + 2 * nz + e] = Tk[3 * ROT_TSZ + off];
        } else {
            out[e] = Tk[ROT_TSZ + off];
            out[nz + e] = Tk[2 * ROT_TSZ + off];
        }
    }
}
// ... and the axial values of every length
__global__ void k_axial_pack(const double* __restrict__ aval, int nnz, const uint2* __restrict__ tasks, int n,
                             double* __restrict__ ax) {
    for (int e = threadIdx.x; e < n; e += blockDim.x)
        ax[(size_t)blockIdx.x * n + e] = aval[(size_t)blockIdx.x * nnz + (tasks[e].x & 0x7fffffffu)];
}

// the float-float split of FP64 rows (n values): hi = fl32(v), lo = fl32(v - hi)
__global__ void k_split_ff(const double* __restrict__ a, float* __restrict__ hi, float* __restrict__ lo, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const ff v(a[i]);
        hi[i] = v.hi;
        lo[i] = v.lo;
    }
}

// float-float copies of the rotation tables and axial values (n doubles each)
__global__ void k_to_ff(const double* __restrict__ a, ff* __restrict__ b, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        b[i] = ff(a[i]);
}

// ---- leaves: P2P over the 27 neighbours + L2P --------------------------------------------------
// 1/sqrt(x) of the PTX instruction rsqrt.approx.ftz.f32 (relative error about 2^-23, the
// size of an FP32 rounding, so no Newton step is needed)
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// the same, and 0 for x below the smallest normal float, which covers coincident points
// (r = 0 contributes nothing, as everywhere else)
__device__ __forceinline__ float rsqrt_or_zero(float x) {
    const float y = rsqrt_approx(x);
    return x >= 1.17549435e-38f ? y : 0.f;
}

// Shared-memory source list of the near field, one segment of kSegPairs pairs of records per
// warp, in the target leaf's frame and negated (a difference is then one addition), as four
// planes of float4 so that a warp stores 32 pairs without bank conflicts:
//   plane 0 (-X, -X', -Y, -Y')  1 (-Z, -Z', Q, Q')    offsets and charges rounded to FP32
//         2 (-x, -x', -y, -y')  3 (-z, -z', q, q')    their FP32 remainders
constexpr int kSegPairs = 64;

// (H, L) = -(hi + lo + d) with the rounding of hi + d moved into L (Fast2Sum: exact when
// |d| >= |hi| or d = 0, which holds for the integer leaf offsets d in {-1, 0, 1} of a uniform
// tree and |hi| <= 1/2)
__device__ __forceinline__ void shift_neg(float hi, float lo, float d, float& H, float& L) {
    H = -hi - d;
    L = (-hi - (H + d)) - lo;
}
// (H, L) = (hi + lo) * r + oh for a power of two r, with the rounding of hi * r + oh moved into L
// (TwoSum: exact for any ordering of the two terms)
__device__ __forceinline__ void scale_shift_exact(float hi, float lo, float r, float oh, float& H, float& L) {
    const float a = hi * r;  // exact
    H = a + oh;
    const float bb = H - a;
    const float err = (a - (H - bb)) + (oh - bb);
    L = fmaf(lo, r, err);
}

// pair `pair` of the records into slot j of the segment, scaled by r and shifted by (ox, oy, oz)
// (UNIT: r = 1 and integer offsets -- the leaves of a uniform tree)
template <bool UNIT>
__device__ __forceinline__ void stage_pair(float4* buf, int j, const float4* __restrict__ xq,
                                           const float4* __restrict__ xl, int pair, float r, float ox, float oy,
                                           float oz) {
    const float4 a = xq[2 * pair], b = xq[2 * pair + 1], c = xl[2 * pair], d = xl[2 * pair + 1];
    float4 A, B, C, D;
    if constexpr (UNIT) {
        shift_neg(a.x, c.x, ox, A.x, C.x);
        shift_neg(a.y, c.y, ox, A.y, C.y);
        shift_neg(a.z, c.z, oy, A.z, C.z);
        shift_neg(a.w, c.w, oy, A.w, C.w);
        shift_neg(b.x, d.x, oz, B.x, D.x);
        shift_neg(b.y, d.y, oz, B.y, D.y);
    } else {
        scale_shift_exact(-a.x, -c.x, r, -ox, A.x, C.x);
        scale_shift_exact(-a.y, -c.y, r, -ox, A.y, C.y);
        scale_shift_exact(-a.z, -c.z, r, -oy, A.z, C.z);
        scale_shift_exact(-a.w, -c.w, r, -oy, A.w, C.w);
        scale_shift_exact(-b.x, -d.x, r, -oz, B.x, D.x);
        scale_shift_exact(-b.y, -d.y, r, -oz, B.y, D.y);
    }
    B.z = b.z;
    B.w = b.w;
    D.z = d.z;
    D.w = d.w;
    buf[j] = A;
    buf[kSegPairs + j] = B;
    buf[2 * kSegPairs + j] = C;
    buf[3 * kSegPairs + j] = D;
}

// the pairs of up to 32 source leaves (lane e: np pairs from pair0, their scale and shift), end to
// end, segment by segment: the warp stages each segment -- every lane finds the leaf of its pair
// in the prefix sums, so that leaves of any size fill the lanes -- and body(first pair, pairs)
// works on it; of NW warps that share a leaf, warp w takes every NW-th segment from the w-th
template <bool UNIT, int NW, class Body>
__device__ __forceinline__ void near_segments(float4* buf, const float4* __restrict__ xq,
                                              const float4* __restrict__ xl, int np, int pair0, float r, float ox,
                                              float oy, float oz, int lane, int warp, Body&& body) {
    int incl = np;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += v;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31), at0 = pair0 - (incl - np);
    for (int seg0 = warp * kSegPairs; seg0 < total; seg0 += NW * kSegPairs) {
        const int segn = min(kSegPairs, total - seg0);
        __syncwarp();  // the previous segment is no longer read
#pragma unroll
        for (int k = 0; k < kSegPairs; k += 32) {
            const int j = seg0 + k + lane;
            int e = 0;  // the first leaf with incl > j
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) {
                const int v = __shfl_sync(0xffffffffu, incl, e + d - 1);
                if (v <= j) e += d;
            }
            const int pair = __shfl_sync(0xffffffffu, at0, e) + j;
            const float er = UNIT ? 1.f : __shfl_sync(0xffffffffu, r, e);
            const float ex = __shfl_sync(0xffffffffu, ox, e), ey = __shfl_sync(0xffffffffu, oy, e),
                        ez = __shfl_sync(0xffffffffu, oz, e);
            if (k + lane < segn) stage_pair<UNIT>(buf, k + lane, xq, xl, pair, er, ex, ey, ez);
        }
        __syncwarp();
        body(seg0, segn);
    }
}

// a pair closer than this (in leaf widths of the target's leaf) takes the remainders of its
// offsets into its difference: beyond it, T - S alone is within a few FP32 roundings of the
// difference's own size (the remainders are below 2^-23 leaf widths)
constexpr float kCloseR2 = 0.01f;

// a target: its offset in the leaf's frame (splat for the packed instructions) and the remainders
struct NearTarget {
    float2 tx, ty, tz;
    float lx, ly, lz;
};
__device__ __forceinline__ NearTarget near_target(const float4* __restrict__ xq, const float4* __restrict__ xl, int r) {
    const float4 t = xq_load(xq, r), l = xq_load(xl, r);
    return NearTarget{make_float2(t.x, t.x), make_float2(t.y, t.y), make_float2(t.z, t.z), l.x, l.y, l.z};
}

// running sums of one target: potential and field (without its sign convention), the two
// sources of a packed instruction separately
struct NearSums {
    float2 P, X, Y, Z;
};

__device__ __forceinline__ float2 splat2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 norm2(float2 ex, float2 ey, float2 ez, float2 r0) {
    return __ffma2_rn(ex, ex, __ffma2_rn(ey, ey, __ffma2_rn(ez, ez, r0)));
}

// the remainders of list pair p in the difference of target t
__device__ __forceinline__ void near_rest(const float4* buf, int p, const NearTarget& t, float2 ex, float2 ey,
                                          float2 ez, float2& fx, float2& fy, float2& fz) {
    const float4 C = buf[2 * kSegPairs + p], D = buf[3 * kSegPairs + p];
    fx = __fadd2_rn(ex, __fadd2_rn(splat2(t.lx), make_float2(C.x, C.y)));
    fy = __fadd2_rn(ey, __fadd2_rn(splat2(t.ly), make_float2(C.z, C.w)));
    fz = __fadd2_rn(ez, __fadd2_rn(splat2(t.lz), make_float2(D.x, D.y)));
}

// a pair closer than 0.1 leaf widths takes the remainders into its difference (halves whose
// r^2 is below kCloseR2; the others keep T - S)
__device__ __forceinline__ void near_close(const float4* buf, int p, const NearTarget& t, float2& ex, float2& ey,
                                           float2& ez, float2& r2) {
    float2 fx, fy, fz;
    near_rest(buf, p, t, ex, ey, ez, fx, fy, fz);
    if (r2.x < kCloseR2) {
        ex.x = fx.x;
        ey.x = fy.x;
        ez.x = fz.x;
    }
    if (r2.y < kCloseR2) {
        ex.y = fx.y;
        ey.y = fy.y;
        ez.y = fz.y;
    }
    r2 = norm2(ex, ey, ez, splat2(1.17549435e-38f));
}

// the pair's terms into the sums
template <bool GUARD>
__device__ __forceinline__ void near_add(float2 ex, float2 ey, float2 ez, float2 r2, float2 q, NearSums& s) {
    const float2 ir = GUARD ? make_float2(rsqrt_or_zero(r2.x), rsqrt_or_zero(r2.y))
                            : make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
    const float2 qr = __fmul2_rn(q, ir);
    const float2 qr3 = __fmul2_rn(qr, __fmul2_rn(ir, ir));
    s.P = __fadd2_rn(s.P, qr);
    s.X = __ffma2_rn(qr3, ex, s.X);
    s.Y = __ffma2_rn(qr3, ey, s.Y);
    s.Z = __ffma2_rn(qr3, ez, s.Z);
}

// List pairs [p0, p1) of the segment acting on this lane's two targets, both sources of a pair in
// one packed FP32x2 instruction: per source
//   e = T - S  (+ (tl - sl) when |e| < 0.1),  r2 = fma(ex, ex, fma(ey, ey, ez ez)),
//   qr = q / r,  qr3 = qr / r^2.
// e carries the difference of the two particles to a few FP32 roundings of itself however close
// they are: pairs closer than 0.1 leaf widths -- rare -- take the remainders, loaded and added only
// in an iteration where a lane of the warp has one.  GUARD (the target's own leaf, which holds the
// target and any coincident particles) always takes them and gives r = 0 no contribution; without
// it r2 starts from the smallest normal float, so distinct particles -- which never coincide
// across leaves -- always give a finite 1/r.  (A null record -- q = 0 at its leaf's centre -- adds
// exactly nothing either way.)
// Two targets per lane: the FP32 pipe needs 26 cycles per packed pair and target, and the two
// 16-byte broadcast loads of a pair return 1 KB to the registers, 8 cycles of the SM's L1 -- 32
// for its four partitions.  With one target per lane the L1 was the bound (ncu: L1 80 % busy, the
// FMA pipe 48 %); two targets halve the loads per interaction.  With the conflict-free staging:
// uniform N = 1e6, p = 8: the kernel 0.80 -> 0.63 ms (5 or 6 blocks per SM; 4: 0.68); clustered
// N = 4e6, p = 10: 10.5 -> 8.1 ms; 64-problem forest, p = 6: 2.74 -> 2.06 ms.  (The adaptive kernel
// compiled for 24 warps per SM instead of 16: 7.4 and 2.04 ms, with one leaf per block 6.7 and 1.88.)
template <bool GUARD>
__device__ __forceinline__ void near_pairs(const float4* buf, int p0, int p1, const NearTarget (&t)[2],
                                           NearSums (&s)[2]) {
#pragma unroll 1
    for (int p = p0; p < p1; ++p) {
        const float4 A = buf[p], B = buf[kSegPairs + p];
        const float2 sx = make_float2(A.x, A.y), sy = make_float2(A.z, A.w), sz = make_float2(B.x, B.y),
                     q = make_float2(B.z, B.w);
        float2 ex[2], ey[2], ez[2], r2[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            ex[u] = __fadd2_rn(t[u].tx, sx);
            ey[u] = __fadd2_rn(t[u].ty, sy);
            ez[u] = __fadd2_rn(t[u].tz, sz);
            if (GUARD) {
                near_rest(buf, p, t[u], ex[u], ey[u], ez[u], ex[u], ey[u], ez[u]);
                r2[u] = __ffma2_rn(ex[u], ex[u], __ffma2_rn(ey[u], ey[u], __fmul2_rn(ez[u], ez[u])));
            } else {
                r2[u] = norm2(ex[u], ey[u], ez[u], splat2(1.17549435e-38f));
            }
        }
        if (!GUARD) {
            const float rmin = fminf(fminf(r2[0].x, r2[0].y), fminf(r2[1].x, r2[1].y));
            if (__any_sync(__activemask(), rmin < kCloseR2)) {
#pragma unroll
                for (int u = 0; u < 2; ++u) near_close(buf, p, t[u], ex[u], ey[u], ez[u], r2[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) near_add<GUARD>(ex[u], ey[u], ez[u], r2[u], q, s[u]);
    }
}

__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float v) {
    const float s = hi + v;
    const float bp = s - hi;
    lo += (hi - (s - bp)) + (v - bp);
    hi = s;
}

// compensated (hi, lo) sums of the near field: FP32 partial sums over at most 128 sources (one
// segment) are folded into them, so that long neighbour lists keep FP32-level error.  Each lane's
// sums for its two targets live in shared memory behind the segment (float [u][8][32]): they are
// touched once per segment, and 16 registers fewer let more warps hide the pair loop's latencies.
struct CompSums {
    float ph = 0.f, pl = 0.f, xh = 0.f, xl = 0.f, yh = 0.f, yl = 0.f, zh = 0.f, zl = 0.f;
};
constexpr int kNearSmem = 4 * kSegPairs + 2 * 8 * 32 / 4;  // float4s per warp: the segment and the sums
__device__ __forceinline__ float* near_acc(float4* buf) { return reinterpret_cast<float*>(buf + 4 * kSegPairs); }

// The lanes of a pass over m <= 32 targets: groups of W lanes, lane l of a group with the targets
// l and l + W, the groups sharing out the sources.  W = 16, 8 or 4, so that a pass costs about
// m / 32 of a full one.
__device__ __forceinline__ int near_width(int m) { return m > 16 ? 16 : (m > 8 ? 8 : 4); }

// the pairwise sums of one segment of n pairs, the first `own` of the target's own leaf (guarded)
__device__ __forceinline__ void near_segment(float4* buf, int n, int own, int W, int lane, const NearTarget (&t)[2]) {
    own = max(0, min(own, n));
    const int lg = __ffs(32 / W) - 1, g = lane / W;  // 2^lg groups
    NearSums s[2] = {};
    if (own > 0) {
        const int h = (own + (1 << lg) - 1) >> lg, pa = min(g * h, own);
        near_pairs<true>(buf, pa, min(pa + h, own), t, s);
    }
    const int h = (n - own + (1 << lg) - 1) >> lg, pa = min(own + g * h, n);
    near_pairs<false>(buf, pa, min(pa + h, n), t, s);
    float* acc = near_acc(buf) + lane;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const float v[4] = {s[u].P.x + s[u].P.y, s[u].X.x + s[u].X.y, s[u].Y.x + s[u].Y.y, s[u].Z.x + s[u].Z.y};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float hi = acc[(u * 8 + 2 * j) * 32], lo = acc[(u * 8 + 2 * j + 1) * 32];
            two_sum_add(hi, lo, v[j]);
            acc[(u * 8 + 2 * j) * 32] = hi;
            acc[(u * 8 + 2 * j + 1) * 32] = lo;
        }
    }
}

__device__ __forceinline__ void near_zero(float4* buf, int lane) {
    float* acc = near_acc(buf) + lane;
#pragma unroll
    for (int j = 0; j < 16; ++j) acc[j * 32] = 0.f;
}

// the sums of target tl < 2 W of the pass over the groups of NW warps (their segments follow one
// another from buf on), in that order
template <int NW>
__device__ __forceinline__ CompSums near_join(float4* buf, int W, int tl) {
    if constexpr (NW > 1) __syncthreads();
    else __syncwarp();
    float k[8] = {};
#pragma unroll 1
    for (int w = 0; w < NW; ++w) {
        const float* acc = near_acc(buf + w * kNearSmem) + (tl >= W ? 8 * 32 : 0) + (tl & (W - 1));
        for (int d = 0; d < 32; d += W) {
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                two_sum_add(k[j], k[j + 1], acc[j * 32 + d]);
                k[j + 1] += acc[(j + 1) * 32 + d];
            }
        }
    }
    // the other lanes' (and warps') sums are read: the next pass may start from zero (near_zero)
    if constexpr (NW > 1) __syncthreads();
    else __syncwarp();
    CompSums r;
    r.ph = k[0]; r.pl = k[1]; r.xh = k[2]; r.xl = k[3]; r.yh = k[4]; r.yl = k[5]; r.zh = k[6]; r.zl = k[7];
    return r;
}

// ---- float-float near field (the DAFMM_FF mode) ----
// a cascaded float-float sum (as Ogita, Rump and Oishi's Sum2): the high parts through TwoSum,
// their rounding errors and the low parts into the low sum; renormalised once, by get()
struct FFCasc {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(ff v) {
        const ff t = two_sum(hi, v.hi);
        hi = t.hi;
        lo += t.lo + v.lo;
    }
    __device__ __forceinline__ ff get() const { return fast_two_sum(hi, lo); }
};
struct FFSums {
    FFCasc p, x, y, z;
};

// the difference (T + tl) - (S + sl) in float-float: TwoSum of the rounded parts (exact), the
// remainders' difference (below 2^-23 leaf widths, one FP32 rounding) added, renormalised
// (the list holds -S and -sl)
__device__ __forceinline__ ff ff_diff(float T, float tl, float nS, float nsl) {
    const ff d = two_sum(T, nS);
    return two_sum(d.hi, d.lo + (tl + nsl));
}

// list records [2 pa, 2 pe) acting on the target t = T + tl, every step in float-float (about
// 48 bits): e as above, r^2 = e.e, 1/r by the Newton-refined float-float 1/sqrt, q (rounded
// charge plus its remainder) / r and q / r^3 into float-float sums.  The records below 2 pown
// are the target's own leaf: a pair at r = 0 (the target itself, coincident particles) adds
// nothing; elsewhere r^2 is kept at least the smallest normal float.
__device__ __forceinline__ void p2p_segment_ff(const float4* __restrict__ buf, int pa, int pe, int pown, float tx,
                                               float ty, float tz, float tlx, float tly, float tlz, FFSums& acc) {
#pragma unroll 1
    for (int p = pa; p < pe; ++p) {
        const float4 A = buf[p], B = buf[kSegPairs + p], C = buf[2 * kSegPairs + p], D = buf[3 * kSegPairs + p];
        const bool own = p < pown;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const ff ex = ff_diff(tx, tlx, h ? A.y : A.x, h ? C.y : C.x);
            const ff ey = ff_diff(ty, tly, h ? A.w : A.z, h ? C.w : C.z);
            const ff ez = ff_diff(tz, tlz, h ? B.y : B.x, h ? D.y : D.x);
            ff r2 = ff_acc(ff_acc(ff_mul(ex, ex), ff_mul(ey, ey)), ff_mul(ez, ez));
            if (own && r2.hi == 0.f) continue;
            r2.hi = fmaxf(r2.hi, 1.17549435e-38f);
            const ff ir = ff_rsqrt(r2);
            const ff qr = ff_mul(ff(h ? B.w : B.z, h ? D.w : D.z), ir);
            const ff qr3 = ff_mul(qr, ff_mul(ir, ir));
            acc.p.add(qr);
            acc.x.add(ff_mul(qr3, ex));
            acc.y.add(ff_mul(qr3, ey));
            acc.z.add(ff_mul(qr3, ez));
        }
    }
}

__device__ __forceinline__ ff ff_shfl_down(ff v, int d) {
    return ff(__shfl_down_sync(0xffffffffu, v.hi, d), __shfl_down_sync(0xffffffffu, v.lo, d));
}

// The uniform FP32 leaf kernel: a block per leaf -- a block of four leaves holds its registers until
// its longest leaf is done -- compiled for 28 warps per SM.  N = 1e6, p = 8: 0.63 ms with four
// leaves per block at 20 warps per SM, 0.61 with one, 0.60 with the sums in shared memory at 28
// warps.  (More warps or independent pairs in flight do not help further, nor do scalar field
// sums, although a packed FMA of three distinct registers takes 3.9 cycles in a loop of its own
// and two scalar ones 2.3: 0.61-0.62 ms.)  A tree of few leaves gives each 8 warps, which share
// out the segments of its source list (leaf_warps): 64 leaves, N = 3001, p = 4: 91 -> 24 us.
constexpr int kLeafMinWarps = 28;

// ---- FP64 near field ----
// 1/sqrt(x) for x well inside the normal range: the PTX approximation y (rsqrt.approx.ftz.f64, which works on
// the upper 32 bits of x and fills those of y: 20 explicit significand bits) and the binomial series of
// (1 - e)^(-1/2) in its residual e = 1 - x y^2 up to e^2: five FP64 instructions.  y y is exact, so that e
// carries no error to speak of, and with a seed good to 2^-19 (the two truncations leave 2^-21 + 2^-20;
// PTX states no bound) |e| <= 2^-18 and the first term left out is 5/16 e^3 <= 5/32 2^-53 of the result.  Measured
// on 300,000 arguments over the whole range: at most 1.003 2^-53 (one rounding alone: 1), every result
// equal to CUDA's rsqrt.
__device__ __forceinline__ double rsqrt_series(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y * y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}

struct Sum64 {
    double p = 0.0, x = 0.0, y = 0.0, z = 0.0;
};
__device__ __forceinline__ Sum64 sum64_shfl(const Sum64& s, int d) {
    Sum64 r;
    r.p = s.p + __shfl_xor_sync(0xffffffffu, s.p, d);
    r.x = s.x + __shfl_xor_sync(0xffffffffu, s.x, d);
    r.y = s.y + __shfl_xor_sync(0xffffffffu, s.y, d);
    r.z = s.z + __shfl_xor_sync(0xffffffffu, s.z, d);
    return r;
}

// targets of the next pass over `rem` particles: 32 lanes, or the largest power of two that they
// fill (or fill to four fifths), the sources shared out over the 32 / W groups of lanes
__device__ __forceinline__ int pass_width(int rem) {
    if (rem >= 32) return 32;
    const int w = 1 << (31 - __clz(rem));
    return 5 * rem >= 8 * w ? 2 * w : w;
}

// The particles of up to 32 source leaves (lane e: cnt particles from `first`), end to end, every
// G-th from the g-th, on one target.  The FP64 pipe (1/64 of the FP32 rate on this part) is the
// bound, so everything else is spent to feed it: every lane has a target or a share of the
// sources (the list position of a source is a search in the prefix sums), 1/r takes five FP64
// instructions, and a pair takes 18 (20 with CUDA's rsqrt and an FP64 comparison).  r^2 outside
// the series' window (2^-991 to 2^977) is seen in the exponent by an integer comparison: positive it takes
// CUDA's rsqrt (an infinite one adds 1/inf = 0); zero -- the target itself and coincident particles --
// and NaN add nothing.
__device__ __forceinline__ void near64_list(const double* __restrict__ x, const double* __restrict__ y,
                                            const double* __restrict__ z, const double* __restrict__ q, int cnt,
                                            int first, int G, int g, int lane, double xt, double yt, double zt,
                                            Sum64& s) {
    int incl = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += v;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31), at0 = first - (incl - cnt);
#pragma unroll 2
    for (int j0 = 0; j0 < total; j0 += G) {
        const int j = j0 + g;
        int e = 0;  // the first leaf with incl > j
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const int v = __shfl_sync(0xffffffffu, incl, e + d - 1);
            if (v <= j) e += d;
        }
        const int i = __shfl_sync(0xffffffffu, at0, e) + j;
        if (j >= total) continue;
        const double ex = xt - x[i], ey = yt - y[i], ez = zt - z[i];
        const double r2 = fma(ez, ez, fma(ey, ey, ex * ex));
        double ir;
        if ((unsigned)__double2hiint(r2) - 0x02000000u < 0x7b000000u) ir = rsqrt_series(r2);
        else if (r2 > 0.0) ir = rsqrt(r2);
        else continue;
        const double qr = q[i] * ir, w = qr * (ir * ir);
        s.p += qr;
        s.x = fma(w, ex, s.x);
        s.y = fma(w, ey, s.y);
        s.z = fma(w, ez, s.z);
    }
}

// the sums of a pass: over the lanes' groups, then over the block's NW warps (red: two buffers in
// turn, so that one barrier per pass does); warp 0 has the result
template <int NW>
__device__ __forceinline__ Sum64 pass_join(Sum64 s, int W, int warp, int lane, Sum64 (*red)[NW][32], int& turn) {
    for (int d = W; d < 32; d <<= 1) s = sum64_shfl(s, d);
    if constexpr (NW > 1) {
        red[turn][warp][lane] = s;
        __syncthreads();
        if (warp == 0) {
            for (int v = 1; v < NW; ++v) {
                const Sum64 o = red[turn][v][lane];
                s.p += o.p;
                s.x += o.x;
                s.y += o.y;
                s.z += o.z;
            }
        }
        turn ^= 1;
    }
    return s;
}

// the neighbour slot (0..26, slot 13 = the leaf itself) held by lane k of the list: the leaf
// itself first, so that its records -- the only ones that can coincide with a target -- form
// the guarded head of the list
__device__ __forceinline__ int own_first_slot(int k) { return k == 0 ? 13 : (k <= 13 ? k - 1 : k); }

template <class T, int NW>
constexpr size_t leaf_smem() {  // the warps' segments and sums, and the leaf's local expansion
    return (size_t)NW * kNearSmem * sizeof(float4) + NCP * sizeof(T);
}

template <class T, int NW>
__global__ void __launch_bounds__(32 * NW, (std::is_same<T, float>::value ? kLeafMinWarps : 16) / NW)
    k_leaf(TreeView tv, const double* __restrict__ Lleaf, double* __restrict__ phi, double* __restrict__ field) {
    static_assert(NW == 1 || std::is_same<T, float>::value, "float-float: one warp per leaf");
    extern __shared__ __align__(16) float4 s_near[];
    T* lrow = reinterpret_cast<T*>(s_near + NW * kNearSmem);
    const int lane = threadIdx.x, warp = NW > 1 ? threadIdx.y : 0, leaf = blockIdx.x;
    float4* buf = s_near + warp * kNearSmem;
    int i0 = tv.leaf_start[leaf], i1 = tv.leaf_start[leaf + 1];
    if (!DAFMM_RANGE(i0, i1, tv.n, kChkLeafRange)) i0 = i1 = 0;
    int a, b, c;
    octmajor_decode(tv.depth, leaf, a, b, c);
    const int nside = 1 << tv.depth;
    const double cx = tv.x0 + ((double)a + 0.5) * tv.h_leaf;
    const double cy = tv.y0 + ((double)b + 0.5) * tv.h_leaf;
    const double cz = tv.z0 + ((double)c + 0.5) * tv.h_leaf;
    const double* Lrow = Lleaf ? Lleaf + (size_t)leaf * NCP : nullptr;
    if (Lrow && warp == 0) {  // the leaf's local expansion, in T (FP32 rows: NCP floats per leaf)
        const float* Lf = reinterpret_cast<const float*>(Lleaf) + (size_t)leaf * NCP;
        for (int k = lane; k < NC; k += 32) {
            if constexpr (std::is_same<T, float>::value) lrow[k] = tv.locals_f32 ? Lf[k] : (float)Lrow[k];
            else lrow[k] = ff(Lrow[k]);
        }
        __syncwarp();
    }
    // FP32: the 27 neighbour leaves, one per lane (none outside the domain): their pairs of
    // records -- an odd leaf's last pair ends in its null record -- and their offsets in leaf
    // widths; the leaf itself first (lane 0), its pairs the guarded head of the list
    int nb_np = 0, nb_pair = 0, own_pairs = 0;
    float nb_x = 0.f, nb_y = 0.f, nb_z = 0.f;
    {
        if (lane < 27) {
            const int slot = own_first_slot(lane);
            const int dx = slot % 3 - 1, dy = (slot / 3) % 3 - 1, dz = slot / 9 - 1;
            const int na = a + dx, nb = b + dy, nc2 = c + dz;
            if (na >= 0 && nb >= 0 && nc2 >= 0 && na < nside && nb < nside && nc2 < nside) {
                const int nl = octmajor_index(tv.depth, na, nb, nc2);
                int nb_s0 = tv.leaf_start[nl], nb_s1 = tv.leaf_start[nl + 1];
                if (!DAFMM_RANGE(nb_s0, nb_s1, tv.n, kChkLeafRange)) nb_s0 = nb_s1 = 0;
                nb_pair = xq_base(nb_s0, nl) >> 1;
                nb_np = (nb_s1 - nb_s0 + 1) >> 1;
                nb_x = (float)dx;
                nb_y = (float)dy;
                nb_z = (float)dz;
            }
        }
        own_pairs = __shfl_sync(0xffffffffu, nb_np, 0);
    }
    const int r_own = xq_base(i0, leaf) - i0;  // record of sorted position t: t + r_own
    for (int base = i0; base < i1; base += 32) {
        const int m = min(32, i1 - base);
        // float-float: a pass of at most 16 targets splits the sources between the two half-warps,
        // lane l and lane l + 16 taking the same target; FP32: see near_width
        const bool split = std::is_same<T, ff>::value && m <= 16;
        const int W = near_width(m);
        const int per = std::is_same<T, float>::value ? 2 * W : (split ? 16 : 32);
        const int tl = lane & (per - 1);
        const int t = base + tl;
        const bool valid = tl < m && lane < per;  // the lanes that write
        const int tt = tl < m ? t : i0;
        double fphi = 0.0, fx = 0.0, fy = 0.0, fz = 0.0;  // near field, physical units
        {
            const float4* xl = tv.xq + xq_records(tv.n, tv.nleaf);  // the remainder records
            // The neighbours' records are copied into one shared-memory list, shifted into this
            // leaf's frame (source + neighbour offset, in leaf widths, exactly: the rounding of
            // the shift joins the remainder); the pairwise sum runs over each segment of it.
            CompSums sum;
            FFSums fs;
            if constexpr (std::is_same<T, float>::value) {
                near_zero(buf, lane);
                const int l0 = lane & (W - 1);
                const NearTarget nt[2] = {near_target(tv.xq, xl, (l0 < m ? base + l0 : i0) + r_own),
                                          near_target(tv.xq, xl, (l0 + W < m ? base + l0 + W : i0) + r_own)};
                near_segments<true, NW>(buf, tv.xq, xl, nb_np, nb_pair, 1.f, nb_x, nb_y, nb_z, lane, warp,
                                        [&](int seg0, int n) { near_segment(buf, n, own_pairs - seg0, W, lane, nt); });
                sum = near_join<NW>(s_near, W, tl);
                if (warp != 0) continue;
            } else {
                const float4 pt = xq_load(tv.xq, tt + r_own), pl = xq_load(xl, tt + r_own);
                near_segments<true, 1>(buf, tv.xq, xl, nb_np, nb_pair, 1.f, nb_x, nb_y, nb_z, lane, 0, [&](int seg0, int n) {
                    const int h = split ? (n + 1) >> 1 : n, g = split ? lane >> 4 : 0;
                    p2p_segment_ff(buf, g ? h : 0, g ? n : h, own_pairs - seg0, pt.x, pt.y, pt.z, pl.x, pl.y, pl.z, fs);
                });
            }
            const double ih = tv.inv_h_leaf, ih2 = ih * ih;
            if constexpr (std::is_same<T, float>::value) {
                fphi = ((double)sum.ph + (double)sum.pl) * ih;
                fx = ((double)sum.xh + (double)sum.xl) * ih2;
                fy = ((double)sum.yh + (double)sum.yl) * ih2;
                fz = ((double)sum.zh + (double)sum.zl) * ih2;
            } else {
                ff sp = fs.p.get(), sx = fs.x.get(), sy = fs.y.get(), sz = fs.z.get();
                if (split) {  // the upper half-warp's sums join the lower one's
                    sp = ff_add(sp, ff_shfl_down(sp, 16));
                    sx = ff_add(sx, ff_shfl_down(sx, 16));
                    sy = ff_add(sy, ff_shfl_down(sy, 16));
                    sz = ff_add(sz, ff_shfl_down(sz, 16));
                }
                fphi = sp.to_double() * ih;
                fx = sx.to_double() * ih2;
                fy = sy.to_double() * ih2;
                fz = sz.to_double() * ih2;
            }
        }
        // far field from the leaf's local expansion
        if (Lrow) {
            T F, g0, g1, g2;
            T xs, ys, zs;
            if constexpr (sizeof(T) == 8) {
                xs = (T)((tv.x[tt] - cx) * tv.inv_h_leaf);
                ys = (T)((tv.y[tt] - cy) * tv.inv_h_leaf);
                zs = (T)((tv.z[tt] - cz) * tv.inv_h_leaf);
            } else {
                const float4 pt = xq_load(tv.xq, tt + r_own);
                xs = (T)pt.x; ys = (T)pt.y; zs = (T)pt.z;
            }
            if constexpr (sizeof(T) == 4) gen::GEN(l2p)<T>(SmemRowF{lrow}, xs, ys, zs, F, g0, g1, g2);
            else gen::GEN(l2p)<T>(SmemRowFF{lrow}, xs, ys, zs, F, g0, g1, g2);
            fphi += (double)F;
            fx -= (double)g0 * tv.inv_h_leaf;
            fy -= (double)g1 * tv.inv_h_leaf;
            fz -= (double)g2 * tv.inv_h_leaf;
        }
        if (valid && DAFMM_IN(tv.perm[t], tv.n, kChkPerm)) {
            const int o = tv.perm[t];
            if (phi) phi[o] = fphi;
            if (field) {
                field[3 * (size_t)o] = fx;
                field[3 * (size_t)o + 1] = fy;
                field[3 * (size_t)o + 2] = fz;
            }
        }
    }
}

// The same in FP64: a block of NW warps per leaf, the warps sharing out the sources of each pass.
// NW is 8 or 1 (leaf_warps), so that a tree of 64 or 512 leaves still gives every SM its share.
// Measured against one warp per leaf with passes of 32 and CUDA's rsqrt: uniform N = 200,003, depth 4,
// p = 8: 13.1 -> 9.6 ms; N = 1e4, depth 3, p = 6: the evaluation 2.57 -> 2.20 ms (this kernel 0.28).
template <int NW>
__global__ void __launch_bounds__(32 * NW, 24 / NW) k_leaf64(TreeView tv, const double* __restrict__ Lleaf,
                                                             double* __restrict__ phi, double* __restrict__ field) {
    __shared__ Sum64 red[2][NW][32];
    const int lane = threadIdx.x, warp = threadIdx.y, leaf = blockIdx.x;
    int i0 = tv.leaf_start[leaf], i1 = tv.leaf_start[leaf + 1];
    if (!DAFMM_RANGE(i0, i1, tv.n, kChkLeafRange)) i0 = i1 = 0;
    int a, b, c;
    octmajor_decode(tv.depth, leaf, a, b, c);
    const int nside = 1 << tv.depth;
    const double cx = tv.x0 + ((double)a + 0.5) * tv.h_leaf;
    const double cy = tv.y0 + ((double)b + 0.5) * tv.h_leaf;
    const double cz = tv.z0 + ((double)c + 0.5) * tv.h_leaf;
    // the 27 neighbour leaves, one per lane (none outside the domain)
    int cnt = 0, first = 0;
    if (lane < 27) {
        const int na = a + lane % 3 - 1, nb = b + (lane / 3) % 3 - 1, nc2 = c + lane / 9 - 1;
        if (na >= 0 && nb >= 0 && nc2 >= 0 && na < nside && nb < nside && nc2 < nside) {
            const int nl = octmajor_index(tv.depth, na, nb, nc2);
            int s0 = tv.leaf_start[nl], s1 = tv.leaf_start[nl + 1];
            if (!DAFMM_RANGE(s0, s1, tv.n, kChkLeafRange)) s0 = s1 = 0;
            first = s0;
            cnt = s1 - s0;
        }
    }
    int turn = 0;
    for (int base = i0, W; base < i1; base += W) {
        W = pass_width(i1 - base);
        const int t = base + (lane & (W - 1)), tt = t < i1 ? t : i0;
        const double xt = tv.x[tt], yt = tv.y[tt], zt = tv.z[tt];
        Sum64 s;
        near64_list(tv.x, tv.y, tv.z, tv.q, cnt, first, NW * (32 / W), warp * (32 / W) + lane / W, lane, xt, yt, zt, s);
        s = pass_join<NW>(s, W, warp, lane, red, turn);
        if (warp != 0) continue;
        if (Lleaf) {  // far field from the leaf's local expansion
            double F, g0, g1, g2;
            gen::GEN(l2p)<double>(RowLoad<double>{Lleaf + (size_t)leaf * NCP}, (xt - cx) * tv.inv_h_leaf,
                                  (yt - cy) * tv.inv_h_leaf, (zt - cz) * tv.inv_h_leaf, F, g0, g1, g2);
            s.p += F;
            s.x -= g0 * tv.inv_h_leaf;
            s.y -= g1 * tv.inv_h_leaf;
            s.z -= g2 * tv.inv_h_leaf;
        }
        if (lane < W && t < i1 && DAFMM_IN(tv.perm[t], tv.n, kChkPerm)) {
            const size_t o = (size_t)tv.perm[t];
            if (phi) phi[o] = s.p;
            if (field) {
                field[3 * o] = s.x;
                field[3 * o + 1] = s.y;
                field[3 * o + 2] = s.z;
            }
        }
    }
}

// ---- adaptive trees ---------------------------------------------------------------------------
// Box geometry of an adaptive box (centre and width, precomputed per box at build time).
__device__ __forceinline__ void abox_geom(const AdaptiveView& av, int b, double& cx, double& cy, double& cz,
                                          double& h) {
    const double4 g = av.geom[b];
    cx = g.x;
    cy = g.y;
    cz = g.z;
    h = g.w;
}

// P2M (Eq. 2) at the leaves listed in `leaves`: one warp per leaf, as in k_p2m (H: the
// harmonic basis's free coefficients only, written at their layout positions)
template <class T, bool H = false>
__global__ void k_p2m_a(AdaptiveView av, const int* __restrict__ leaves, int nleaves, double* __restrict__ M) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw) + threadIdx.y * (32 * 33);
    const int lane = threadIdx.x;
    const int li = blockIdx.x * blockDim.y + threadIdx.y;
    if (li >= nleaves) return;
    const int b = leaves[li];
    if (!DAFMM_IN(b, av.nbox, kChkBoxIndex)) return;
    double cx, cy, cz, h;
    abox_geom(av, b, cx, cy, cz, h);
    const double ih = 1.0 / h;
    int i0 = av.pbeg[b], i1 = av.pend[b];
    if (!DAFMM_RANGE(i0, i1, av.n, kChkBoxRange)) i0 = i1 = 0;
    if constexpr (sizeof(T) == 4) {  // the leaf's records
        if (!DAFMM_RANGE(av.xq0[b], (long long)av.xq0[b] + (i1 - i0), av.nrec, kChkRecord)) i0 = i1 = 0;
    }
    constexpr int NO = H ? nharm_of(P) : NC;
    constexpr int NJ = (NO + 31) / 32;
    T acc[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[j] = T(0);
    ChunkSink<T, NJ, NO> sink{sm, lane, acc};
    for (int base = i0; base < i1; base += 32) {
        const int i = base + lane;
        T x = T(0), y = T(0), z = T(0), q = T(0);
        if (i < i1) {
            if constexpr (sizeof(T) == 4) {
                // the particle's FP32 record: its offset from this leaf's centre in leaf widths
                // (what the FP64 form computes, rounded once) and its charge, without FP64
                // instructions (1/64 of the FP32 rate on this part)
                const float4 r = xq_load(av.xq, av.xq0[b] + (i - i0));
                x = r.x;
                y = r.y;
                z = r.z;
                q = r.w;
            } else {
                x = (T)((av.x[i] - cx) * ih);
                y = (T)((av.y[i] - cy) * ih);
                z = (T)((av.z[i] - cz) * ih);
                q = (T)av.q[i];
            }
        }
        if constexpr (H) gen::GEN(p2mh)<T>(x, y, z, q, sink);
        else gen::GEN(p2m)<T>(x, y, z, q, sink);
    }
    if constexpr (H && sizeof(T) == 8) {
        p2m_row(acc, sm, M + (size_t)b * NCP, lane);
        return;
    }
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = lane + 32 * j;
        if (k < NO) M[(size_t)b * NCP + (H ? harm_full_index(k) : k)] = (double)acc[j];
    }
}

// M2L (Eq. 5) into the boxes tg[0..ntg) of one level that share the octant `oct`; the source
// of displacement v is child sc of the parent's colleague at offset a (c - v = 2a + sc)
template <class T, class Src>
__global__ void __launch_bounds__(256) k_m2l_a(const T* __restrict__ K, AdaptiveView av, const int* __restrict__ tg,
                                               const int* __restrict__ grp_ptr, int grp0, const Src* __restrict__ M,
                                               double* __restrict__ L) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* src = reinterpret_cast<T*>(smem_raw);  // [32][NCP + 1]
    __shared__ int sidx[32];
    const int oct = blockIdx.y;
    int g0 = grp_ptr[grp0 + oct], g1 = grp_ptr[grp0 + oct + 1];
    if (!DAFMM_RANGE(g0, g1, av.nbox, kChkListPtr)) g0 = g1 = 0;
    const int t0 = g0 + blockIdx.x * 32;
    if (t0 >= g1) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ox = oct & 1, oy = (oct >> 1) & 1, oz = (oct >> 2) & 1;
    T acc[SH_ROWS];
#pragma unroll
    for (int j = 0; j < SH_ROWS; ++j) acc[j] = T(0);
    for (int vx = -3 + ox; vx <= 2 + ox; ++vx)
        for (int vy = -3 + oy; vy <= 2 + oy; ++vy)
            for (int vz = -3 + oz; vz <= 2 + oz; ++vz) {
                if (abs(vx) <= 1 && abs(vy) <= 1 && abs(vz) <= 1) continue;
                if (threadIdx.x < 32) {
                    const int ti = t0 + threadIdx.x;
                    int sbox = -1;
                    if (ti < g1 && DAFMM_IN(tg[ti], av.nbox, kChkBoxIndex) &&
                        DAFMM_IN(av.parent[tg[ti]], av.nbox, kChkBoxIndex)) {
                        const int P = av.parent[tg[ti]];
                        const int dx = ox - vx, dy = oy - vy, dz = oz - vz;  // = 2a + sc
                        const int scx = dx & 1, scy = dy & 1, scz = dz & 1;
                        const int ax = (dx - scx) >> 1, ay = (dy - scy) >> 1, az = (dz - scz) >> 1;
                        const int Q = av.colleague[27 * (size_t)P + (ax + 1) * 9 + (ay + 1) * 3 + (az + 1)];
                        if (Q >= 0 && DAFMM_IN(Q, av.nbox, kChkBoxIndex))
                            sbox = av.child[8 * (size_t)Q + (scx | (scy << 1) | (scz << 2))];
                        if (sbox >= 0 && !DAFMM_IN(sbox, av.nbox, kChkBoxIndex)) sbox = -1;
                    }
                    sidx[threadIdx.x] = sbox;
                }
                __syncthreads();
                for (int e = threadIdx.x; e < 32 * NC; e += 256) {
                    const int r = e / NC, k = e - r * NC;
                    const int sb = sidx[r];
                    src[r * (NCP + 1) + k] = sb >= 0 ? (T)M[(size_t)sb * NCP + k] : T(0);
                }
                __syncthreads();
                const int key = (vx + 3) * 49 + (vy + 3) * 7 + (vz + 3);
                const T* Kv = K + (size_t)key * NC * NCP;
                const T* srow = src + lane * (NCP + 1);
                const T* kw = Kv + (size_t)w * NCP;
#pragma unroll 1
                for (int a = 0; a < NC; ++a) {
                    const T sv = srow[a];
#pragma unroll
                    for (int j = 0; j < SH_ROWS; ++j)
                        if (w + 8 * j < NC) acc[j] = fma(kw[(size_t)(8 * j) * NCP + a], sv, acc[j]);
                }
                __syncthreads();
            }
    const int ti = t0 + lane;
    if (ti < g1 && DAFMM_IN(tg[ti], av.nbox, kChkBoxIndex)) {
        const int t = tg[ti];
        const double inv_h = 1.0 / av.geom[t].w;  // the target box's width (each tree has its own)
#pragma unroll
        for (int j = 0; j < SH_ROWS; ++j) {
            const int b = w + 8 * j;
            if (b < NC) L[(size_t)t * NCP + b] = (double)acc[j] * inv_h;
        }
    }
}

// P2L (Eq. 6): particles of the X-list leaves of each box of [lb, le) into its local expansion,
// one warp per box, all levels in one launch.
//   1 / |w + d| = |w|^-1 (1 - 2 s.d + s^2 d^2)^(-1/2) with s = -w / |w|^2, so the P2L of w is the
// generated P2M (Eq. 2) of s with the charge q / |w|; and since a local expansion is harmonic,
// only its (p + 1)^2 free coefficients are generated and summed (121 instead of 286 at p = 10),
// the others restored once per box by Laplace's equation.  The X lists' particles are taken as
// one sequence -- 32 list entries at a time, prefix sums over the lanes -- so that every lane has
// a particle whatever the leaves' sizes.  FP32: the source's offset in this box's frame comes
// from its record (hi + lo) and the exact integer offset of the two boxes, rounded once to FP32,
// as the FP64 difference was, but without FP64 instructions (they ran at 69 % of the FP64 pipe,
// 1/64 of the FP32 rate, and bound the kernel).
// Measured against the full-basis form before (one launch per level, a leaf at a time, FP64
// differences): 64-problem forest, p = 6 (FP32): 0.913 -> 0.296 ms; Gaussian N = 1e6, p = 4 (FP32):
// 0.444 -> 0.159 ms; Gaussian N = 1e5, s = 256, p = 8 (FP64): 9.89 -> 2.44 ms.
template <class T>
__global__ void __launch_bounds__(128) k_p2l_a(AdaptiveView av, int lb, int le, double* __restrict__ L) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw) + threadIdx.y * (32 * 33);
    static_assert(NCP <= 32 * 33, "the staging block holds a row");
    const int lane = threadIdx.x;
    const int b = lb + blockIdx.x * blockDim.y + threadIdx.y;
    if (b >= le) return;
    int x0i = av.x_ptr[b], x1i = av.x_ptr[b + 1];
    if (!DAFMM_RANGE(x0i, x1i, av.nx, kChkListPtr)) x0i = x1i = 0;
    if (x0i == x1i) return;
    double cx, cy, cz, h;
    abox_geom(av, b, cx, cy, cz, h);
    const double ih = 1.0 / h;
    const int lev = av.level[b];
    const int* ib = av.ijk + 3 * (size_t)b;
    constexpr int NO = nharm_of(P);
    constexpr int NJ = (NO + 31) / 32;
    T acc[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[j] = T(0);
    ChunkSink<T, NJ, NO> sink{sm, lane, acc};
    for (int xg = x0i; xg < x1i; xg += 32) {
        // one list entry per lane: its particles (FP32: its first record, its centre offset and
        // width in this box's widths), and the inclusive prefix sum of the counts
        int cnt = 0, first = 0;
        float r = 1.f, ox = 0.f, oy = 0.f, oz = 0.f;
        if (xg + lane < x1i) {
            const int c = av.x_idx[xg + lane];
            if (DAFMM_IN(c, av.nbox, kChkBoxIndex) && DAFMM_RANGE(av.pbeg[c], av.pend[c], av.n, kChkBoxRange)) {
                first = av.pbeg[c];
                cnt = av.pend[c] - first;
                if constexpr (sizeof(T) == 4) {
                    first = av.xq0[c];
                    if (!DAFMM_RANGE(first, (long long)first + cnt, av.nrec, kChkRecord)) cnt = 0;
                    const int d = lev - av.level[c];  // > 0: the leaves of an X list are coarser
                    const int* ic = av.ijk + 3 * (size_t)c;
                    r = __int_as_float((127 + d) << 23);
                    ox = 0.5f * (float)(((2 * ic[0] + 1) << d) - (2 * ib[0] + 1));
                    oy = 0.5f * (float)(((2 * ic[1] + 1) << d) - (2 * ib[1] + 1));
                    oz = 0.5f * (float)(((2 * ic[2] + 1) << d) - (2 * ib[2] + 1));
                }
            }
        }
        int incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += v;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        for (int base = 0; base < total; base += 32) {
            const int j = base + lane;
            int e = 0;  // the entry that holds particle j: the first with incl > j
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) {
                const int v = __shfl_sync(0xffffffffu, incl, e + d - 1);
                if (v <= j) e += d;
            }
            const int i = __shfl_sync(0xffffffffu, first - (incl - cnt), e) + j;
            T X = T(1), Y = T(0), Z = T(0), q = T(0);  // a dummy far point for idle lanes
            if constexpr (sizeof(T) == 4) {
                const float er = __shfl_sync(0xffffffffu, r, e), ex = __shfl_sync(0xffffffffu, ox, e),
                            ey = __shfl_sync(0xffffffffu, oy, e), ez = __shfl_sync(0xffffffffu, oz, e);
                if (j < total) {
                    const float4 rec = xq_load(av.xq, i), rl = xq_load(av.xl, i);
                    float lx, ly, lz;
                    scale_shift_exact(rec.x, rl.x, er, ex, X, lx);
                    scale_shift_exact(rec.y, rl.y, er, ey, Y, ly);
                    scale_shift_exact(rec.z, rl.z, er, ez, Z, lz);
                    X += lx;
                    Y += ly;
                    Z += lz;
                    q = rec.w;
                }
            } else if (j < total) {
                X = (av.x[i] - cx) * ih;
                Y = (av.y[i] - cy) * ih;
                Z = (av.z[i] - cz) * ih;
                q = av.q[i];
            }
            // w = -(X, Y, Z); s = -w / |w|^2
            const T ir = dafmm_rsqrt(X * X + Y * Y + Z * Z), rho = ir * ir;
            gen::GEN(p2mh)<T>(X * rho, Y * rho, Z * rho, q * ir, sink);
        }
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = lane + 32 * j;
        if (k < NO) sm[harm_full_index(k)] = acc[j];
    }
    __syncwarp();
    harm_expand_warp(sm, lane);
    for (int k = lane; k < NC; k += 32) L[(size_t)b * NCP + k] += (double)sm[k] * ih;
}

// per warp of the FP32 adaptive leaf kernel: the source list's segment (the M2P stages up to two
// W boxes' multipoles in it afterwards), then the leaf's locals in FP32
constexpr size_t kLeafWarpSmem = kNearSmem * sizeof(float4) + NCP * sizeof(float);
static_assert(2 * NCP * sizeof(float) <= 4 * kSegPairs * sizeof(float4), "two rows fit the segment");

// leaves: P2P over the U list, M2P over the W list, L2P of the leaf's local expansion (FP32)
// One warp per leaf, and one leaf per block unless the context says otherwise: the leaves' lists differ
// in length, and a block holds its place on the SM until its longest leaf is done (with four leaves
// 4.0 of the 6 warps per scheduler were there on average).  Four leaves per block against one:
// clustered N = 4e6, p = 10: 7.46 -> 6.72 ms; 64-problem forest, p = 6: 2.02 -> 1.88 ms; Gaussian
// N = 1e6, p = 4: 1.52 -> 1.49 ms.  Compiled for 16 or 32 warps per SM instead of 24: 7.88 and 6.73,
// 2.16 and 2.02, 1.64 and 1.59 ms.
// Block (.., y) takes every gridDim.y-th pass of its leaves from the y-th on (leaf_a_split).
__global__ void __launch_bounds__(256, 3) k_leaf_a(AdaptiveView av, const int* __restrict__ leaves, int nleaves,
                                                   const double* __restrict__ L, const double* __restrict__ M,
                                                   const float* __restrict__ Mf, double* __restrict__ phi,
                                                   double* __restrict__ field) {
    extern __shared__ __align__(16) unsigned char s_leaf[];
    const int lane = threadIdx.x;
    const int li = blockIdx.x * blockDim.y + threadIdx.y;
    if (li >= nleaves) return;
    float4* buf = reinterpret_cast<float4*>(s_leaf + threadIdx.y * kLeafWarpSmem);
    float* lrow = reinterpret_cast<float*>(buf + kNearSmem);
    const int b = leaves[li];
    if (!DAFMM_IN(b, av.nbox, kChkBoxIndex)) return;
    double cx, cy, cz, h;
    abox_geom(av, b, cx, cy, cz, h);
    const double ih = 1.0 / h;
    const int lev = av.level[b];
    if (lev >= 2) warp_row_to_f32(L + (size_t)b * NCP, lrow, lane);
    int i0 = av.pbeg[b], i1 = av.pend[b];
    if (!DAFMM_RANGE(i0, i1, av.n, kChkBoxRange)) i0 = i1 = 0;
    // the leaf's own records (its targets)
    if (!DAFMM_RANGE(av.xq0[b], (long long)av.xq0[b] + (i1 - i0), av.nrec, kChkRecord)) i0 = i1 = 0;
    const int base0 = i0 + 32 * (int)blockIdx.y;
    if (base0 >= i1) return;
    int u0 = av.u_ptr[b], u1 = av.u_ptr[b + 1];
    int w0 = av.w_ptr[b], w1 = av.w_ptr[b + 1];
    if (!DAFMM_RANGE(u0, u1, av.nu, kChkListPtr)) u0 = u1 = 0;
    if (!DAFMM_RANGE(w0, w1, av.nw, kChkListPtr)) w0 = w1 = 0;
    for (int base = base0; base < i1; base += 32 * gridDim.y) {
        const int m = min(32, i1 - base);
        const int W = near_width(m), per = 2 * W;  // the lanes' split, see near_width
        const int tl = lane & (per - 1);
        const int t = base + tl;
        const bool valid = tl < m && lane < per;  // the lanes that write
        const int tt = tl < m ? t : i0;
        double fphi = 0.0, fx = 0.0, fy = 0.0, fz = 0.0;
        {
            // The U-list leaves' records are copied into one shared-memory list in this leaf's
            // frame (source x h_s / h + centre offset / h, exactly: h_s / h is a power of two and
            // the rounding of the sum joins the remainder), 32 leaves at a time; the list begins
            // with the leaf itself (the only records that can coincide with a target).
            const int l0 = lane & (W - 1), rb = av.xq0[b] - i0;
            const NearTarget nt[2] = {near_target(av.xq, av.xl, (l0 < m ? base + l0 : i0) + rb),
                                      near_target(av.xq, av.xl, (l0 + W < m ? base + l0 + W : i0) + rb)};
            near_zero(buf, lane);  // sums in leaf widths of this leaf
            const int* ijk_b = av.ijk + 3 * (size_t)b;
            for (int ug = u0; ug < u1; ug += 32) {
                int np = 0, pair = 0;
                float r = 1.f, ox = 0.f, oy = 0.f, oz = 0.f;
                const int sb = ug + lane < u1 ? av.u_idx[ug + lane] : -1;
                if (sb >= 0 && DAFMM_IN(sb, av.nbox, kChkBoxIndex) &&
                    DAFMM_RANGE(av.pbeg[sb], av.pend[sb], av.n, kChkBoxRange) &&
                    DAFMM_RANGE(av.xq0[sb], (long long)av.xq0[sb] + (av.pend[sb] - av.pbeg[sb]), av.nrec, kChkRecord)) {
                    pair = av.xq0[sb] >> 1;
                    np = (av.pend[sb] - av.pbeg[sb] + 1) >> 1;
                    // the source leaf's centre offset in this leaf's widths and its width ratio,
                    // from the integer box coordinates (same tree): with d = lev_b - lev_s,
                    // (c_s - c_b) / h_b = N / 2^(1 + max(0, -d)),
                    // N = (2 i_s + 1) 2^max(0, d) - (2 i_b + 1) 2^max(0, -d).  Levels go to 20, so
                    // both terms stay below 2^22, and adjacent boxes have |N| <= 2^|d| + 1 < 2^24:
                    // N is exact in an int and in a float.  (64-bit N took nine conversions per
                    // list entry on the FP64 pipe, 1/64 of the FP32 rate here: 35 % of that
                    // pipe's cycles, Gaussian N = 1e6, p = 4: the kernel 2.28 -> 1.73 ms, FP32
                    // results unchanged bit for bit.)
                    const int d = lev - av.level[sb];
                    const int up = d > 0 ? d : 0, dn = d < 0 ? -d : 0;
                    r = __int_as_float((127 + d) << 23);                      // h_s / h_b = 2^d
                    const float sc = __int_as_float((127 - 1 - dn) << 23);    // 2^-(1 + dn)
                    const int* ijk_s = av.ijk + 3 * (size_t)sb;
                    ox = (float)(((2 * ijk_s[0] + 1) << up) - ((2 * ijk_b[0] + 1) << dn)) * sc;
                    oy = (float)(((2 * ijk_s[1] + 1) << up) - ((2 * ijk_b[1] + 1) << dn)) * sc;
                    oz = (float)(((2 * ijk_s[2] + 1) << up) - ((2 * ijk_b[2] + 1) << dn)) * sc;
                }
                const int own = ug == u0 ? (i1 - i0 + 1) >> 1 : 0;
                near_segments<false, 1>(buf, av.xq, av.xl, np, pair, r, ox, oy, oz, lane, 0,
                                        [&](int seg0, int n) { near_segment(buf, n, own - seg0, W, lane, nt); });
            }
            const CompSums sum = near_join<1>(buf, W, tl);
            fphi = ((double)sum.ph + (double)sum.pl) * ih;
            fx = ((double)sum.xh + (double)sum.xl) * ih * ih;
            fy = ((double)sum.yh + (double)sum.yl) * ih * ih;
            fz = ((double)sum.zh + (double)sum.zl) * ih * ih;
        }
        // M2P from the W list (Sec. 3.2): phi = F/h_w, E = -grad_s F / h_w^2
        {
            // FP32, without FP64 instructions (this part runs FP64 at 1/64 of the FP32 rate): the
            // W box is finer than the leaf by dl levels of the same tree, so with integer box
            // coordinates i at each level (c_b - c_w) / h_w = ((2 i_b + 1) 2^dl - (2 i_w + 1)) / 2
            // per axis, exactly; the target in the W box's frame is its leaf-frame offset (record
            // and remainder) times 2^dl plus that; the box's multipoles come as FP32 rows (Mf).
            // Its terms are summed in FP32 and join the FP64 sums once per target.
            const float4 pw = xq_load(av.xq, av.xq0[b] + (tt - i0)), plw = xq_load(av.xl, av.xq0[b] + (tt - i0));
            const float ihf = (float)ih;
            float wphi = 0.f, wfx = 0.f, wfy = 0.f, wfz = 0.f;
            const int* ib = av.ijk + 3 * (size_t)b;
            // a pass of at most 16 targets works on two W boxes at a time
            const int two = per < 32 ? 2 : 1, rep = two == 2 ? (lane / per) & 1 : 0;
            float* mrow = reinterpret_cast<float*>(buf) + rep * NCP;
            for (int wi = w0; wi < w1; wi += two) {
                __syncwarp();  // the list and the previous boxes are no longer read
                for (int e = 0; e < two; ++e) {
                    const int eb = wi + e < w1 ? av.w_idx[wi + e] : -1;
                    if (eb < 0 || !DAFMM_IN(eb, av.nbox, kChkBoxIndex)) continue;
                    float* row = reinterpret_cast<float*>(buf) + e * NCP;
                    for (int k = lane; k < NC; k += 32)
                        row[k] = Mf ? Mf[(size_t)eb * NCP + k] : (float)M[(size_t)eb * NCP + k];
                }
                __syncwarp();
                const int wb = wi + rep < w1 ? av.w_idx[wi + rep] : -1;
                if (wb < 0 || !DAFMM_IN(wb, av.nbox, kChkBoxIndex)) continue;
                const int dl = av.level[wb] - lev;
                // (finer boxes of the same tree, levels up to 20: both terms below 2^22, exact)
                const float r = __int_as_float((127 + dl) << 23);
                const int* iwb = av.ijk + 3 * (size_t)wb;
                const float ox = 0.5f * (float)(((2 * ib[0] + 1) << dl) - (2 * iwb[0] + 1));
                const float oy = 0.5f * (float)(((2 * ib[1] + 1) << dl) - (2 * iwb[1] + 1));
                const float oz = 0.5f * (float)(((2 * ib[2] + 1) << dl) - (2 * iwb[2] + 1));
                const float sx0 = fmaf(plw.x, r, fmaf(pw.x, r, ox));
                const float sy0 = fmaf(plw.y, r, fmaf(pw.y, r, oy));
                const float sz0 = fmaf(plw.z, r, fmaf(pw.z, r, oz));
                const float iw = ihf * r;
                float F, g0, g1, g2;
                gen::GEN(m2p)<float>(SmemRowF{mrow}, sx0, sy0, sz0, F, g0, g1, g2);
                wphi = fmaf(F, iw, wphi);
                const float iw2 = iw * iw;
                wfx = fmaf(-g0, iw2, wfx);
                wfy = fmaf(-g1, iw2, wfy);
                wfz = fmaf(-g2, iw2, wfz);
            }
            if (two == 2) {
                __syncwarp();
                wphi += __shfl_xor_sync(0xffffffffu, wphi, per);
                wfx += __shfl_xor_sync(0xffffffffu, wfx, per);
                wfy += __shfl_xor_sync(0xffffffffu, wfy, per);
                wfz += __shfl_xor_sync(0xffffffffu, wfz, per);
            }
            fphi += (double)wphi;
            fx += (double)wfx;
            fy += (double)wfy;
            fz += (double)wfz;
        }
        // L2P of this leaf's local expansion
        if (lev >= 2) {
            float F, g0, g1, g2;
            const float4 pt = xq_load(av.xq, av.xq0[b] + (tt - i0));
            gen::GEN(l2p)<float>(SmemRowF{lrow}, pt.x, pt.y, pt.z, F, g0, g1, g2);
            fphi += (double)F;
            fx -= (double)g0 * ih;
            fy -= (double)g1 * ih;
            fz -= (double)g2 * ih;
        }
        if (valid && DAFMM_IN(av.perm[t], av.n, kChkPerm)) {
            const int o = av.perm[t];
            if (phi) phi[o] = fphi;
            if (field) {
                field[3 * (size_t)o] = fx;
                field[3 * (size_t)o + 1] = fy;
                field[3 * (size_t)o + 2] = fz;
            }
        }
    }
}

// The same in FP64: a block of kLeaf64Warps warps per leaf and every blockIdx.y-th of its passes;
// the warps share out the U-list sources and the W boxes of a pass.  How a leaf's sums are split
// depends on the leaf and its lists alone (a member of a forest sums as the same tree built
// alone).  Measured against one warp per leaf with passes of 32 and CUDA's rsqrt: Gaussian
// N = 100,003, s = 256, p = 8: 37.4 -> 10.1 ms (the few largest leaves held the others up).
constexpr int kLeaf64Warps = 4;
__global__ void __launch_bounds__(32 * kLeaf64Warps, 4)
    k_leaf64_a(AdaptiveView av, const int* __restrict__ leaves, const double* __restrict__ L,
               const double* __restrict__ M, double* __restrict__ phi, double* __restrict__ field) {
    constexpr int NW = kLeaf64Warps;
    __shared__ Sum64 red[2][NW][32];
    const int lane = threadIdx.x, warp = threadIdx.y;
    const int b = leaves[blockIdx.x];
    if (!DAFMM_IN(b, av.nbox, kChkBoxIndex)) return;
    int i0 = av.pbeg[b], i1 = av.pend[b];
    if (!DAFMM_RANGE(i0, i1, av.n, kChkBoxRange)) i0 = i1 = 0;
    int u0 = av.u_ptr[b], u1 = av.u_ptr[b + 1];
    int w0 = av.w_ptr[b], w1 = av.w_ptr[b + 1];
    if (!DAFMM_RANGE(u0, u1, av.nu, kChkListPtr)) u0 = u1 = 0;
    if (!DAFMM_RANGE(w0, w1, av.nw, kChkListPtr)) w0 = w1 = 0;
    int turn = 0, pass = 0;
    for (int base = i0, W; base < i1; base += W, ++pass) {
        W = pass_width(i1 - base);
        if (pass % gridDim.y != blockIdx.y) continue;
        const int G = NW * (32 / W), g = warp * (32 / W) + lane / W;
        const int t = base + (lane & (W - 1)), tt = t < i1 ? t : i0;
        const double xt = av.x[tt], yt = av.y[tt], zt = av.z[tt];
        Sum64 s;
        for (int ug = u0; ug < u1; ug += 32) {
            int cnt = 0, first = 0;
            const int sb = ug + lane < u1 ? av.u_idx[ug + lane] : -1;
            if (sb >= 0 && DAFMM_IN(sb, av.nbox, kChkBoxIndex) &&
                DAFMM_RANGE(av.pbeg[sb], av.pend[sb], av.n, kChkBoxRange)) {
                first = av.pbeg[sb];
                cnt = av.pend[sb] - first;
            }
            near64_list(av.x, av.y, av.z, av.q, cnt, first, G, g, lane, xt, yt, zt, s);
        }
        // M2P from the W list (Sec. 3.2): phi = F / h_w, E = -grad_s F / h_w^2
        for (int wi = w0 + g; wi < w1; wi += G) {
            const int wb = av.w_idx[wi];
            if (!DAFMM_IN(wb, av.nbox, kChkBoxIndex)) continue;
            double wx, wy, wz, wh;
            abox_geom(av, wb, wx, wy, wz, wh);
            const double iwh = 1.0 / wh;
            double F, g0, g1, g2;
            gen::GEN(m2p)<double>(RowLoad<double>{M + (size_t)wb * NCP}, (xt - wx) * iwh, (yt - wy) * iwh,
                                  (zt - wz) * iwh, F, g0, g1, g2);
            s.p += F * iwh;
            s.x -= g0 * iwh * iwh;
            s.y -= g1 * iwh * iwh;
            s.z -= g2 * iwh * iwh;
        }
        __syncwarp();
        s = pass_join<NW>(s, W, warp, lane, red, turn);
        if (warp != 0) continue;
        if (av.level[b] >= 2) {  // L2P of this leaf's local expansion
            double cx, cy, cz, h;
            abox_geom(av, b, cx, cy, cz, h);
            const double ih = 1.0 / h;
            double F, g0, g1, g2;
            gen::GEN(l2p)<double>(RowLoad<double>{L + (size_t)b * NCP}, (xt - cx) * ih, (yt - cy) * ih, (zt - cz) * ih,
                                  F, g0, g1, g2);
            s.p += F;
            s.x -= g0 * ih;
            s.y -= g1 * ih;
            s.z -= g2 * ih;
        }
        if (lane < W && t < i1 && DAFMM_IN(av.perm[t], av.n, kChkPerm)) {
            const size_t o = (size_t)av.perm[t];
            if (phi) phi[o] = s.p;
            if (field) {
                field[3 * o] = s.x;
                field[3 * o + 1] = s.y;
                field[3 * o + 2] = s.z;
            }
        }
    }
}

// ---- single-operator batches ------------------------------------------------------------------
template <class T>
struct RowStore {
    double* o;
    __device__ __forceinline__ void operator()(int k, T v) const { o[k] = (double)v; }
};

template <class T>
__global__ void k_op_p2m(int64_t n, const double* __restrict__ s, const double* __restrict__ q, double* out) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    gen::GEN(p2m)<T>((T)s[3 * i], (T)s[3 * i + 1], (T)s[3 * i + 2], (T)q[i], RowStore<T>{out + i * NC});
}
template <class T>
__global__ void k_op_p2l(int64_t n, const double* __restrict__ w, const double* __restrict__ q, double* out) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    gen::GEN(p2l)<T>((T)w[3 * i], (T)w[3 * i + 1], (T)w[3 * i + 2], (T)q[i], RowStore<T>{out + i * NC});
}
template <class T, bool M2P>
__global__ void k_op_eval(int64_t n, const double* __restrict__ C, const double* __restrict__ x, double* out4) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    T F, g0, g1, g2;
    if (M2P) gen::GEN(m2p)<T>(RowLoad<T>{C + i * NC}, (T)x[3 * i], (T)x[3 * i + 1], (T)x[3 * i + 2], F, g0, g1, g2);
    else gen::GEN(l2p)<T>(RowLoad<T>{C + i * NC}, (T)x[3 * i], (T)x[3 * i + 1], (T)x[3 * i + 2], F, g0, g1, g2);
    out4[4 * i] = (double)F;
    out4[4 * i + 1] = (double)g0;
    out4[4 * i + 2] = (double)g1;
    out4[4 * i + 3] = (double)g2;
}
template <class T>
__global__ void k_op_shift(ShiftTab tab, int64_t n, const int* __restrict__ oct, const double* __restrict__ in,
                           double* out) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = oct[i] & 7;
    for (int b = 0; b < NC; ++b) {
        T s = T(0);
        for (int e = tab.rowptr[b]; e < tab.rowptr[b + 1]; ++e) {
            T v = tab_val<T>(tab, e);
            if (__popc(tab.par[e] & c) & 1) v = -v;
            s += v * (T)in[i * NC + tab.col[e]];
        }
        out[i * NC + b] = (double)s;
    }
}

// ---- launchers ---------------------------------------------------------------------------------
template <class K>
static cudaError_t set_smem(K kernel, size_t bytes) {
    if (bytes > 48 * 1024) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    return cudaSuccess;
}

static cudaError_t p2m_launch(const TreeView& tv, int prec, double* M, const F16Rows* f16, cudaStream_t s) {
    if (tv.nleaf == 0) return cudaSuccess;
    const F16Rows fr = f16 ? *f16 : F16Rows{};
    const int rows32 = (prec & kRowsF32) ? 1 : 0;
    const bool harm = (prec & kRowsHarm) != 0;
    prec &= ~(kRowsF32 | kRowsHarm);
    const bool f64 = prec == DAFMM_FP64, fff = prec == DAFMM_FF;
    if (harm && (f64 || fff)) return cudaErrorInvalidValue;  // (the FP32 kernel only)
    // the fused F16 split: FP32 harmonic rows, every padded row position held by the warp
    if (fr.hi && (!harm || !rows32 || !fr.lo || !fr.inv || fr.rowlen < nharm_of(P) ||
                  fr.rowlen > 32 * ((nharm_of(P) + 31) / 32)))
        return cudaErrorInvalidValue;
    const size_t per_warp = (size_t)32 * 33 * (f64 || fff ? 8 : 4);
    int wpb = (int)((96 * 1024) / per_warp);
    wpb = wpb < 1 ? 1 : (wpb > 4 ? 4 : wpb);
    const size_t smem = per_warp * wpb;
    dim3 blk(32, wpb), grd((tv.nleaf + wpb - 1) / wpb);
    cudaError_t e;
    if (f64) {
        if ((e = set_smem(k_p2m<double, true>, smem)) != cudaSuccess) return e;
        k_p2m<double, true><<<grd, blk, smem, s>>>(tv, M, 0, F16Rows{});
    } else if (fff) {
        if ((e = set_smem(k_p2m<ff, true>, smem)) != cudaSuccess) return e;
        k_p2m<ff, true><<<grd, blk, smem, s>>>(tv, M, 0, F16Rows{});
    } else if (harm) {
        if ((e = set_smem(k_p2m<float, true>, smem)) != cudaSuccess) return e;
        k_p2m<float, true><<<grd, blk, smem, s>>>(tv, M, rows32, fr);
    } else {
        if ((e = set_smem(k_p2m<float>, smem)) != cudaSuccess) return e;
        k_p2m<float><<<grd, blk, smem, s>>>(tv, M, rows32, F16Rows{});
    }
    return cudaGetLastError();
}

template <class T, bool H, class Fam>
static cudaError_t m2m_run(const ShiftTab& tab, const Fam& fam, const double* Mc, double* Mp, int rows32,
                           cudaStream_t s) {
    const size_t smem = m2m_smem<T, H>(H ? tab.nnz : 0);
    const cudaError_t e = set_smem(k_m2m<T, H, Fam>, smem);
    if (e != cudaSuccess) return e;
    k_m2m<T, H, Fam><<<(fam.n + kM2MParents - 1) / kM2MParents, 256, smem, s>>>(tab, fam, Mc, Mp, rows32);
    return cudaGetLastError();
}

template <class Fam>
static cudaError_t m2m_any(const OrderData& od, int prec, const Fam& fam, const double* Mc, double* Mp,
                           cudaStream_t s) {
    const int rows32 = (prec & kRowsF32) ? 1 : 0;
    const bool harm = (prec & kRowsHarm) != 0;
    prec &= ~(kRowsF32 | kRowsHarm);
    if (harm && (prec == DAFMM_FP64 || prec == DAFMM_FF || !od.m2mh_rowptr)) return cudaErrorInvalidValue;
    if (prec != DAFMM_FP32)
        return harm ? m2m_run<double, true>(od.m2mh(), fam, Mc, Mp, 0, s)
                    : m2m_run<double, false>(od.m2m(), fam, Mc, Mp, 0, s);
    return harm ? m2m_run<float, true>(od.m2mh(), fam, Mc, Mp, rows32, s)
                : m2m_run<float, false>(od.m2m(), fam, Mc, Mp, rows32, s);
}

static cudaError_t m2m_launch(const OrderData& od, int prec, int lc, const double* Mc, double* Mp,
                              cudaStream_t s) {
    return m2m_any(od, prec, ShiftUniform{lc, 1 << (3 * (lc - 1))}, Mc, Mp, s);
}

// most table entries in one block's rows of the L2L
static int l2l_max_entries() {
    int mx = 1;
    for (int b = 0; b < NC; b += kL2LRows) {
        const int e = b + kL2LRows < NC ? b + kL2LRows : NC;
        const int n = gen::GENT(l2l, _rowptr)[e] - gen::GENT(l2l, _rowptr)[b];
        if (n > mx) mx = n;
    }
    return mx;
}

template <class T, class Fam>
static cudaError_t l2l_run(const ShiftTab& tab, const Fam& fam, const double* Lp, double* Lc, cudaStream_t s) {
    static const int maxe = (l2l_max_entries() + 3) & ~3;
    const size_t smem = l2l_smem<T>(maxe);
    const cudaError_t e = set_smem(k_l2l<T, Fam>, smem);
    if (e != cudaSuccess) return e;
    const dim3 grd((fam.n + 31) / 32, (NC + kL2LRows - 1) / kL2LRows);
    k_l2l<T, Fam><<<grd, 32 * kL2LRows, smem, s>>>(tab, fam, maxe, Lp, Lc);
    return cudaGetLastError();
}

static cudaError_t l2l_launch(const OrderData& od, int prec, int lc, const double* Lp, double* Lc,
                              cudaStream_t s) {
    const ShiftUniform fam{lc, 1 << (3 * (lc - 1))};
    return prec == DAFMM_FP32 ? l2l_run<float>(od.l2l(), fam, Lp, Lc, s) : l2l_run<double>(od.l2l(), fam, Lp, Lc, s);
}

static cudaError_t m2l_launch(const OrderData& od, int prec, int l, const double* M, const float* Mf,
                              double* L, double inv_h, cudaStream_t s) {
    const int Pp = 1 << (l - 1);
    const int nlin = Pp * Pp * Pp;
    dim3 grd((nlin + 31) / 32, 8);
    cudaError_t e;
    if (prec == DAFMM_FP64) {
        const size_t smem = (size_t)32 * (NCP + 1) * 8;
        if ((e = set_smem(k_m2l<double, double>, smem)) != cudaSuccess) return e;
        k_m2l<double, double><<<grd, 256, smem, s>>>(od.K64, l, M, L, inv_h);
    } else {
        const size_t smem = (size_t)32 * (NCP + 1) * 4;
        if ((e = set_smem(k_m2l<float, float>, smem)) != cudaSuccess) return e;
        k_m2l<float, float><<<grd, 256, smem, s>>>(od.K32, l, Mf, L, inv_h);
    }
    return cudaGetLastError();
}

template <class T, int NW>
static cudaError_t leaf_run(const TreeView& tv, const double* Lleaf, double* phi, double* field, cudaStream_t s) {
    const cudaError_t e = set_smem(k_leaf<T, NW>, leaf_smem<T, NW>());
    if (e != cudaSuccess) return e;
    k_leaf<T, NW><<<tv.nleaf, dim3(32, NW), leaf_smem<T, NW>(), s>>>(tv, Lleaf, phi, field);
    return cudaGetLastError();
}

static cudaError_t leaf_launch(const TreeView& tv, int prec, const double* Lleaf, double* phi, double* field,
                               cudaStream_t s) {
    if (tv.nleaf == 0) return cudaSuccess;
    if (prec == DAFMM_FF) return leaf_run<ff, 1>(tv, Lleaf, phi, field, s);
    const bool f64 = prec == DAFMM_FP64;
    const bool shared = leaf_warps(tv.nleaf, tv.n, f64) > 1;
    if (!f64) return shared ? leaf_run<float, kLeafWarps>(tv, Lleaf, phi, field, s) : leaf_run<float, 1>(tv, Lleaf, phi, field, s);
    if (shared) k_leaf64<kLeafWarps><<<tv.nleaf, dim3(32, kLeafWarps), 0, s>>>(tv, Lleaf, phi, field);
    else k_leaf64<1><<<tv.nleaf, dim3(32, 1), 0, s>>>(tv, Lleaf, phi, field);
    return cudaGetLastError();
}

// M2L by rotation: the tables of a form, harmonic (free outputs only) or full
static RotStream rot_stream(const OrderData& od, bool harm) {
    const RotForm& f = od.rot[harm];
    return RotStream{f.idx, f.lx, f.lz, f.la, od.rot_rho};
}

// targets: the most in one group (octant); groups: blockIdx.y
template <class R, bool HARM, int NT, int MINB = 2, class Fam>
static cudaError_t rot_run(const OrderData& od, const R* val, const R* ax, const Fam& fam, const RotRows& m, double* L,
                           int targets, int groups, int KS, cudaStream_t s) {
    const size_t smem = rot_smem<R>(NT);
    const cudaError_t e = set_smem(k_m2l_rot<R, HARM, NT, MINB, Fam>, smem);
    if (e != cudaSuccess) return e;
    const int per = NT * (8 / KS);
    k_m2l_rot<R, HARM, NT, MINB, Fam>
        <<<dim3((targets + per - 1) / per, groups), 256, smem, s>>>(rot_stream(od, HARM), val, ax, fam, m, L, KS);
    return cudaGetLastError();
}

// a uniform level (rot_targets, rot_share)
template <class R>
static cudaError_t rot_uniform(const OrderData& od, const R* val, const R* ax, int l, const RotRows& m, double* L,
                               double inv_h, bool harm, cudaStream_t s) {
    const int nbox = 1 << (3 * l), per = nbox / 8, nt = rot_targets(nbox, harm, std::is_same<R, double>::value);
    const RotUniform fam{l, inv_h};
    const int KS = rot_share(nbox, nt);
    if (!harm) return rot_run<R, false, 1>(od, val, ax, fam, m, L, per, 8, KS, s);
    if (nt == 2) return rot_run<R, true, 2>(od, val, ax, fam, m, L, per, 8, KS, s);
    if constexpr (std::is_same<R, double>::value) {
        if (KS == 1) return rot_run<R, true, 1, 4>(od, val, ax, fam, m, L, per, 8, KS, s);
    }
    return rot_run<R, true, 1>(od, val, ax, fam, m, L, per, 8, KS, s);
}

static cudaError_t m2l_rot_launch(const OrderData& od, int l, const double* M, double* L, double inv_h, bool harm,
                                  cudaStream_t s) {
    return rot_uniform<double>(od, od.rot[harm].val, od.rot[harm].ax, l, RotRows{M, nullptr, nullptr}, L, inv_h, harm, s);
}

// the same in float-float (DAFMM_FF): the source rows' FP32 parts Mh, Ml (k_split_ff)
static cudaError_t m2l_rot_ff_launch(const OrderData& od, int l, const float* Mh, const float* Ml, double* L,
                                     double inv_h, bool harm, cudaStream_t s) {
    return rot_uniform<ff>(od, reinterpret_cast<const ff*>(od.rot[harm].valf), reinterpret_cast<const ff*>(od.rot[harm].axf),
                           l, RotRows{nullptr, Mh, Ml}, L, inv_h, harm, s);
}

// the kernel's tables of a form; tasks: its x-step, z-step and axial lists end to end
static cudaError_t rot_pack_launch(const OrderData& od, const RotForm& f, const uint2* tasks, cudaStream_t s) {
    k_rot_pack<<<kNumKeys, 128, 0, s>>>(od.rot_T, tasks, f.lx, f.lz, f.val);
    k_axial_pack<<<od.n_rho, 128, 0, s>>>(od.ax_val, od.ax_nnz, tasks + 32 * (f.lx + f.lz), 32 * f.la, f.ax);
    return cudaGetLastError();
}

static cudaError_t split_ff_launch(const double* a, float* hi, float* lo, size_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const size_t blocks = (n + 255) / 256;
    k_split_ff<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, s>>>(a, hi, lo, n);
    return cudaGetLastError();
}

static cudaError_t to_ff_launch(const double* a, float2* b, size_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const size_t blocks = (n + 255) / 256;
    k_to_ff<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, s>>>(a, reinterpret_cast<ff*>(b), n);
    return cudaGetLastError();
}

// the rotation tables of all keys and the axial matrices of the nrho lengths in r0s (3 per
// length, along x); Kscratch holds nrho dense matrices
static cudaError_t rot_setup_launch(OrderData& od, const double* r0s, int nrho, double* Kscratch, cudaStream_t s) {
    k_kgen<<<nrho, 256, 0, s>>>(od.mul(), Kscratch, nullptr, -1, nullptr, r0s);
    k_axial_gather<<<nrho, 256, 0, s>>>(Kscratch, od.ax_rowptr, od.ax_col, od.ax_nnz, od.ax_val);
    k_rot_tables<<<kNumKeys, 128, 0, s>>>(od.rot_T);
    return cudaGetLastError();
}

// the matrices of the given keys (all keys when key_list is null)
static cudaError_t kgen_launch(OrderData& od, const short* key_list, int nkeys, cudaStream_t s) {
    if (nkeys <= 0) return cudaSuccess;
    k_kgen<<<key_list ? nkeys : kNumKeys, 256, 0, s>>>(od.mul(), od.K64, od.K32, -1, key_list, nullptr);
    return cudaGetLastError();
}

// ---- adaptive launchers ----
static cudaError_t p2m_a_launch(const AdaptiveView& av, const int* leaves, int nleaves, int prec, double* M,
                                cudaStream_t s) {
    if (nleaves == 0) return cudaSuccess;
    const bool harm = (prec & kRowsHarm) != 0;
    prec &= ~kRowsHarm;
    const bool f64 = prec == DAFMM_FP64;
    if (harm && (f64 || prec == DAFMM_FF)) return cudaErrorInvalidValue;  // (the FP32 kernel only)
    const size_t per_warp = (size_t)32 * 33 * (f64 ? 8 : 4);
    int wpb = (int)((96 * 1024) / per_warp);
    wpb = wpb < 1 ? 1 : (wpb > 4 ? 4 : wpb);
    const size_t smem = per_warp * wpb;
    dim3 blk(32, wpb), grd((nleaves + wpb - 1) / wpb);
    cudaError_t e;
    if (f64) {
        if ((e = set_smem(k_p2m_a<double, true>, smem)) != cudaSuccess) return e;
        k_p2m_a<double, true><<<grd, blk, smem, s>>>(av, leaves, nleaves, M);
    } else if (harm) {
        if ((e = set_smem(k_p2m_a<float, true>, smem)) != cudaSuccess) return e;
        k_p2m_a<float, true><<<grd, blk, smem, s>>>(av, leaves, nleaves, M);
    } else {
        if ((e = set_smem(k_p2m_a<float>, smem)) != cudaSuccess) return e;
        k_p2m_a<float><<<grd, blk, smem, s>>>(av, leaves, nleaves, M);
    }
    return cudaGetLastError();
}

static cudaError_t m2m_a_launch(const OrderData& od, const AdaptiveView& av, int prec, const int* parents, int np,
                                double* M, cudaStream_t s) {
    if (np <= 0) return cudaSuccess;
    return m2m_any(od, prec, ShiftAdaptive{av, parents, np}, M, M, s);
}

static cudaError_t m2l_a_launch(const OrderData& od, const AdaptiveView& av, int prec, const int* tg,
                                const int* grp_ptr, int grp0, int ngrp, int max_group, const double* M,
                                const float* Mf, double* L, cudaStream_t s) {
    if (max_group == 0) return cudaSuccess;
    if (prec & kM2LRot) {  // FP64 by rotation (Sec. 3.4), ngrp groups from grp0 in one launch
        // (two warps per pair of targets whatever their number: a member of a forest sums as alone)
        const bool harm = (prec & kM2LHarm) != 0;
        const RotAdaptive fam{av, tg, grp_ptr, grp0};
        const RotRows m{M, nullptr, nullptr};
        const RotForm& f = od.rot[harm];
        if (harm) return rot_run<double, true, 2>(od, f.val, f.ax, fam, m, L, max_group, ngrp, 2, s);
        return rot_run<double, false, 1>(od, f.val, f.ax, fam, m, L, max_group, ngrp, 2, s);
    }
    dim3 grd((max_group + 31) / 32, 8);
    cudaError_t e;
    if (prec == DAFMM_FP64) {
        const size_t smem = (size_t)32 * (NCP + 1) * 8;
        if ((e = set_smem(k_m2l_a<double, double>, smem)) != cudaSuccess) return e;
        k_m2l_a<double, double><<<grd, 256, smem, s>>>(od.K64, av, tg, grp_ptr, grp0, M, L);
    } else {
        const size_t smem = (size_t)32 * (NCP + 1) * 4;
        if ((e = set_smem(k_m2l_a<float, float>, smem)) != cudaSuccess) return e;
        k_m2l_a<float, float><<<grd, 256, smem, s>>>(od.K32, av, tg, grp_ptr, grp0, Mf, L);
    }
    return cudaGetLastError();
}

static cudaError_t p2l_a_launch(const AdaptiveView& av, int prec, int lb, int le, double* L, cudaStream_t s) {
    if (le <= lb) return cudaSuccess;
    const bool f64 = prec == DAFMM_FP64;
    const size_t per_warp = (size_t)32 * 33 * (f64 ? 8 : 4);
    // FP64: a box per block, as the X lists differ and a block stays until its longest is done
    // (Gaussian N = 1e5, s = 256, p = 8: 2.90 ms with four warps, 2.68 with two, 2.44 with one); FP32
    // does not care (clustered N = 4e6, p = 10: 2.44, 2.43 and 2.44 ms) and keeps the fewer blocks
    const int wpb = f64 ? 1 : 4;
    const size_t smem = per_warp * wpb;
    dim3 blk(32, wpb), grd((le - lb + wpb - 1) / wpb);
    cudaError_t e;
    if (f64) {
        if ((e = set_smem(k_p2l_a<double>, smem)) != cudaSuccess) return e;
        k_p2l_a<double><<<grd, blk, smem, s>>>(av, lb, le, L);
    } else {
        if ((e = set_smem(k_p2l_a<float>, smem)) != cudaSuccess) return e;
        k_p2l_a<float><<<grd, blk, smem, s>>>(av, lb, le, L);
    }
    return cudaGetLastError();
}

static cudaError_t l2l_a_launch(const OrderData& od, const AdaptiveView& av, int prec, const int* parents, int np,
                                double* L, cudaStream_t s) {
    if (np <= 0) return cudaSuccess;
    const ShiftAdaptive fam{av, parents, np};
    return prec == DAFMM_FP32 ? l2l_run<float>(od.l2l(), fam, L, L, s) : l2l_run<double>(od.l2l(), fam, L, L, s);
}

static cudaError_t leaf_a_launch(const AdaptiveView& av, const int* leaves, int nleaves, int prec, const double* L,
                                 const double* M, const float* Mf, double* phi, double* field, int warps,
                                 int max_leaf, cudaStream_t s) {
    if (nleaves == 0) return cudaSuccess;
    warps = warps < 1 ? 1 : (warps > 8 ? 8 : warps);
    dim3 blk(32, warps), grd((nleaves + warps - 1) / warps, leaf_a_split(nleaves, max_leaf));
    if (prec == DAFMM_FP64) {
        // blocks per leaf: one per pass of the largest leaf, up to 8
        const int ny = max_leaf < 32 ? 1 : (max_leaf > 8 * 32 ? 8 : (max_leaf + 31) / 32);
        k_leaf64_a<<<dim3(nleaves, ny), dim3(32, kLeaf64Warps), 0, s>>>(av, leaves, L, M, phi, field);
    } else {
        const size_t smem = (size_t)warps * kLeafWarpSmem;
        cudaError_t e = cudaFuncSetAttribute(k_leaf_a, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_leaf_a<<<grd, blk, smem, s>>>(av, leaves, nleaves, L, M, Mf, phi, field);
    }
    return cudaGetLastError();
}

static unsigned nblk(int64_t n) { return (unsigned)((n + 127) / 128); }

static cudaError_t op_p2m(int prec, int64_t n, const double* sv, const double* q, double* out, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (prec == DAFMM_FP64) k_op_p2m<double><<<nblk(n), 128, 0, s>>>(n, sv, q, out);
    else k_op_p2m<float><<<nblk(n), 128, 0, s>>>(n, sv, q, out);
    return cudaGetLastError();
}
static cudaError_t op_p2l(int prec, int64_t n, const double* w, const double* q, double* out, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (prec == DAFMM_FP64) k_op_p2l<double><<<nblk(n), 128, 0, s>>>(n, w, q, out);
    else k_op_p2l<float><<<nblk(n), 128, 0, s>>>(n, w, q, out);
    return cudaGetLastError();
}
static cudaError_t op_l2p(int prec, int64_t n, const double* L, const double* x, double* out4, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (prec == DAFMM_FP64) k_op_eval<double, false><<<nblk(n), 128, 0, s>>>(n, L, x, out4);
    else k_op_eval<float, false><<<nblk(n), 128, 0, s>>>(n, L, x, out4);
    return cudaGetLastError();
}
static cudaError_t op_m2p(int prec, int64_t n, const double* M, const double* x, double* out4, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (prec == DAFMM_FP64) k_op_eval<double, true><<<nblk(n), 128, 0, s>>>(n, M, x, out4);
    else k_op_eval<float, true><<<nblk(n), 128, 0, s>>>(n, M, x, out4);
    return cudaGetLastError();
}
static cudaError_t op_shift(const OrderData& od, int which, int prec, int64_t n, const int* oct,
                            const double* in, double* out, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const ShiftTab t = which == 0 ? od.m2m() : od.l2l();
    if (prec == DAFMM_FP64) k_op_shift<double><<<nblk(n), 128, 0, s>>>(t, n, oct, in, out);
    else k_op_shift<float><<<nblk(n), 128, 0, s>>>(t, n, oct, in, out);
    return cudaGetLastError();
}

}  // namespace ord_P

const OrderOps* DAFMM_CAT(order_ops_p, DAFMM_P)() {
    using namespace DAFMM_CAT(ord_, DAFMM_P);
    static const OrderOps ops = {
        P, NC, NCP,
        HostShiftTable{gen::GENT(m2m, _nnz), gen::GENT(m2m, _rowptr), gen::GENT(m2m, _col), gen::GENT(m2m, _par),
                       gen::GENT(m2m, _val)},
        HostShiftTable{gen::GENT(l2l, _nnz), gen::GENT(l2l, _rowptr), gen::GENT(l2l, _col), gen::GENT(l2l, _par),
                       gen::GENT(l2l, _val)},
        HostShiftTable{gen::GENT(m2mh, _nnz), gen::GENT(m2mh, _rowptr), gen::GENT(m2mh, _col), gen::GENT(m2mh, _par),
                       gen::GENT(m2mh, _val)},
        p2m_launch, m2m_launch, l2l_launch, m2l_launch, leaf_launch, kgen_launch, m2l_rot_launch, rot_setup_launch,
        rot_pack_launch, ROT_TSZ,
        op_p2m, op_p2l, op_l2p, op_m2p, op_shift,
        p2m_a_launch, m2m_a_launch, m2l_a_launch, p2l_a_launch, l2l_a_launch, leaf_a_launch,
        m2l_rot_ff_launch, to_ff_launch, split_ff_launch};
    return &ops;
}

}  // namespace dafmm
