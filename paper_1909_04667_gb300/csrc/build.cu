// Oct-tree construction on the GPU (paper Sec. 3.1).
//
// The paper inserts particles one at a time and splits every leaf that would
// hold two of them.  The cells that exist at the end do not depend on the
// insertion order -- a cell exists when its parent holds more than the leaf
// bucket B -- so the same tree is built here in parallel from sorted keys:
//
//   1. root cube and 21-bit integer cell coordinates -> 63-bit Morton keys
//   2. stable radix sort of (key, particle index)
//   3. the nodes straight from the sorted keys, in depth-first pre-order:
//      with w(j) the deepest level shared by keys j and j + B, the cell
//      around particle i holds more than B particles down to level
//      max w(j) over j in [i - B, i], so i's leaf level D(i) is one below
//      (capped at 21); the nodes whose first particle is i are its cells at
//      the levels below the level it shares with particle i - 1, down to
//      D(i).  Nodes ordered by (first particle, level) are the pre-order,
//      so a scan of the per-particle node counts places every node; particle
//      ranges, skip indices and parents follow from searches in the sorted
//      keys.  No level-by-level passes and no host round trip but one (the
//      node count, to size the node tables)
//   4. FP64 masses and mass-weighted positions summed bottom-up, stretches of
//      the key order by their own blocks and what reaches past them
//      afterwards, children in ascending octant order and a leaf's particles in sorted
//      order, with explicit round-to-nearest operations (no contraction), so
//      the result is the same bit for bit on any correct implementation of
//      that order
//   5. pre-order and breadth-first tables for the walks: per node the FP32 geometric
//      centre (exact: it lies on the 2^-22 L0 grid), side, centre of mass
//      relative to the centre, mass, skip index, particle range and leaf flag
//      -- three 16-byte records loaded with one vector load each -- and per
//      sorted particle its position relative to its leaf centre plus mass.
#include <cub/cub.cuh>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>

#include "tpm_internal.cuh"

namespace tpm {
namespace {

constexpr int kThreads = 256;

inline unsigned blocks_for(int64_t n, int t = kThreads) { return (unsigned)((n + t - 1) / t); }

// Order-preserving map of a double to a signed 64-bit integer (for atomic
// min / max of doubles).
__device__ __forceinline__ long long ordered_bits(double v) {
    long long b = __double_as_longlong(v);
    return b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
}
__host__ __device__ inline double from_ordered_bits(long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b >= 0 ? b : (b ^ 0x7fffffffffffffffLL));
#else
    long long r = b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
    double d;
    memcpy(&d, &r, sizeof d);
    return d;
#endif
}

// Device-side bookkeeping of one build (its host copy also receives the node
// count).
struct BuildState {
    long long bbox[6];
    int bad;
    unsigned total;  // nodes of the tree
    double x0[3];
    double L0;
    double scale;  // 2^21 / L0
    unsigned blocks_done;  // k_prepare blocks that have reduced their bounding box
};

__device__ double pow2_ceil_d(double x) {
    int e;
    const double f = frexp(x, &e);
    return (f == 0.5) ? ldexp(1.0, e - 1) : ldexp(1.0, e);
}

// Root cube (one thread, once the bounding box is complete): periodic
// [0, box); open boundaries: the smallest power of two L0 >= 1.25 x the
// largest extent, x0 = lo - shift (L0 - extent) rounded down to the 2^-21 L0
// grid.  Round-to-nearest operations only.
__device__ void root_cube(BuildState *__restrict__ st, int periodic, double box, double s0, double s1, double s2) {
    if (periodic) {
        st->x0[0] = st->x0[1] = st->x0[2] = 0.0;
        st->L0 = box;
    } else {
        double lo[3], hi[3], ext = 0.0;
        for (int a = 0; a < 3; a++) {
            lo[a] = from_ordered_bits(__ldcg(&st->bbox[a]));  // reduced by other blocks' atomics
            hi[a] = from_ordered_bits(__ldcg(&st->bbox[3 + a]));
            ext = fmax(ext, __dsub_rn(hi[a], lo[a]));
        }
        if (!(ext > 0.0))
            ext = 1.0;
        const double L0 = pow2_ceil_d(__dmul_rn(1.25, ext));
        const double unit = ldexp(L0, -kMaxLevel);
        const double sh[3] = {s0, s1, s2};
        for (int a = 0; a < 3; a++) {
            const double slack = __dsub_rn(L0, __dsub_rn(hi[a], lo[a]));
            const double x0 = __dsub_rn(lo[a], __dmul_rn(sh[a], slack));
            st->x0[a] = __dmul_rn(floor(__ddiv_rn(x0, unit)), unit);
        }
        st->L0 = L0;
    }
    st->scale = __ddiv_rn(ldexp(1.0, kMaxLevel), st->L0);
}

// Copies positions and masses into the system, applies the periodic shift and
// wrap, checks finiteness and ranges (and the per-particle softening lengths,
// if any), and reduces the bounding box (open boundaries); the last block to
// finish computes the root cube from it.
__global__ void k_prepare(const double *__restrict__ pin, const float *__restrict__ mass_in,
                          const float *__restrict__ hsoft, int64_t n, int periodic, double box, double s0, double s1,
                          double s2, double *__restrict__ pout, float *__restrict__ mout,
                          BuildState *__restrict__ state) {
    long long *bbox = state->bbox;
    long long lo[3] = {LLONG_MAX, LLONG_MAX, LLONG_MAX}, hi[3] = {LLONG_MIN, LLONG_MIN, LLONG_MIN};
    int bad = 0;
    // comparisons on the bits: non-negative doubles order like integers, and
    // FP64 instructions (comparisons too) are what bounds this kernel
    const uint64_t box_bits = (uint64_t)__double_as_longlong(box), inf_bits = 0x7ffull << 52, minus0 = 1ull << 63;
    const double sh[3] = {__dmul_rn(s0, box), __dmul_rn(s1, box), __dmul_rn(s2, box)};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
            double v = pin[3 * i + a];
            const uint64_t vb = (uint64_t)__double_as_longlong(v);
            bad |= (vb & inf_bits) == inf_bits ? 1 : 0;
            if (periodic) {
                bad |= vb < box_bits || vb == minus0 ? 0 : 2;
                v = __dadd_rn(v, sh[a]);
                if (__double_as_longlong(v) >= (long long)box_bits)  // signed: -0.0 stays below
                    v = __dsub_rn(v, box);
            } else {
                lo[a] = min(lo[a], ordered_bits(v));
                hi[a] = max(hi[a], ordered_bits(v));
            }
            pout[3 * i + a] = v;
        }
        const float m = mass_in[i];
        bad |= m > 0.0f && isfinite(m) ? 0 : 4;
        mout[i] = m;
        if (hsoft) {
            const float h = hsoft[i];
            bad |= h > 0.0f && isfinite(h) ? 0 : 8;
        }
    }
    if (bad)
        atomicOr(&state->bad, bad);
    if (periodic) {  // the root is the box
        if (blockIdx.x == 0 && threadIdx.x == 0)
            root_cube(state, periodic, box, s0, s1, s2);
        return;
    }
    // warp-level min / max, then one atomic per block
    __shared__ long long red[2][3][32];
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        long long l = lo[a], h = hi[a];
        for (int o = 16; o > 0; o >>= 1) {
            l = min(l, __shfl_xor_sync(0xffffffffu, l, o));
            h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
        }
        if ((threadIdx.x & 31) == 0) {
            red[0][a][w] = l;
            red[1][a][w] = h;
        }
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        const int a = threadIdx.x;
        long long l = LLONG_MAX, h = LLONG_MIN;
        for (int i = 0; i < nw; i++) {
            l = min(l, red[0][a][i]);
            h = max(h, red[1][a][i]);
        }
        atomicMin(&bbox[a], l);
        atomicMax(&bbox[3 + a], h);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&state->blocks_done, 1u) == gridDim.x - 1) {
        __threadfence();
        root_cube(state, periodic, box, s0, s1, s2);
    }
}

// Spreads the low 21 bits of v to every third bit (bit b -> bit 3b).
__device__ __forceinline__ uint64_t spread3(uint64_t v) {
    v &= 0x1fffffull;
    v = (v | (v << 32)) & 0x001f00000000ffffull;
    v = (v | (v << 16)) & 0x001f0000ff0000ffull;
    v = (v | (v << 8)) & 0x100f00f00f00f00full;
    v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
    v = (v | (v << 2)) & 0x1249249249249249ull;
    return v;
}

__device__ __forceinline__ uint32_t compact3(uint64_t v) {
    v &= 0x1249249249249249ull;
    v = (v ^ (v >> 2)) & 0x10c30c30c30c30c3ull;
    v = (v ^ (v >> 4)) & 0x100f00f00f00f00full;
    v = (v ^ (v >> 8)) & 0x001f0000ff0000ffull;
    v = (v ^ (v >> 16)) & 0x001f00000000ffffull;
    v = (v ^ (v >> 32)) & 0x1fffffull;
    return (uint32_t)v;
}

// floor(v 2^shift) clamped to [0, 2^21 - 1], read off the bits of v (integer
// operations only: FP64 arithmetic is scarce on this GPU).  With v 2^shift =
// m 2^(e - 52), m the 53-bit significand, the integer part for 1 <= v 2^shift
// < 2^21 is m >> (52 - e); negative v (sign bit set) and values below 1 give
// 0, values from 2^21 on (and non-finite v) the largest coordinate.
__device__ __forceinline__ uint32_t cell_coord(double v, int shift) {
    const long long b = __double_as_longlong(v);
    if (b < 0 || b < (1ll << 52))  // negative, zero or denormal
        return 0u;
    const int e = (int)(b >> 52) - 1023 + shift;
    if (e < 0)
        return 0u;
    if (e >= kMaxLevel)
        return (1u << kMaxLevel) - 1u;
    const uint64_t m = ((uint64_t)b & 0xfffffffffffffull) | (1ull << 52);
    return (uint32_t)(m >> (52 - e));
}

// K1: Morton keys of the 21-bit cell coordinates q = floor((x - x0) 2^21 / L0).
__global__ void k_keys(const double *__restrict__ pos, int64_t n, const BuildState *__restrict__ st,
                       uint64_t *__restrict__ key, uint32_t *__restrict__ idx) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    // One FP64 operation per coordinate (they bound this kernel): with open
    // boundaries the scale is a power of two, 2^shift, and the product an
    // addition to the exponent; a periodic box has its corner at 0.
    const double o[3] = {st->x0[0], st->x0[1], st->x0[2]};
    const double scale = st->scale;
    const uint64_t sb = (uint64_t)__double_as_longlong(scale);
    // (roots below 2^-580 keep the product: their coordinates may be denormal)
    const bool pow2 = (sb & 0xfffffffffffffull) == 0ull && sb < (1623ull << 52);
    const int shift = pow2 ? (int)(sb >> 52) - 1023 : 0;
    double v[3] = {pos[3 * i], pos[3 * i + 1], pos[3 * i + 2]};
    if (o[0] != 0.0 || o[1] != 0.0 || o[2] != 0.0) {
#pragma unroll
        for (int a = 0; a < 3; a++)
            v[a] = __dsub_rn(v[a], o[a]);
    }
    if (!pow2) {
#pragma unroll
        for (int a = 0; a < 3; a++)
            v[a] = __dmul_rn(v[a], scale);
    }
    const uint64_t k = spread3(cell_coord(v[0], shift)) | spread3(cell_coord(v[1], shift)) << 1 |
                       spread3(cell_coord(v[2], shift)) << 2;
    key[i] = k;
    idx[i] = (uint32_t)i;
}

// Deepest level whose cell holds both keys (kMaxLevel when they are equal).
__device__ __forceinline__ int common_level(uint64_t a, uint64_t b) {
    const uint64_t x = a ^ b;
    return x ? (kMaxLevel - 1) - (63 - __clzll((long long)x)) / 3 : kMaxLevel;
}

// Smallest e in [lo, hi] with e == hi or key[e] >= bound (keys ascending,
// key[lo - 1] < bound): exponential search from lo, then bisection.
__device__ __forceinline__ uint32_t search_up(const uint64_t *__restrict__ key, uint32_t lo, uint32_t hi,
                                              uint64_t bound) {
    uint32_t a = lo, b = lo;
    uint64_t step = 1;
    while (b < hi && key[b] < bound) {
        a = b + 1;
        b = (uint64_t)(hi - b) > step ? b + (uint32_t)step : hi;
        step <<= 1;
    }
    while (a < b) {
        const uint32_t mid = a + ((b - a) >> 1);
        if (key[mid] < bound)
            a = mid + 1;
        else
            b = mid;
    }
    return a;
}

// Smallest f <= i with key[f] >= bound, given key[i] >= bound: exponential
// search downwards from i, then bisection.
__device__ __forceinline__ uint32_t search_down(const uint64_t *__restrict__ key, uint32_t i, uint64_t bound) {
    int64_t hi = i, lo = (int64_t)i - 1, step = 1;
    while (lo >= 0 && key[lo] >= bound) {
        hi = lo;
        lo -= step;
        step <<= 1;
    }
    int64_t a = lo + 1 > 0 ? lo + 1 : 0, b = hi;
    while (a < b) {
        const int64_t mid = a + ((b - a) >> 1);
        if (key[mid] < bound)
            a = mid + 1;
        else
            b = mid;
    }
    return (uint32_t)a;
}

// K3a. Which cells hold more than B particles.  The level-m cell around sorted
// particle i holds more than B particles iff some run of B + 1 consecutive
// particles inside it contains i, i.e. iff w(j) >= m for some j in [i - B, i],
// where w(j) = common_level(key[j], key[j + B]).  The window maximum over
// [i - B, i] comes from prefix and suffix maxima inside blocks of B + 1
// entries (one thread per block); this kernel writes them.
__global__ void k_window_max(const uint64_t *__restrict__ key, int64_t n, int B, int8_t *__restrict__ pre_max,
                             int8_t *__restrict__ suf_max) {
    const int64_t W = (int64_t)B + 1;
    const int64_t j0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * W;
    if (j0 >= n)
        return;
    const int64_t j1 = min(j0 + W, n);
    int m = -1;
    for (int64_t j = j0; j < j1; j++) {
        const int w = j + B < n ? common_level(key[j], key[j + B]) : -1;
        suf_max[j] = (int8_t)w;
        m = max(m, w);
        pre_max[j] = (int8_t)m;
    }
    m = -1;
    for (int64_t j = j1 - 1; j >= j0; j--) {
        m = max(m, (int)suf_max[j]);
        suf_max[j] = (int8_t)m;
    }
}

// K3b. Per sorted particle i: the level of its leaf, D(i) = min(1 + deepest
// level whose cell around i holds more than B particles, 21), and the levels
// at which i is the first particle of its cell, (common_level(key[i-1],
// key[i]), D(i)].  Those cells are exactly the nodes whose first particle is
// i, and ordering all nodes by (first particle, level) is the depth-first
// pre-order: an exclusive scan of the per-particle counts gives every node
// its pre-order index directly.
__global__ void k_node_counts(const uint64_t *__restrict__ key, int64_t n, int B, const int8_t *__restrict__ pre_max,
                              const int8_t *__restrict__ suf_max, uint8_t *__restrict__ top_level,
                              uint8_t *__restrict__ leaf_level, uint32_t *__restrict__ cnt) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    const int lp = i ? common_level(key[i - 1], key[i]) : -1;
    int split = pre_max[i];  // deepest level whose cell around i holds > B particles
    if (i - B >= 0)
        split = max(split, (int)suf_max[i - B]);
    const int D = min(split + 1, kMaxLevel);
    top_level[i] = (uint8_t)(lp + 1);
    leaf_level[i] = (uint8_t)D;
    cnt[i] = (uint32_t)max(D - lp, 0);
}

// Exact centre of node (lvl, pre) relative to x0: (2 i + 1) L0 2^-(lvl + 1)
// per axis, i the cell index along the axis read off the key prefix; the
// power of two is built from its bits (exact scaling, lvl <= 21).
struct NodeGeom {
    double rx, ry, rz, side;
};
__device__ __forceinline__ NodeGeom node_geom(uint64_t pre, int lvl, double L0) {
    const double half = __dmul_rn(L0, __longlong_as_double((long long)(1022 - lvl) << 52));
    NodeGeom g;
    g.rx = __dmul_rn((double)(2 * (uint64_t)compact3(pre) + 1), half);
    g.ry = __dmul_rn((double)(2 * (uint64_t)compact3(pre >> 1) + 1), half);
    g.rz = __dmul_rn((double)(2 * (uint64_t)compact3(pre >> 2) + 1), half);
    g.side = 2.0 * half;
    return g;
}

// K2 for small systems: the sorted position of every particle by counting the
// particles before it, (key, index) below its own, over chunks of kRankChunk
// others (a block per 256 particles and chunk, the chunk's keys in shared
// memory).  n^2 comparisons, but two launches: the radix sort takes eight
// passes of two launches each, some 100 us however few the particles.  A step
// (build and forces) with the sort / with this: 4096 particles 270 / 190 us,
// 8192 290 / 222, 16384 340 / 286; the count grows as n^2 (some 45 us at
// 16384), so the line is drawn at 20480.
constexpr int64_t kRankSort = 5 << 12;
constexpr int kRankChunk = 512;
__global__ void __launch_bounds__(kThreads)
    k_count_before(const uint64_t *__restrict__ key, int n, uint32_t *__restrict__ rank) {
    __shared__ __align__(16) uint64_t other[kRankChunk];
    const int j0 = blockIdx.y * kRankChunk, m = min(kRankChunk, n - j0);
    for (int e = threadIdx.x; e < kRankChunk; e += kThreads)
        other[e] = e < m ? key[j0 + e] : ~0ull;  // padding counts for nobody: keys have 63 bits
    __syncthreads();
    const int i0 = blockIdx.x * kThreads, i = i0 + threadIdx.x;
    if (i >= n)
        return;
    const uint64_t own = key[i];
    uint32_t before = 0u;
    if (j0 + kRankChunk <= i0 || j0 >= i0 + kThreads) {
        // all of the chunk before this block's particles (equal keys count) or after
        const uint64_t bound = own + (j0 < i0 ? 1u : 0u);
        const ulonglong2 *two = reinterpret_cast<const ulonglong2 *>(other);
#pragma unroll 8
        for (int e = 0; e < kRankChunk / 2; e++) {
            const ulonglong2 k = two[e];
            before += (k.x < bound ? 1u : 0u) + (k.y < bound ? 1u : 0u);
        }
    } else {
        for (int e = 0; e < m; e++)
            before += other[e] < own + (j0 + e < i ? 1u : 0u) ? 1u : 0u;
    }
    atomicAdd(&rank[i], before);
}

__global__ void k_place(const uint64_t *__restrict__ key, int n, const uint32_t *__restrict__ rank,
                        uint64_t *__restrict__ sorted, uint32_t *__restrict__ perm) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        sorted[rank[i]] = key[i];
        perm[rank[i]] = (uint32_t)i;
    }
}

// FP32 centre, relative to x0, of the level-lvl cell around a key.  With L0 a
// power of two (open boundaries) the FP32 product of the odd cell index (at
// most 22 bits) and half the side is exact, so it has the bits of the FP64
// product rounded to FP32; FP64 instructions are what bounds k_rank.
__device__ __forceinline__ float3 leaf_centre(uint64_t key, int lvl, double L0) {
    const uint64_t pre = key >> (3 * (kMaxLevel - lvl));
    if (((uint64_t)__double_as_longlong(L0) & 0xfffffffffffffull) == 0ull) {
        const float half = (float)__dmul_rn(L0, __longlong_as_double((long long)(1022 - lvl) << 52));
        return make_float3((float)(2u * compact3(pre) + 1u) * half, (float)(2u * compact3(pre >> 1) + 1u) * half,
                           (float)(2u * compact3(pre >> 2) + 1u) * half);
    }
    const NodeGeom g = node_geom(pre, lvl, L0);
    return make_float3((float)g.rx, (float)g.ry, (float)g.rz);
}

// K3d. Inverse permutation, positions and masses gathered into key order for
// the sums over leaves, and each particle's walk record: its position relative
// to the FP32 centre of its leaf (FP64 difference rounded to FP32) and its
// mass.  The leaf is known from the key and the leaf level, so this runs while
// the host reads the node count.
__global__ void k_rank(const uint32_t *__restrict__ perm, int64_t n, const double *__restrict__ pos,
                       const float *__restrict__ mass, const float *__restrict__ hsoft,
                       const uint64_t *__restrict__ key, const uint8_t *__restrict__ leaf_level,
                       const BuildState *__restrict__ st, uint32_t *__restrict__ rank, double *__restrict__ spos,
                       float *__restrict__ smass, float *__restrict__ psoft, float4 *__restrict__ spart) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= n)
        return;
    const uint32_t j = perm[s];
    rank[j] = (uint32_t)s;
    const double x = pos[3 * (size_t)j], y = pos[3 * (size_t)j + 1], z = pos[3 * (size_t)j + 2];
    const float m = mass[j];
    spos[3 * s] = x;
    spos[3 * s + 1] = y;
    spos[3 * s + 2] = z;
    smass[s] = m;
    if (hsoft)  // per-particle softening, in key order (checked by k_prepare)
        psoft[s] = hsoft[j];
    const float3 c = leaf_centre(key[s], leaf_level[s], st->L0);
    spart[s] = make_float4((float)__dsub_rn(x, __dadd_rn(st->x0[0], (double)c.x)),
                           (float)__dsub_rn(y, __dadd_rn(st->x0[1], (double)c.y)),
                           (float)__dsub_rn(z, __dadd_rn(st->x0[2], (double)c.z)), m);
}

// Pre-order node arrays of the build.
struct NodeArrays {
    uint32_t *first, *count, *skip, *nchild;
    uint8_t *level;
    uint64_t *prefix;
};

constexpr int kLevels = kMaxLevel + 1;

// K3c. The nodes, one thread each (a thread per particle with nodes left the
// first particle's thread, which starts a node on every level, with some 500
// dependent loads: 51 us at 2^20, 25 us now): the particle a node starts with
// is found in the scanned node counts, its level counted from that particle's
// top one, its end by searching the sorted keys; then the skip index (the
// first node of the particle just past the cell), the key prefix, the parent
// (the node above with the same first particle, else the cell found by
// searching downwards) and, by one atomic per node, the parent's child count.
// The block's nodes per level go to hist[level][block] for the breadth-first
// order.
__global__ void __launch_bounds__(kThreads)
    k_nodes(const uint64_t *__restrict__ key, int64_t n, int64_t total, const uint32_t *__restrict__ base,
            const uint8_t *__restrict__ top_level, NodeArrays t, uint32_t *__restrict__ hist) {
    __shared__ uint32_t h[kLevels];
    if (threadIdx.x < kLevels)
        h[threadIdx.x] = 0u;
    __syncthreads();
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < total) {
        // the last particle whose first node is at or before p
        int64_t lo = 0, hi = n - 1;
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (base[mid] <= (uint32_t)p)
                lo = mid;
            else
                hi = mid - 1;
        }
        const uint32_t i = (uint32_t)lo, k = (uint32_t)p - base[i];
        const int l = top_level[i] + (int)k;
        const int sh = 3 * (kMaxLevel - l);
        const uint64_t pre = key[i] >> sh;
        const uint32_t end = search_up(key, i + 1, (uint32_t)n, (pre + 1) << sh);
        t.first[p] = i;
        t.count[p] = end - i;
        t.skip[p] = end < n ? base[end] : (uint32_t)total;
        t.level[p] = (uint8_t)l;
        t.prefix[p] = pre;
        if (l > 0) {
            uint32_t par = (uint32_t)p - 1;
            if (k == 0) {
                const uint32_t f = search_down(key, i, (pre >> 3) << (sh + 3));
                par = base[f] + (uint32_t)(l - 1 - top_level[f]);
            }
            atomicAdd(&t.nchild[par], 1u);
        }
        atomicAdd(&h[l], 1u);
    }
    __syncthreads();
    if (threadIdx.x < kLevels)
        hist[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = h[threadIdx.x];
}

// K3e. Breadth-first order: a stable counting sort of the pre-order by level.
// place holds, per level and block of K3c, how many nodes come before; within
// a block the nodes of a level keep their order.
__global__ void __launch_bounds__(kThreads)
    k_level_rank(const uint8_t *__restrict__ level, int64_t total, const uint32_t *__restrict__ place,
                 uint32_t *__restrict__ pre2bfs) {
    __shared__ uint32_t h[kThreads / 32][kLevels];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int e = threadIdx.x; e < (kThreads / 32) * kLevels; e += kThreads)
        (&h[0][0])[e] = 0u;
    __syncthreads();
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int l = p < total ? (int)level[p] : kLevels;
    const unsigned same = __match_any_sync(0xffffffffu, l);
    const unsigned before = __popc(same & ((1u << lane) - 1u));
    if (l < kLevels && before == 0)
        h[w][l] = (uint32_t)__popc(same);
    __syncthreads();
    if (l < kLevels) {
        uint32_t q = place[(size_t)l * gridDim.x + blockIdx.x] + before;
        for (int v = 0; v < w; v++)
            q += h[v][l];
        pre2bfs[p] = q;
    }
}

// K4: FP64 monopoles, bottom-up.  Each leaf sums its particles in sorted
// order, each node its children in ascending octant order, with explicit
// round-to-nearest adds / muls, so every sum has the same fixed order and
// value however the work is divided.  Sums are stored by breadth-first index,
// where a node's children are contiguous, so that the children's sums load
// independently.
//
// A block takes the nodes that start in a stretch of kStretch sorted particles
// -- contiguous in the pre-order -- and sums level by level, a block barrier
// between the levels, the nodes whose subtree ends in the stretch too.  Those
// that reach past its end all hold the stretch's last particle, so there is
// one a level at most; they go to late[level][stretch], and k_multipole_late
// does the same for 32 stretches by one block, again and again until one block
// has them all.
//
// FP64 bounds this (two lanes a cycle and SM, so a warp's FP64 instruction
// takes the unit 16 cycles however few lanes need it).  Hence the block sorts
// its leaves by particle count and its nodes by level before it sums: the
// lanes of a warp have equal work.  (One launch in which the last child of a
// node to finish, counted with an atomic, sums the node and climbs on: 136 us
// at 2^20, leaf bucket 16; this without the sort: 100 + 81 with one block for
// all late nodes; as it is 46 + 28.)
constexpr int kStretch = 1024;
constexpr int kLateFan = 32;
constexpr int kLeafClasses = 17;  // leaves of 1 .. 16 and of more particles

struct Sums {
    double *v;          // per node mass, mass-weighted x, y, z
    float *hmx, *hmn;   // largest and smallest support (per-particle softening only)
};

// Sums the children [c0, c0 + nc) of node q (nc <= 8) in octant order, one of
// the four components per lane: four lanes share a node's chain of additions.
__device__ __forceinline__ void sum_children(const Sums &o, uint32_t q, uint32_t c0, uint32_t nc, int comp) {
    double x[8], sum = 0.0;
#pragma unroll
    for (uint32_t u = 0; u < 8; u++)
        x[u] = __ldcg(&o.v[4 * (size_t)(c0 + min(u, nc - 1)) + comp]);
#pragma unroll
    for (uint32_t u = 0; u < 8; u++)
        if (u < nc)
            sum = __dadd_rn(sum, x[u]);
    o.v[4 * (size_t)q + comp] = sum;
    if (o.hmx && comp < 2) {
        float *h = comp ? o.hmn : o.hmx;
        float r = comp ? INFINITY : 0.0f;
        for (uint32_t c = c0; c < c0 + nc; c++)
            r = comp ? fminf(r, __ldcg(&h[c])) : fmaxf(r, __ldcg(&h[c]));
        h[q] = r;
    }
}

__global__ void __launch_bounds__(kThreads)
    k_multipole(NodeArrays t, int64_t n, const uint32_t *__restrict__ base, const uint32_t *__restrict__ pre2bfs,
                const double *__restrict__ spos, const float *__restrict__ smass, const float *__restrict__ psoft,
                Sums o, uint32_t *__restrict__ list, uint32_t *__restrict__ late) {
    constexpr int kClasses = kLeafClasses + kLevels;  // leaves by size, then nodes from the deepest level up
    __shared__ uint32_t count[kClasses], start[kClasses + 1];
    const int64_t i0 = (int64_t)blockIdx.x * kStretch, i1 = min(i0 + kStretch, n);
    const uint32_t p0 = base[i0], p1 = base[i1];
    if (threadIdx.x < kClasses)
        count[threadIdx.x] = 0u;
    if (threadIdx.x < kLevels)
        late[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = 0xffffffffu;
    __syncthreads();
    auto class_of = [&](uint32_t p) {  // -1: late
        if (t.nchild[p] == 0)
            return (int)min(t.count[p], (uint32_t)kLeafClasses) - 1;
        return t.skip[p] > p1 ? -1 : kLeafClasses + kMaxLevel - (int)t.level[p];
    };
    for (uint32_t p = p0 + threadIdx.x; p < p1; p += kThreads) {
        const int c = class_of(p);
        if (c >= 0)
            atomicAdd(&count[c], 1u);
        else
            late[(size_t)t.level[p] * gridDim.x + blockIdx.x] = p;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t at = p0;
        for (int c = 0; c < kClasses; c++) {
            start[c] = at;
            at += count[c];
            count[c] = start[c];
        }
        start[kClasses] = at;
    }
    __syncthreads();
    for (uint32_t p = p0 + threadIdx.x; p < p1; p += kThreads) {  // any order within a class: each sums by itself
        const int c = class_of(p);
        if (c >= 0)
            list[atomicAdd(&count[c], 1u)] = p;
    }
    __syncthreads();
    for (uint32_t e = start[0] + threadIdx.x; e < start[kLeafClasses]; e += kThreads) {
        const uint32_t p = list[e];
        const uint32_t f = t.first[p], end = f + t.count[p], q = pre2bfs[p];
        double m = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
        float hi = 0.0f, lo = INFINITY;
        for (uint32_t s = f; s < end; s += 4) {  // four particles loaded at a time
            float ms[4], hs[4];
            double px[4], py[4], pz[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const size_t j = min(s + u, end - 1);
                ms[u] = smass[j];
                px[u] = spos[3 * j];
                py[u] = spos[3 * j + 1];
                pz[u] = spos[3 * j + 2];
                hs[u] = psoft ? psoft[j] : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                if (s + u < end) {
                    const double md = (double)ms[u];
                    m = __dadd_rn(m, md);
                    sx = __dadd_rn(sx, __dmul_rn(md, px[u]));
                    sy = __dadd_rn(sy, __dmul_rn(md, py[u]));
                    sz = __dadd_rn(sz, __dmul_rn(md, pz[u]));
                    if (psoft) {
                        hi = fmaxf(hi, hs[u]);
                        lo = fminf(lo, hs[u]);
                    }
                }
            }
        }
        double2 *v = reinterpret_cast<double2 *>(o.v + 4 * (size_t)q);
        v[0] = make_double2(m, sx);
        v[1] = make_double2(sy, sz);
        if (psoft) {
            o.hmx[q] = hi;
            o.hmn[q] = lo;
        }
    }
    for (int c = kLeafClasses; c < kClasses; c++) {
        if (start[c] == start[c + 1])
            continue;
        __syncthreads();
        for (uint32_t e = start[c] + (threadIdx.x >> 2); e < start[c + 1]; e += kThreads / 4) {
            const uint32_t p = list[e];
            sum_children(o, pre2bfs[p], pre2bfs[p + 1], t.nchild[p], threadIdx.x & 3);
        }
    }
}

// The nodes that reach past their stretch: a block per 32 stretches (which
// together are one stretch of `span` particles), four lanes per stretch, from
// the deepest level up; those that reach past the block's end go on to out.
// The links of all levels are loaded first: the chain over the levels is then
// one load of the children's sums and their additions each.
__global__ void __launch_bounds__(4 * kLateFan)
    k_multipole_late(NodeArrays t, int64_t n, const uint32_t *__restrict__ base, const uint32_t *__restrict__ pre2bfs,
                     Sums o, const uint32_t *__restrict__ late, int64_t stretches, int64_t span,
                     uint32_t *__restrict__ out) {
    __shared__ uint32_t node[kLevels][kLateFan], child[kLevels][kLateFan];
    __shared__ uint8_t number[kLevels][kLateFan];  // of children, 0 for no node
    __shared__ unsigned levels;
    const uint32_t end = base[min(((int64_t)blockIdx.x + 1) * span, n)];
    if (threadIdx.x < kLevels)
        out[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = 0xffffffffu;
    if (threadIdx.x == 0)
        levels = 0u;
    __syncthreads();
    for (int e = threadIdx.x; e < kLevels * kLateFan; e += 4 * kLateFan) {
        const int l = e / kLateFan, u = e % kLateFan;
        const int64_t b = (int64_t)blockIdx.x * kLateFan + u;
        const uint32_t p = b < stretches ? late[(size_t)l * stretches + b] : 0xffffffffu;
        uint32_t nc = 0u;
        if (p != 0xffffffffu) {
            if (t.skip[p] > end) {
                out[(size_t)l * gridDim.x + blockIdx.x] = p;
            } else {
                nc = t.nchild[p];
                node[l][u] = pre2bfs[p];
                child[l][u] = pre2bfs[p + 1];
                atomicOr(&levels, 1u << l);
            }
        }
        number[l][u] = (uint8_t)nc;
    }
    __syncthreads();
    const int u = threadIdx.x >> 2, comp = threadIdx.x & 3;
    for (unsigned todo = levels; todo;) {
        const int l = 31 - __clz(todo);
        todo &= ~(1u << l);
        if (number[l][u])
            sum_children(o, node[l][u], child[l][u], number[l][u], comp);
        __syncthreads();
    }
}

struct NodeOut {
    float4 *cen, *com;
    int4 *link;
    uint8_t *level;
    uint64_t *prefix;
    float4 *bcen, *bcom;
    int4 *blink;
    float *nsoft, *bsoft;  // per-particle softening only
};

// K5: walk tables.  Pre-order: FP32 geometric centre (exact, on the 2^-22 L0
// grid) and side, centre of mass relative to the exact centre (FP32) and mass,
// (skip, first particle, count, leaf flag), level and key prefix for export;
// breadth-first: centre, centre of mass and (first child, child count, first
// particle, particle count); and the largest softening per node (negative when
// the node mixes softenings).  S / m is S times the correctly rounded 1 / m:
// one FP64 reciprocal instead of three divisions; the FP64 product is within
// an ulp of the quotient, far below the FP32 rounding of the offset.
__global__ void k_tables(NodeArrays t, const uint32_t *__restrict__ pre2bfs, int64_t total, Sums sums, double x0,
                         double y0, double z0, double L0, NodeOut o) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= total)
        return;
    const uint32_t f = t.first[p], c = t.count[p], nch = t.nchild[p];
    const int lvl = t.level[p];
    const uint64_t pre = t.prefix[p];
    const uint32_t q = pre2bfs[p];
    const NodeGeom g = node_geom(pre, lvl, L0);
    const float4 cen = make_float4((float)g.rx, (float)g.ry, (float)g.rz, (float)g.side);
    o.cen[p] = cen;
    o.link[p] = make_int4((int)t.skip[p], (int)f, (int)c, nch == 0);
    o.level[p] = (uint8_t)lvl;
    o.prefix[p] = pre;
    o.bcen[q] = cen;
    o.blink[q] = make_int4(nch ? (int)pre2bfs[p + 1] : 0, (int)nch, (int)f, (int)c);
    const double2 ms = reinterpret_cast<const double2 *>(sums.v + 4 * (size_t)q)[0],
                  yz = reinterpret_cast<const double2 *>(sums.v + 4 * (size_t)q)[1];
    const double m = ms.x;
    const double rm = __drcp_rn(m);
    const double cx = __dmul_rn(ms.y, rm), cy = __dmul_rn(yz.x, rm), cz = __dmul_rn(yz.y, rm);
    const float4 com = make_float4((float)__dsub_rn(cx, __dadd_rn(x0, g.rx)), (float)__dsub_rn(cy, __dadd_rn(y0, g.ry)),
                                   (float)__dsub_rn(cz, __dadd_rn(z0, g.rz)), (float)m);
    o.com[p] = com;
    o.bcom[q] = com;
    if (sums.hmx) {
        const float v = sums.hmn[q] < sums.hmx[q] ? -sums.hmx[q] : sums.hmx[q];
        o.nsoft[p] = v;
        o.bsoft[q] = v;
    }
}

}  // namespace

int build_tree_device(Ctx *c, System *s, const double *pos_in, const float *mass_in, const float *hsoft_in,
                      cudaStream_t st) {
    const int64_t n = s->n;
    const int B = s->bp.leaf_bucket;
    AllocSet tmp;
    tmp.ctx = c;
    struct Guard {
        AllocSet &t;
        cudaStream_t st;
        ~Guard() { t.release(st); }
    } guard{tmp, st};

    // ---- memory for the particle passes: the system's arrays in one block,
    // the build's scratch in another (the CUB scratch sized for the key sort
    // and the node-count scan, whichever is larger)
    size_t sort_bytes = 0, scan_bytes = 0;
    TPM_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, sort_bytes, (const uint64_t *)nullptr, (uint64_t *)nullptr,
                                             (const uint32_t *)nullptr, (uint32_t *)nullptr, (int)n, 0, 3 * kMaxLevel,
                                             st));
    TPM_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, scan_bytes, (const uint32_t *)nullptr, (uint32_t *)nullptr,
                                           (int)(n + 1), st));
    const size_t cub_bytes = std::max(sort_bytes, scan_bytes);
    Carve sys_a;
    sys_a.add(&s->pos, 3 * n);
    sys_a.add(&s->mass, n);
    sys_a.add(&s->key, n);
    sys_a.add(&s->perm, n);
    sys_a.add(&s->rank, n);
    sys_a.add(&s->spart, n);
    sys_a.add(&s->err, 1);
    if (hsoft_in)
        sys_a.add(&s->psoft, n);
    TPM_CHECK(sys_a.commit(s->mem, st));
    BuildState *dst;
    uint64_t *key_raw;
    uint32_t *idx_raw;
    char *cub_tmp;
    double *spos;
    float *smass;
    int8_t *pre_max, *suf_max;
    uint8_t *top_level, *leaf_level;
    uint32_t *cnt, *base;
    Carve tmp_a;
    tmp_a.add(&dst, 1);
    tmp_a.add(&key_raw, n);
    tmp_a.add(&idx_raw, n);
    tmp_a.add(&cub_tmp, cub_bytes);
    tmp_a.add(&spos, 3 * n);
    tmp_a.add(&smass, n);
    tmp_a.add(&pre_max, n);
    tmp_a.add(&suf_max, n);
    tmp_a.add(&top_level, n);
    tmp_a.add(&leaf_level, n);
    tmp_a.add(&cnt, n + 1);
    tmp_a.add(&base, n + 1);
    TPM_CHECK(tmp_a.commit(tmp, st));
    TPM_CUDA(cudaMemsetAsync(s->err, 0, sizeof(int), st));

    // the context's pinned page holds the host copy of the build state; one
    // build at a time per context uses it
    static_assert(sizeof(BuildState) <= kPinnedStateBytes, "build state exceeds the pinned page");
    std::lock_guard<std::mutex> build_lock(c->build_mu);
    BuildState *hst = static_cast<BuildState *>(c->pinned_state);
    memset(hst, 0, sizeof(BuildState));
    for (int a = 0; a < 3; a++) {
        hst->bbox[a] = LLONG_MAX;
        hst->bbox[3 + a] = LLONG_MIN;
    }
    TPM_CUDA(cudaMemcpyAsync(dst, hst, sizeof(BuildState), cudaMemcpyHostToDevice, st));

    // ---- prepare, bounding box and root (last block), keys, sort
    // (few blocks, several particles a thread: each block ends in a reduction and
    // six atomics on the same words)
    k_prepare<<<std::min(blocks_for(n), (unsigned)(8 * c->num_sms)), kThreads, 0, st>>>(pos_in, mass_in, hsoft_in, n, s->bp.periodic, s->bp.box,
                                                   s->bp.shift[0], s->bp.shift[1], s->bp.shift[2], s->pos, s->mass,
                                                   dst);
    count_launch();
    TPM_CUDA(cudaGetLastError());
    k_keys<<<blocks_for(n), kThreads, 0, st>>>(s->pos, n, dst, key_raw, idx_raw);
    count_launch();
    TPM_CUDA(cudaGetLastError());
    if (n <= kRankSort) {
        TPM_CUDA(cudaMemsetAsync(s->rank, 0, n * sizeof(uint32_t), st));
        k_count_before<<<dim3(blocks_for(n), blocks_for(n, kRankChunk)), kThreads, 0, st>>>(key_raw, (int)n, s->rank);
        k_place<<<blocks_for(n), kThreads, 0, st>>>(key_raw, (int)n, s->rank, s->key, s->perm);
        count_launch(2);
        TPM_CUDA(cudaGetLastError());
    } else {
        TPM_CUDA(cub::DeviceRadixSort::SortPairs(cub_tmp, sort_bytes, key_raw, s->key, idx_raw, s->perm, (int)n, 0,
                                                 3 * kMaxLevel, st));
        count_cub_call();
    }

    // ---- node counts per particle and their scan: the pre-order indices
    k_window_max<<<blocks_for((n + B) / ((int64_t)B + 1)), kThreads, 0, st>>>(s->key, n, B, pre_max, suf_max);
    count_launch();
    TPM_CUDA(cudaGetLastError());
    TPM_CUDA(cudaMemsetAsync(cnt + n, 0, sizeof(uint32_t), st));
    k_node_counts<<<blocks_for(n), kThreads, 0, st>>>(s->key, n, B, pre_max, suf_max, top_level, leaf_level, cnt);
    count_launch();
    TPM_CUDA(cudaGetLastError());
    TPM_CUDA(cub::DeviceScan::ExclusiveSum(cub_tmp, scan_bytes, cnt, base, (int)(n + 1), st));
    count_cub_call();
    TPM_CUDA(cudaMemcpyAsync(hst, dst, sizeof(BuildState), cudaMemcpyDeviceToHost, st));
    TPM_CUDA(cudaMemcpyAsync(&hst->total, base + n, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    TPM_CUDA(cudaEventRecord(c->ev_state, st));
    // the particles in key order and their walk records while the host reads the state
    k_rank<<<blocks_for(n), kThreads, 0, st>>>(s->perm, n, s->pos, s->mass, hsoft_in, s->key, leaf_level, dst, s->rank,
                                               spos, smass, s->psoft, s->spart);
    count_launch();
    TPM_CUDA(cudaGetLastError());
    TPM_CUDA(cudaEventSynchronize(c->ev_state));
    if (hst->bad & 1) {
        set_error("non-finite position");
        return TPM_ENAN;
    }
    if (hst->bad & 4) {
        set_error("masses must be finite and > 0");
        return TPM_ENAN;
    }
    if (hst->bad & 2) {
        set_error("periodic positions must lie in [0, box)");
        return TPM_EINVAL;
    }
    if (hst->bad & 8) {
        set_error("softening lengths must be finite and > 0");
        return TPM_ENAN;
    }
    for (int a = 0; a < 3; a++) {
        s->x0[a] = hst->x0[a];
        // a periodic build takes no bounding box: the positions' region is the box
        s->bb_lo[a] = s->bp.periodic ? 0.0 : from_ordered_bits(hst->bbox[a]);
        s->bb_hi[a] = s->bp.periodic ? s->bp.box : from_ordered_bits(hst->bbox[3 + a]);
    }
    s->L0 = hst->L0;
    const int64_t nn = hst->total;
    s->nnodes = nn;

    // ---- memory for the node passes: scratch in one block, the system's
    // node tables in another
    NodeArrays t{};
    uint32_t *hist, *place, *list, *late, *later;
    Sums sums{};
    const unsigned node_blocks = blocks_for(nn);
    const int64_t cells = (int64_t)kLevels * node_blocks, stretches = (n + kStretch - 1) / kStretch;
    size_t place_bytes = 0;
    TPM_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, place_bytes, (const uint32_t *)nullptr, (uint32_t *)nullptr,
                                           (int)cells, st));
    char *place_tmp = cub_tmp;
    Carve tmp_b;
    tmp_b.add(&t.nchild, nn);
    tmp_b.add(&t.first, nn);
    tmp_b.add(&t.count, nn);
    tmp_b.add(&t.skip, nn);
    tmp_b.add(&t.level, nn);
    tmp_b.add(&t.prefix, nn);
    tmp_b.add(&hist, cells);
    tmp_b.add(&place, cells);
    tmp_b.add(&list, nn);
    // the lists of nodes that reach past their stretch, by particles and not by
    // nodes, lie in the unsorted keys, which the sort has done with (a system of
    // few, large leaves needs no more memory for them)
    const int64_t late_n = kLevels * stretches, later_n = kLevels * ((stretches + kLateFan - 1) / kLateFan);
    late = reinterpret_cast<uint32_t *>(key_raw);
    later = late + late_n;
    if (late_n + later_n > 2 * n) {  // n below 22
        tmp_b.add(&late, late_n);
        tmp_b.add(&later, later_n);
    }
    if (place_bytes > cub_bytes)
        tmp_b.add(&place_tmp, place_bytes);
    if (s->psoft) {
        tmp_b.add(&sums.hmx, nn);
        tmp_b.add(&sums.hmn, nn);
    }
    TPM_CHECK(tmp_b.commit(tmp, st));
    Carve sys_b;
    sys_b.add(&s->msum, 4 * nn);  // FP64 sums by breadth-first index, kept with the system for export
    sys_b.add(&s->pre2bfs, nn);
    sys_b.add(&s->ncen, nn);
    sys_b.add(&s->ncom, nn);
    sys_b.add(&s->nlink, nn);
    sys_b.add(&s->nlevel, nn);
    sys_b.add(&s->nprefix, nn);
    sys_b.add(&s->bcen, nn);
    sys_b.add(&s->bcom, nn);
    sys_b.add(&s->blink, nn);
    if (s->psoft) {
        sys_b.add(&s->nsoft, nn);
        sys_b.add(&s->bsoft, nn);
    }
    TPM_CHECK(sys_b.commit(s->mem, st));
    sums.v = s->msum;
    uint32_t *pre2bfs = s->pre2bfs;

    // ---- nodes in pre-order, their breadth-first order, monopoles, tables
    TPM_CUDA(cudaMemsetAsync(t.nchild, 0, nn * sizeof(uint32_t), st));
    k_nodes<<<node_blocks, kThreads, 0, st>>>(s->key, n, nn, base, top_level, t, hist);
    count_launch();
    TPM_CUDA(cudaGetLastError());
    TPM_CUDA(cub::DeviceScan::ExclusiveSum(place_tmp, place_bytes, hist, place, (int)cells, st));
    count_cub_call();
    k_level_rank<<<node_blocks, kThreads, 0, st>>>(t.level, nn, place, pre2bfs);
    count_launch();
    TPM_CUDA(cudaGetLastError());
    k_multipole<<<(unsigned)stretches, kThreads, 0, st>>>(t, n, base, pre2bfs, spos, smass, s->psoft, sums, list, late);
    count_launch();
    TPM_CUDA(cudaGetLastError());
    for (int64_t left = stretches, span = (int64_t)kStretch * kLateFan;; span *= kLateFan) {
        const int64_t blocks = (left + kLateFan - 1) / kLateFan;
        k_multipole_late<<<(unsigned)blocks, 4 * kLateFan, 0, st>>>(t, n, base, pre2bfs, sums, late, left, span, later);
        count_launch();
        TPM_CUDA(cudaGetLastError());
        if (blocks == 1)
            break;
        std::swap(late, later);  // the lists shrink: both have room
        left = blocks;
    }
    NodeOut o{s->ncen, s->ncom, s->nlink, s->nlevel, s->nprefix, s->bcen, s->bcom, s->blink, s->nsoft, s->bsoft};
    k_tables<<<node_blocks, kThreads, 0, st>>>(t, pre2bfs, nn, sums, s->x0[0], s->x0[1], s->x0[2], s->L0, o);
    count_launch();
    TPM_CUDA(cudaGetLastError());
    return TPM_OK;
}

}  // namespace tpm
