// Kernels of the high-dimensional path (5 <= d <= 64), templated on the coordinate type T and
// the padded row width DP (8, 16, 32 or 64 >= d; the padding coordinates are zero and add
// exact zeros to every distance).
//
// In d dimensions the hypercubes of side eps/sqrt(d) (Sec. 2, Algorithm 1) hold about one point
// each on spread data and their neighbour block (2 ceil(sqrt d) + 1)^d (Sec. 2, "Depth First
// Search") is astronomically large, so the neighbour search uses a coarse grid instead: cells
// of side >= eps over the three dimensions of largest extent.  Two points within eps differ by
// at most eps in every coordinate, so they lie in the same or adjacent coarse cells (the 3x3x3
// block).  The coarse cells are binned, sorted, run-length encoded, hashed and given neighbour
// ranges by the same kernels as the hypercube path (D = 3 on the projected coordinates).  The
// clustering itself then works on points: exact counts with early exit at MINPTS
// (Definition 2), union-find over core points (Definitions 3-5) and the canonical labels.
//
// Neighbour lists.  The counts write down the first nl_k neighbours that they find of every
// point, and the later phases start from those instead of comparing points again:
//   - a non-core point has fewer than MINPTS neighbours, so with nl_k >= MINPTS - 1 its list is
//     complete and its label is the smallest cluster id among the listed core points;
//   - the listed core neighbours of a core point are edges of the core graph: joined first, they
//     leave one tree per cluster and cell but for a few odd points, so that the unions only
//     compare the odd points with their neighbourhood and the cells whose trees still differ.
//
// Double input.  With the filter on (FILTER = true) the pair tests of double input run on a float
// copy of the points, taken relative to the set's smallest coordinates, against thresholds that
// bound the copy's rounding (make_coarse_grid); the pairs between the thresholds are decided by
// the exact predicate on the double coordinates.
//
// Layout: pts[j * DP + i] (cell order, zero padded), perm[j], cell_start/cell_key/ranges of
// the coarse cells, core[j], parent[j] and comp_min[j] over points.
#pragma once

#include <type_traits>

#include "lowd_kernels.cuh"

namespace hca {

template <typename T, int DP>
struct HdView {
    GridParams g;                 // coarse grid on the projected dimensions; eps2, lo32, hi32, min_pts, n
    const GridParams *gtab;       // batched calls: parameters of every set (same key layout)
    const int64_t *set_off;       // batched calls: first point of every set
    int d;
    const T *pts;                 // sorted, n x DP
    const float *fpts;            // float rows of the filter: pts itself, or the copy of double input
    const uint32_t *perm;
    const uint32_t *cell_of;      // coarse cell of every sorted point
    const uint32_t *cell_start;
    const uint32_t *chunk_off;    // first 32-point chunk of each coarse cell
    const uint64_t *cell_key;
    const uint2 *ranges;
    uint8_t *core;
    uint8_t *cell_core;
    uint32_t *parent;
    uint32_t *comp_min;
    int32_t *labels;
    uint8_t *core_out;
    DevCounters *ctr;
    int n_all, n_half;
    uint8_t near[16];             // the pencils nearest first (n_all of them; the coarse grid has 9)
    // cells left to the tensor-core kernels (float input): those with at least tc_min[phase] rows
    // of a phase (counts, unions, labels; 0: none); cx = exclusive scan of the core flags, for
    // the per-cell core counts; tc_hook: listed edges joined in cells whose unions run there too
    uint32_t tc_min[3];
    uint32_t tc_hook;
    uint32_t tc_handoff;  // open count rows at which a tensor-core chunk hands over
    const uint32_t *cx;
    // rows the tensor-core count handed over: count so far and candidate-stream position
    uint32_t *tc_cnt;
    uint32_t *tc_pos;
    // per coarse cell, the smallest and largest coordinate of its points in every dimension
    // (DP values each, of the type of the rows that the pair tests read): a point farther than
    // eps from a cell's box is farther than eps from every point of the cell
    T *box_lo;
    T *box_hi;
    // windows of long candidate streams (k_count_hd, k_labels_hd): the queue (chunk, window |
    // windows << 16), the windows of a chunk not yet done, and per row the count so far (counts)
    // or the smallest cluster id so far (labels)
    uint2 *sp_queue;
    uint32_t *sp_pending;
    uint32_t *sp_val;
    uint32_t sp_cap;
    // neighbour lists: entry i < min(nl_cnt[p], nl_k) of point p at nl[p * nl_k + i] is a point
    // within eps of p, or with kListNear set one that only the exact predicate can tell; nl_cnt
    // counts all that were found
    uint32_t *nl;
    uint32_t *nl_cnt;
    uint32_t nl_k;
    // after the lists are joined: the tree of most of a cell's core points (kNoRoot: no core
    // point; kMixedRoot: too mixed for one), the core points of other trees per cell, and which
    // points of every 32-point chunk they are
    uint32_t *cell_root;
    uint32_t *odd_cnt;
    uint32_t *odd_mask;
};

constexpr uint32_t kNoRoot = 0xffffffffu, kMixedRoot = 0xfffffffeu;
constexpr uint32_t kListNear = 0x80000000u;
// Most list entries: MINPTS up to kListMax + 1 has its labels from the lists.  The limit is one of memory,
// 80 bytes a point for the MINPTS of up to 20 that the workloads use.  With 32 entries (128 bytes)
// calls of MINPTS 22 gain what those of 21 have (9-D, 200,003 points 3.06 -> 2.48 ms, 16-D, a million
// 3.07 -> 2.61, 7-D double, 60,007 1.51 -> 1.01), those of up to 20 nothing; with 12 calls of MINPTS 20
// lose it (2.36 -> 2.97, 2.57 -> 3.17, 0.97 -> 1.49).
constexpr uint32_t kListMax = 20;

// List entries per point for the largest MINPTS of a call: MINPTS - 1 (a non-core point has no
// more neighbours), at least 8 (with only the three or four of a small MINPTS the joined lists
// leave many small trees), a multiple of 4 (16-byte loads).
inline uint32_t list_len(uint32_t min_pts) {
    uint32_t k = min_pts > 1 ? min_pts - 1 : 1;
    k = k < 8 ? 8 : k > kListMax ? kListMax : k;
    return (k + 3u) & ~3u;
}

// The lists take the space of the pencil table or hash (table_bytes, at least 24 bytes a point), which is
// free once the neighbour ranges are known, and more where they need it.  Entries that fit without
// more: 4 or, from 32 bytes a point on, 8.  Without memory for the whole lists a call runs with
// those (labels by comparison for MINPTS above 5 or 9): 16-D clusters of a million points, MINPTS 20,
// 2.44 -> 2.96 ms, 128 sets of mixed dimension 5.20 -> 6.00 (with no list at all 5.34 and 7.85).
inline uint32_t list_len_within(uint32_t min_pts, size_t table_bytes, int64_t n) {
    const size_t fit = table_bytes / (sizeof(uint32_t) * (size_t)n) & ~(size_t)3;
    const uint32_t k = list_len(min_pts);
    return fit < k ? (uint32_t)fit : k;
}

// A chunk scans the first kSpillWin candidates of its stream itself; what is left of a longer
// stream goes to a queue in windows of that many (at most kSpillMax, then wider ones), which a
// second launch hands to all warps.  Without it the few chunks of border and noise points next
// to a large cluster, whose rows scan the whole neighbourhood (20,000 points and more) 32
// candidates per round of loads, set the time of the pass alone.
constexpr uint32_t kSpillWin = 1024;
constexpr uint32_t kSpillMax = 64;

constexpr int kHdWarps = 4;     // warps per block in the point kernels of this path (default)
constexpr int kHdMaxWarps = 8;  // most warps per block a tuning may choose

// dist(a, q) <= eps with a in shared memory and q in registers (same exact predicate and FP32
// guard band as the hypercube path; summation in dimension order).
template <int DP>
__device__ __forceinline__ bool hd_within(const float *a, const float (&q)[DP], const GridParams &g) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < DP; i += 4) {
        // the sum of squares only grows (fma of a square into a non-negative sum rounds to at
        // least the sum), so a partial sum above hi32 already decides the pair: when every
        // lane of the warp is there, the rest of the dimensions are skipped
        if (i == DP / 2 && s > g.hi32) return false;
        const float4 av = *reinterpret_cast<const float4 *>(a + i);
        float t = __fsub_rn(av.x, q[i]);     s = __fmaf_rn(t, t, s);
        t = __fsub_rn(av.y, q[i + 1]);       s = __fmaf_rn(t, t, s);
        t = __fsub_rn(av.z, q[i + 2]);       s = __fmaf_rn(t, t, s);
        t = __fsub_rn(av.w, q[i + 3]);       s = __fmaf_rn(t, t, s);
    }
    if (s < g.lo32) return true;
    if (s > g.hi32) return false;
    double e = 0.0;
#pragma unroll
    for (int i = 0; i < DP; ++i) {
        const double t = __dsub_rn((double)a[i], (double)q[i]);
        e = __dadd_rn(e, __dmul_rn(t, t));
    }
    return e <= g.eps2;
}
template <int DP>
__device__ __forceinline__ bool hd_within(const double *a, const double (&q)[DP], const GridParams &g) {
    double e = 0.0;
#pragma unroll
    for (int i = 0; i < DP; ++i) {
        const double t = __dsub_rn(a[i], q[i]);
        e = __dadd_rn(e, __dmul_rn(t, t));
    }
    return e <= g.eps2;
}

// True when the point a (DP coordinates) is provably farther than eps from every point of the
// box [lo, hi]: the squared distance to the box, sum_i max(lo_i - a_i, a_i - hi_i, 0)^2, is a
// lower bound of the squared distance to any point inside.  float: summed in FP32 (each term
// and the sum within (DP + 2) 2^-24 of exact) against hi32 = eps^2 (1 + 2^-16) rounded up, so a
// box it calls far is farther than eps in exact arithmetic and in the FP64 predicate (when the
// FP32 filter is off, hi32 is infinite and no box is called far); double: summed in FP64
// against eps^2 (1 + 2^-40).
template <int DP>
__device__ __forceinline__ bool box_far(const float *a, const float *lo, const float *hi, const GridParams &g) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < DP; i += 4) {
        const float4 av = *reinterpret_cast<const float4 *>(a + i);
        const float4 l = ld(reinterpret_cast<const float4 *>(lo + i));
        const float4 h = ld(reinterpret_cast<const float4 *>(hi + i));
        float t = fmaxf(fmaxf(__fsub_rn(l.x, av.x), __fsub_rn(av.x, h.x)), 0.f); s = __fmaf_rn(t, t, s);
        t = fmaxf(fmaxf(__fsub_rn(l.y, av.y), __fsub_rn(av.y, h.y)), 0.f);       s = __fmaf_rn(t, t, s);
        t = fmaxf(fmaxf(__fsub_rn(l.z, av.z), __fsub_rn(av.z, h.z)), 0.f);       s = __fmaf_rn(t, t, s);
        t = fmaxf(fmaxf(__fsub_rn(l.w, av.w), __fsub_rn(av.w, h.w)), 0.f);       s = __fmaf_rn(t, t, s);
    }
    return s > g.hi32;
}
template <int DP>
__device__ __forceinline__ bool box_far(const double *a, const double *lo, const double *hi, const GridParams &g) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < DP; ++i) {
        const double t = fmax(fmax(__dsub_rn(ld(lo + i), a[i]), __dsub_rn(a[i], ld(hi + i))), 0.0);
        s = __fma_rn(t, t, s);
    }
    return s > g.eps2 * (1.0 + 0x1p-40);
}

template <typename T, int DP>
__device__ __forceinline__ void hd_load(const T *pts, uint32_t j, bool valid, T (&q)[DP]) {
    if (sizeof(T) == 4) {
        const float4 *src = reinterpret_cast<const float4 *>(pts + (uint64_t)j * DP);
#pragma unroll
        for (int i = 0; i < DP / 4; ++i) {
            const float4 v4 = valid ? src[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            q[4 * i] = v4.x; q[4 * i + 1] = v4.y; q[4 * i + 2] = v4.z; q[4 * i + 3] = v4.w;
        }
    } else {
        const double2 *src = reinterpret_cast<const double2 *>(pts + (uint64_t)j * DP);
#pragma unroll
        for (int i = 0; i < DP / 2; ++i) {
            const double2 v2 = valid ? src[i] : make_double2(0.0, 0.0);
            q[2 * i] = v2.x; q[2 * i + 1] = v2.y;
        }
    }
}

// The exact predicate on two sorted rows in global memory.
template <typename T, int DP>
__device__ __noinline__ bool hd_exact(const T *pts, uint32_t i, uint32_t j, double eps2) {
    const T *a = pts + (uint64_t)i * DP, *b = pts + (uint64_t)j * DP;
    double e = 0.0;
#pragma unroll 4
    for (int k = 0; k < DP; ++k) {
        const double t = __dsub_rn((double)ld_old(a + k), (double)ld_old(b + k));
        e = __dadd_rn(e, __dmul_rn(t, t));
    }
    return e <= eps2;
}

// One candidate point in registers against rows in shared memory.  FILTER: float coordinates in
// pairs (packed two-way FP32 subtract and multiply-add, half the instructions of the scalar
// form; the sum of squares of even and odd dimensions, within (DP + 2) 2^-24 of exact in any
// order), only the 4-coordinate groups that hold one of the d dimensions; else the exact
// predicate of the input type.
template <typename T, int DP, bool FILTER>
struct Candidate;

template <typename T, int DP>
struct Candidate<T, DP, true> {
    typedef float Row;
    unsigned long long q[DP / 2];
    uint32_t idx;
    static __device__ __forceinline__ const float *src(const HdView<T, DP> &v) { return v.fpts; }
    __device__ __forceinline__ void load(const HdView<T, DP> &v, uint32_t j, bool valid) {
        idx = j;
        const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(v.fpts + (uint64_t)(valid ? j : 0u) * DP);
#pragma unroll
        for (int i = 0; i < DP / 4; ++i) {
            if (4 * i >= v.d) break;
            const ulonglong2 x = ld_old(p + i);
            q[2 * i] = x.x;
            q[2 * i + 1] = x.y;
        }
    }
    __device__ __forceinline__ bool within(const HdView<T, DP> &v, const float *row, uint32_t ri, const GridParams &g) const {
        unsigned long long s2 = 0ull;
        const ulonglong2 *a = reinterpret_cast<const ulonglong2 *>(row);
#pragma unroll
        for (int i = 0; i < DP / 4; ++i) {
            if (4 * i >= v.d) break;
            const ulonglong2 x = a[i];
            unsigned long long t;
            asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(x.x), "l"(q[2 * i]));
            asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(s2) : "l"(t));
            asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(x.y), "l"(q[2 * i + 1]));
            asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(s2) : "l"(t));
        }
        const float s = __uint_as_float((uint32_t)s2) + __uint_as_float((uint32_t)(s2 >> 32));
        if (s > g.hi32) return false;
        if (s < g.lo32) return true;
        return hd_exact<T, DP>(v.pts, ri, idx, g.eps2);
    }
};

template <typename T, int DP>
struct Candidate<T, DP, false> {
    typedef T Row;
    T q[DP];
    static __device__ __forceinline__ const T *src(const HdView<T, DP> &v) { return v.pts; }
    __device__ __forceinline__ void load(const HdView<T, DP> &v, uint32_t j, bool valid) {
        hd_load<T, DP>(v.pts, j, valid, q);
    }
    __device__ __forceinline__ bool within(const HdView<T, DP> &, const T *row, uint32_t, const GridParams &g) const {
        return hd_within<DP>(row, q, g);
    }
};

// The boxes that go with those rows.
template <bool FILTER, int DP>
__device__ __forceinline__ bool cell_far(const HdView<float, DP> &v, const float *row, uint32_t B, const GridParams &g) {
    return box_far<DP>(row, v.box_lo + (uint64_t)B * DP, v.box_hi + (uint64_t)B * DP, g);
}
template <bool FILTER, int DP>
__device__ __forceinline__ bool cell_far(const HdView<double, DP> &v, const typename Candidate<double, DP, FILTER>::Row *row,
                                         uint32_t B, const GridParams &g) {
    typedef typename Candidate<double, DP, FILTER>::Row R;
    const R *lo = reinterpret_cast<const R *>(v.box_lo), *hi = reinterpret_cast<const R *>(v.box_hi);
    return box_far<DP>(row, lo + (uint64_t)B * DP, hi + (uint64_t)B * DP, g);
}

// Declared extents of a plan against the measured ones (complement of the encoded min of dimension
// i of set s at mm[s * 64 + i], encoded max at mm[(nsets + s) * 64 + i]; boxes: mins [s * d + i], maxes
// [(nsets + s) * d + i]): a point outside its box, or a NaN, sets status bit kErrBox.
static __global__ void __launch_bounds__(256) k_box_check_hd(const double *boxes, int nsets, int d,
                                                            const int64_t *set_off,
                                                            const unsigned long long *mm,
                                                            DevCounters *ctr) {
    pdl_enter();
    if (blockIdx.x == 0 && threadIdx.x == 0 && ctr->nan_seen) atomicOr(&ctr->status, kErrBox);
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < (int64_t)nsets * d;
         k += (int64_t)gridDim.x * blockDim.x) {
        const int set = (int)(k / d), i = (int)(k % d);
        if (set_off && set_off[set + 1] == set_off[set]) continue;
        const double lo = dec_double_dev(~mm[(size_t)set * 64 + i]);
        const double hi = dec_double_dev(mm[((size_t)nsets + set) * 64 + i]);
        if (lo < boxes[(size_t)set * d + i] || hi > boxes[((size_t)nsets + set) * d + i])
            atomicOr(&ctr->status, kErrBox);
    }
}

// Per-dimension min / max of row-major n x d input (origin shift, Sec. 2).  Each thread keeps
// one dimension (the stride is a multiple of d).
template <typename T>
__global__ void __launch_bounds__(256) k_minmax_rt(const T *__restrict__ in, int64_t n, int d, DevCounters *ctr,
                                                  unsigned long long *mm /* [2 * 64] */) {
    pdl_enter();
    // each thread walks one dimension (a stride that is a multiple of d), four independent
    // loads in flight; the block folds its threads per dimension in shared memory, then one
    // global atomic per block and dimension
    __shared__ unsigned long long smn[64], smx[64];
    __shared__ int snan;
    for (int i = threadIdx.x; i < 64; i += blockDim.x) {
        smn[i] = 0ull;  // complements of minima, so that both grow from 0
        smx[i] = 0ull;
    }
    if (threadIdx.x == 0) snan = 0;
    __syncthreads();
    const int64_t total = n * d;
    const int64_t threads = (int64_t)gridDim.x * blockDim.x;
    const int64_t stride = (threads / d) * d;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (tid < stride) {
        T mn[4], mx[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            mn[u] = sizeof(T) == 4 ? (T)FLT_MAX : (T)DBL_MAX;
            mx[u] = -mn[u];
        }
        bool nan = false;
        int64_t e = tid;
        for (; e + 3 * stride < total; e += 4 * stride) {
            T x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = ld_old(in + e + u * stride);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                nan |= (x[u] != x[u]);
                mn[u] = x[u] < mn[u] ? x[u] : mn[u];
                mx[u] = x[u] > mx[u] ? x[u] : mx[u];
            }
        }
        for (; e < total; e += stride) {
            const T x = ld_old(in + e);
            nan |= (x != x);
            mn[0] = x < mn[0] ? x : mn[0];
            mx[0] = x > mx[0] ? x : mx[0];
        }
#pragma unroll
        for (int u = 1; u < 4; ++u) {
            mn[0] = mn[u] < mn[0] ? mn[u] : mn[0];
            mx[0] = mx[u] > mx[0] ? mx[u] : mx[0];
        }
        const int dim = (int)(tid % d);
        atomicMax(&smn[dim], ~(unsigned long long)enc_double((double)mn[0]));
        atomicMax(&smx[dim], (unsigned long long)enc_double((double)mx[0]));
        if (nan) snan = 1;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < d; i += blockDim.x) {
        if (smn[i] != 0ull) atomicMax(&mm[i], smn[i]);
        if (smx[i] != 0ull) atomicMax(&mm[64 + i], smx[i]);
    }
    if (threadIdx.x == 0 && snan) atomicOr(&ctr->nan_seen, 1u);
}

// Digit counts of every radix pass, gathered per block in shared memory (h, cleared by the block).
__device__ __forceinline__ void count_digits_begin(uint32_t (&h)[8][256]) {
    for (int i = threadIdx.x; i < 8 * 256; i += blockDim.x) (&h[0][0])[i] = 0;
    __syncthreads();
}
__device__ __forceinline__ void count_digits(uint32_t (&h)[8][256], uint64_t key, int passes) {
    for (int p = 0; p < passes; ++p) atomicAdd(&h[p][(uint32_t)(key >> (8 * p)) & 0xffu], 1u);
}
__device__ __forceinline__ void count_digits_end(uint32_t (&h)[8][256], int passes, uint32_t *digit_counts) {
    __syncthreads();
    for (int i = threadIdx.x; i < passes * 256; i += blockDim.x) {
        const uint32_t c = (&h[0][0])[i];
        if (c) atomicAdd(&digit_counts[i], c);
    }
}

// Coarse cell keys from the three projected dimensions (Algorithm 1 on a grid of side >= eps),
// with the radix digit counts of the sort that follows.
template <typename T, typename K>
__global__ void __launch_bounds__(256) k_bin_proj(const T *__restrict__ in, int d, int3 sel, GridParams g,
                                                 K *__restrict__ keys, uint32_t *__restrict__ digit_counts,
                                                 FillList fill) {
    pdl_enter();
    __shared__ uint32_t h[8][256];
    fill_regions(fill);
    count_digits_begin(h);
    const int passes = (g.key_bits + 7) / 8;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < g.n;
         j += (int64_t)gridDim.x * blockDim.x) {
        const int dims[3] = {sel.x, sel.y, sel.z};
        uint64_t key = 0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double t = __dmul_rn(__dsub_rn((double)ld_old(in + j * d + dims[i]), g.origin[i]), g.inv_side);
            uint32_t c = (uint32_t)floor(t);
            if (c > g.ncell[i] - 1) c = g.ncell[i] - 1;
            key |= (uint64_t)c << g.shift[i];
        }
        keys[j] = (K)key;
        count_digits(h, key, passes);
    }
    count_digits_end(h, passes, digit_counts);
}

// Gather the points into cell order, padded to DP coordinates, and the coarse cells and pencils; one
// block per tile of kScanTileElems rows, DP / 4 threads per row (four coordinates each, one vector
// store).  Also clears the core flags of the points and cells, and with fpts (double input with the
// filter on) writes the float copy of the rows, relative to the set's smallest coordinates (set
// id above set_shift of the key; complements of their encodings at mm[set * 64 + i]).
template <typename T, int DP, typename K>
__global__ void __launch_bounds__(kTileThreads) k_cells_hd(const T *__restrict__ in, int d, CellsArgs<K> a,
                                                          T *__restrict__ pts, uint8_t *__restrict__ core,
                                                          uint8_t *__restrict__ cell_core, float *__restrict__ fpts,
                                                          const unsigned long long *mm, int set_shift) {
    pdl_enter();
    constexpr int G = DP / 4;          // threads per row
    constexpr int R = 256 / G;         // rows per step of the block
    const int g = threadIdx.x % G, r0 = threadIdx.x / G;
    bool ok;
    const uint32_t tile = take_tile(a.l, 0u, &a.ctr->status, ok);
    const int64_t base = (int64_t)tile * kScanTileElems;
    if (!ok) {  // (what follows looks at the flags of all points)
        for (int64_t j = base + threadIdx.x; j < min(base + kScanTileElems, a.n); j += kTileThreads) core[j] = 0;
        return;
    }
    cells_tile(a, tile, [&]() {
#pragma unroll 4
        for (int k = 0; k < kScanTileElems / R; ++k) {
            const int64_t j = base + (int64_t)k * R + r0;
            if (j >= a.n) break;
            const uint32_t o = a.idx[j];
            const T *src = in + (int64_t)o * d;
            T x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = 4 * g + u < d ? ld_old(src + 4 * g + u) : T(0);
            T *dst = pts + j * DP + 4 * g;
            if (sizeof(T) == 4) {
                *reinterpret_cast<float4 *>(dst) = make_float4((float)x[0], (float)x[1], (float)x[2], (float)x[3]);
            } else {
                reinterpret_cast<double2 *>(dst)[0] = make_double2((double)x[0], (double)x[1]);
                reinterpret_cast<double2 *>(dst)[1] = make_double2((double)x[2], (double)x[3]);
                if (fpts) {
                    const uint64_t set = set_shift < 64 ? (uint64_t)a.keys[j] >> set_shift : 0ull;
                    float f[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        f[u] = 4 * g + u < d ? (float)__dsub_rn((double)x[u], dec_double_dev(~ld_old(mm + set * 64 + 4 * g + u))) : 0.f;
                    *reinterpret_cast<float4 *>(fpts + j * DP + 4 * g) = make_float4(f[0], f[1], f[2], f[3]);
                }
            }
            if (g == 0) core[j] = 0;
        }
    }, [cell_core](uint32_t c) { cell_core[c] = 0; });
}

template <typename T, int DP>
__device__ __forceinline__ void stage_rows(T *rows, const T *pts, uint32_t base, uint32_t e) {
    // rows: 32 x DP for this warp; lane L copies row L
    const int lane = threadIdx.x & 31;
    const uint32_t i = base + lane;
    T q[DP];
    hd_load<T, DP>(pts, i, i < e, q);
    if (sizeof(T) == 4) {
        float4 *dst = reinterpret_cast<float4 *>(rows + lane * DP);
#pragma unroll
        for (int k = 0; k < DP / 4; ++k)
            dst[k] = make_float4((float)q[4 * k], (float)q[4 * k + 1], (float)q[4 * k + 2], (float)q[4 * k + 3]);
    } else {
#pragma unroll
        for (int k = 0; k < DP; ++k) rows[lane * DP + k] = q[k];
    }
    __syncwarp();
}

// Work is scheduled in chunks of 32 consecutive points of one coarse cell (a coarse cell can
// hold a whole cluster, so one warp per cell would leave the largest cell to a single warp).
// chunk_off[c] = first chunk of cell c (exclusive scan of ceil(size / 32)).
// The scan also clears the cell's box (codes; see BoxCode).
template <typename V>
struct ChunkCount {
    V v;
    __device__ uint32_t operator()(int64_t c) const { return (v.cell_start[c + 1] - v.cell_start[c] + 31u) / 32u; }
};

// Cell of chunk (or work item) t: the last c with off[c] <= t, by a 32-way search (one round of
// loads per level instead of one per halving).  A full warp calls it; every lane returns the
// result.
__device__ __forceinline__ uint32_t chunk_cell(const uint32_t *off, uint32_t C, uint32_t t) {
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t lo = 0, hi = C;  // off[lo] <= t, and off[hi] > t unless hi == C
    while (hi - lo > 1u) {
        const uint32_t step = (hi - lo + 31u) >> 5;
        const uint32_t piv = lo + lane * step;
        const unsigned ok = __ballot_sync(0xffffffffu, piv < hi && ld(off + piv) <= t);
        lo += (uint32_t)(31 - __clz(ok)) * step;  // the ok lanes are a prefix (off is nondecreasing)
        hi = min(hi, lo + step);
    }
    return lo;
}

// Box of every coarse cell: cleared by the scan of the chunk counts, accumulated over 32-point
// chunks (one warp per chunk, so a large cell is spread over many warps), decoded.  Coordinates are
// accumulated as order-preserving unsigned integers (sign bit flipped for x >= 0, every bit
// for x < 0), so min / max of the codes is min / max of the values and the warps of one cell
// combine with atomicMin / atomicMax.
template <typename T>
struct BoxCode {
    typedef typename std::conditional<sizeof(T) == 4, uint32_t, unsigned long long>::type U;
    static __device__ __forceinline__ U enc(T x) {
        if (sizeof(T) == 4) {
            const uint32_t u = __float_as_uint((float)x);
            return (U)(u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u));
        } else {
            const unsigned long long u = (unsigned long long)__double_as_longlong((double)x);
            return (U)(u ^ ((unsigned long long)((long long)u >> 63) | 0x8000000000000000ull));
        }
    }
    static __device__ __forceinline__ T dec(U c) {
        if (sizeof(T) == 4) {
            const uint32_t u = (uint32_t)c;
            return (T)__uint_as_float(u ^ ((u >> 31) ? 0x80000000u : 0xffffffffu));
        } else {
            const unsigned long long u = (unsigned long long)c;
            return (T)__longlong_as_double((long long)(u ^ ((u >> 63) ? 0x8000000000000000ull : ~0ull)));
        }
    }
    static __device__ __forceinline__ U warp_min(U v) {
        if (sizeof(T) == 4) return (U)__reduce_min_sync(0xffffffffu, (uint32_t)v);
        for (int o = 16; o; o >>= 1) {
            const U t = __shfl_xor_sync(0xffffffffu, v, o);
            v = t < v ? t : v;
        }
        return v;
    }
    static __device__ __forceinline__ U warp_max(U v) {
        if (sizeof(T) == 4) return (U)__reduce_max_sync(0xffffffffu, (uint32_t)v);
        for (int o = 16; o; o >>= 1) {
            const U t = __shfl_xor_sync(0xffffffffu, v, o);
            v = t > v ? t : v;
        }
        return v;
    }
};

template <typename T, int DP, typename R>
struct BoxClear {
    HdView<T, DP> v;
    __device__ void operator()(int64_t c, uint32_t, uint32_t) const {
        uint4 *lo = reinterpret_cast<uint4 *>(reinterpret_cast<R *>(v.box_lo) + c * DP);
        uint4 *hi = reinterpret_cast<uint4 *>(reinterpret_cast<R *>(v.box_hi) + c * DP);
#pragma unroll
        for (int i = 0; i < DP * (int)sizeof(R) / 16; ++i) {
            lo[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
            hi[i] = make_uint4(0u, 0u, 0u, 0u);
        }
    }
};

template <typename T, int DP, typename R>
__global__ void __launch_bounds__(256) k_cell_box_hd(HdView<T, DP> v) {
    pdl_enter();
    typedef BoxCode<R> BC;
    typedef typename BC::U U;
    constexpr int E = DP > 32 ? DP / 32 : 1;  // dimensions per lane in the atomics
    const int lane = lane_id();
    const uint32_t C = v.ctr->n_cells, NC = unless_failed(v.ctr, v.ctr->n_chunks);
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
    U *lo = reinterpret_cast<U *>(v.box_lo), *hi = reinterpret_cast<U *>(v.box_hi);
    const R *pts = sizeof(R) == sizeof(T) ? reinterpret_cast<const R *>(v.pts) : reinterpret_cast<const R *>(v.fpts);
    for (uint32_t t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < NC; t += warps) {
        const uint32_t A = chunk_cell(v.chunk_off, C, t);
        const uint32_t e = v.cell_start[A + 1], base = v.cell_start[A] + 32u * (t - v.chunk_off[A]);
        const uint32_t p = base + lane;
        const bool valid = p < e;
        U mn[E], mx[E];
#pragma unroll
        for (int k = 0; k < E; ++k) {
            mn[k] = ~(U)0;
            mx[k] = (U)0;
        }
#pragma unroll
        for (int g0 = 0; g0 < DP; g0 += 4) {
            R x[4];
            if (sizeof(R) == 4) {
                const float4 f = valid ? ld_old(reinterpret_cast<const float4 *>(pts + (uint64_t)p * DP + g0))
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
                x[0] = (R)f.x; x[1] = (R)f.y; x[2] = (R)f.z; x[3] = (R)f.w;
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) x[i] = valid ? ld_old(pts + (uint64_t)p * DP + g0 + i) : (R)0;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const U c = BC::enc(x[i]);
                const U a = BC::warp_min(valid ? c : ~(U)0);
                const U b = BC::warp_max(valid ? c : (U)0);
                if (lane == ((g0 + i) & 31)) {
                    mn[(g0 + i) >> 5] = a;
                    mx[(g0 + i) >> 5] = b;
                }
            }
        }
        if (lane < DP) {
#pragma unroll
            for (int k = 0; k < E; ++k) {
                atomicMin(lo + (uint64_t)A * DP + lane + 32 * k, mn[k]);
                atomicMax(hi + (uint64_t)A * DP + lane + 32 * k, mx[k]);
            }
        }
    }
}

template <typename T, int DP, typename R>
__global__ void __launch_bounds__(256) k_cell_box_decode(HdView<T, DP> v) {
    pdl_enter();
    typedef BoxCode<R> BC;
    typedef typename BC::U U;
    const uint64_t m = (uint64_t)unless_failed(v.ctr, v.ctr->n_cells) * DP;
    U *lo = reinterpret_cast<U *>(v.box_lo), *hi = reinterpret_cast<U *>(v.box_hi);
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m; i += (uint64_t)gridDim.x * blockDim.x) {
        reinterpret_cast<R *>(lo)[i] = BC::dec(lo[i]);
        reinterpret_cast<R *>(hi)[i] = BC::dec(hi[i]);
    }
}

#define HD_FOR_EACH_CHUNK(v, A, base, e, slot)                                                \
    const uint32_t C_ = (v).ctr->n_cells, NC_ = unless_failed((v).ctr, (v).ctr->n_chunks);   \
    for (uint32_t t_ = next_chunk(&(v).ctr->hd_next[slot]); t_ < NC_;                        \
         t_ = next_chunk(&(v).ctr->hd_next[slot]))                                           \
        for (uint32_t A = chunk_cell((v).chunk_off, C_, t_), once_ = 1; once_; once_ = 0)    \
            for (uint32_t e = (v).cell_start[A + 1],                                         \
                          base = (v).cell_start[A] + 32u * (t_ - (v).chunk_off[A]), o2_ = 1; \
                 o2_; o2_ = 0)

// Candidate stream of a cell: spans of cells laid end to end, the cell itself first, then the rest of
// its pencil, then the other pencils nearest first.  Points within eps differ by a fraction of
// eps in each projected coordinate, so nearly half of a point's neighbours are in its own cell
// (9-D clusters: 44%, in a twentieth of the candidates) and a core point reaches MINPTS early.
constexpr int kSpansExtra = 2;  // spans beyond one per pencil
template <typename V>
__device__ __forceinline__ uint2 stream_span(const V &v, uint32_t A, int k) {
    if (k >= v.n_all + kSpansExtra) return make_uint2(0u, 0u);
    const uint2 rg = v.ranges[(uint64_t)A * v.n_all + (k < 3 ? 0 : v.near[k - 2])];
    return k == 0 ? make_uint2(A, A + 1) : k == 1 ? make_uint2(rg.x, A) : k == 2 ? make_uint2(A + 1, rg.y) : rg;
}

// Its length, from one span per lane.
template <typename V>
__device__ __forceinline__ uint32_t stream_length(const V &v, uint2 rg) {
    return __reduce_add_sync(0xffffffffu, rg.x < rg.y ? v.cell_start[rg.y] - v.cell_start[rg.x] : 0u);
}

// The cells of the part [p0, p1) of that stream, in order: f(B, q0, q1) for the points
// [q0, q1) of cell B.  f returns false to stop.  Warp-uniform.
template <typename V, typename F>
__device__ __forceinline__ void for_stream_cells(const V &v, uint2 rg, uint32_t p0, uint32_t p1, F f) {
    uint32_t pos = 0;
    for (int kk = 0; kk < v.n_all + kSpansExtra; ++kk) {
        const uint32_t lo = __shfl_sync(0xffffffffu, rg.x, kk);
        const uint32_t hi = __shfl_sync(0xffffffffu, rg.y, kk);
        if (lo >= hi) continue;
        const uint32_t s0 = v.cell_start[lo], s1 = v.cell_start[hi];
        if (pos + (s1 - s0) <= p0) {
            pos += s1 - s0;
            continue;
        }
        uint32_t q0 = s0;
        for (uint32_t B = lo; B < hi; ++B) {
            const uint32_t q1 = B + 1 < hi ? v.cell_start[B + 1] : s1;
            const uint32_t a = pos, b = pos + (q1 - q0);  // stream positions of the cell
            if (a >= p1) return;
            if (b > p0 && !f(B, q0 + (p0 > a ? p0 - a : 0u), q1 - (b > p1 ? b - p1 : 0u))) return;
            pos = b;
            q0 = q1;
        }
    }
}

// The window of a chunk's remaining stream [start, total) that entry (chunk, w | nw << 16) of the
// queue stands for.
__device__ __forceinline__ void spill_window(uint32_t entry, uint32_t start, uint32_t total, uint32_t &p0, uint32_t &p1) {
    const uint32_t w = entry & 0xffffu, nw = entry >> 16;
    const uint32_t step = ((total - start + nw - 1u) / nw + 31u) & ~31u;
    p0 = min(total, start + w * step);
    p1 = min(total, p0 + step);
}

// Queue the windows of [start, total) for chunk t; false when the queue is full (the caller then
// scans on by itself).  sp_val of the chunk's rows is written by the caller beforehand.
template <typename V>
__device__ __forceinline__ bool spill_push(const V &v, int slot, uint32_t t, uint32_t start, uint32_t total) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t nw = min(kSpillMax, (total - start + kSpillWin - 1u) / kSpillWin);
    uint32_t at = 0;
    if (lane == 0) {  // (a full queue's counter is left alone, so it cannot wrap)
        at = *(volatile uint32_t *)&v.ctr->hd_spill[slot];
        if (at < v.sp_cap) at = atomicAdd(&v.ctr->hd_spill[slot], nw);
    }
    at = __shfl_sync(0xffffffffu, at, 0);
    const bool fits = at < v.sp_cap && nw <= v.sp_cap - at;
    for (uint32_t w = lane; w < nw; w += 32)  // a reservation cut off by the end is marked empty
        if (at < v.sp_cap && w < v.sp_cap - at) v.sp_queue[at + w] = make_uint2(fits ? t : 0xffffffffu, w | nw << 16);
    if (fits && lane == 0) v.sp_pending[t] = nw;
    return fits;
}

// Definition 2: |N_eps(p)| >= MINPTS, counted over the 27 neighbouring coarse cells (the own
// point included), stopping once every point of the chunk has reached MINPTS.  The chunk's
// points are staged in shared memory, candidates stream through the lanes, and each open
// point is compared with a warp ballot.
//
// Bound by the latency of its loads: a warp has one round of candidate loads in flight, so the
// time is the longest item of a warp.  Windows (SPILL = true: the second launch) bring the
// longest item down to kSpillWin candidates (9-D call of 200,003 points 4.04 -> 3.50 ms).  The
// filter on packed float pairs takes the double-precision call of 60,007 7-D points, whose
// pair tests were bound by the FP64 rate, from 7.4 to 0.95 ms together with the lists.
template <typename T, int DP, bool SPILL, bool FILTER>
__global__ void __launch_bounds__(32 * kHdMaxWarps) k_count_hd(HdView<T, DP> v) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typedef Candidate<T, DP, FILTER> Cand;
    typedef typename Cand::Row R;
    R *rows = reinterpret_cast<R *>(smem_raw) + (threadIdx.x >> 5) * 32 * DP;
    const int lane = lane_id();
    uint32_t chunks = 0;
    const uint32_t C = v.ctr->n_cells, N = unless_failed(v.ctr, SPILL ? min(v.ctr->hd_spill[0], v.sp_cap) : v.ctr->n_chunks);
    ItemQueue items(SPILL ? &v.ctr->hd_spill_next[0] : &v.ctr->hd_next[0], N);
    while (items.next()) {
        const uint32_t item = items.cur;
        const uint2 entry = SPILL ? v.sp_queue[item] : make_uint2(item, 0u);
        if (SPILL && entry.x == 0xffffffffu) continue;
        const uint32_t t = entry.x, A = chunk_cell(v.chunk_off, C, t);
        const uint32_t e = v.cell_start[A + 1], base = v.cell_start[A] + 32u * (t - v.chunk_off[A]);
        const uint32_t p = base + lane;
        // a cell counted on the tensor cores leaves here only the rows it handed over (core = 2)
        const bool tc_cell = v.tc_min[0] && e - v.cell_start[A] >= v.tc_min[0];
        const bool have = p < e && (!tc_cell || v.core[p] == 2);
        const unsigned rows_m = __ballot_sync(0xffffffffu, have);
        if (!rows_m) continue;
        const GridParams &G = params_of(v, set_of_key(v, v.cell_key[A]));
        const uint32_t min_pts = G.min_pts;
        const uint2 rg = stream_span(v, A, lane);
        const uint32_t total = stream_length(v, rg);
        // a row the tensor-core count handed over resumes where it stopped (same candidate order)
        const uint32_t start = tc_cell ? __shfl_sync(0xffffffffu, have ? v.tc_pos[p] : 0u, __ffs(rows_m) - 1) : 0u;
        uint32_t cnt = 0, p0 = start, p1 = start + min(kSpillWin, total - start);
        if (SPILL) {
            if (have) cnt = __ldcg(v.sp_val + p);
            spill_window(entry.y, p1, total, p0, p1);
        } else if (tc_cell && have) {
            cnt = v.tc_cnt[p];
        }
        unsigned open = __ballot_sync(0xffffffffu, have && (!SPILL || cnt < min_pts));
        if (open) stage_rows<R, DP>(rows, Cand::src(v), base, e);
        // one cell at a time: a cell whose box is farther than eps from every open row adds
        // nothing to their counts and is passed over
        auto scan = [&](uint32_t B, uint32_t q0, uint32_t q1) -> bool {
            const unsigned near = open & __ballot_sync(0xffffffffu,
                !cell_far<FILTER, DP>(v, rows + lane * DP, B, G));
            if (!near) return true;
            // two blocks of candidates per step (for wide rows one): the row's loads and the loop
            // around them serve both
            constexpr int NB = DP <= 16 ? 2 : 1;
            for (uint32_t qb = q0; qb < q1 && open; qb += 32 * NB) {
                Cand qv[NB];
                bool in[NB];
#pragma unroll
                for (int u = 0; u < NB; ++u) {
                    in[u] = qb + 32 * u + lane < q1;
                    qv[u].load(v, qb + 32 * u + lane, in[u]);
                }
                chunks += NB;
                unsigned rem = open & near;
                while (rem) {
                    const int jj = __ffs(rem) - 1;
                    rem &= rem - 1;
                    bool hit[NB];
                    unsigned hits[NB], any = 0;
#pragma unroll
                    for (int u = 0; u < NB; ++u) {
                        hit[u] = in[u] && qv[u].within(v, rows + jj * DP, base + jj, G);
                        hits[u] = __ballot_sync(0xffffffffu, hit[u]);
                        any |= hits[u];
                    }
                    if (!any) continue;
                    // the row's count, and its list entries from there on
                    uint32_t found = 0, at = 0;
#pragma unroll
                    for (int u = 0; u < NB; ++u) found += (uint32_t)__popc(hits[u]);
                    if (lane == jj) {
                        at = SPILL ? atomicAdd(v.sp_val + p, found) : cnt;
                        cnt = at + found;
                    }
                    at = __shfl_sync(0xffffffffu, at, jj);
#pragma unroll
                    for (int u = 0; u < NB; ++u) {
                        const uint32_t slot = at + (uint32_t)__popc(hits[u] & ((1u << lane) - 1u));
                        if (hit[u] && slot < v.nl_k) v.nl[(uint64_t)(base + jj) * v.nl_k + slot] = qb + 32 * u + lane;
                        at += (uint32_t)__popc(hits[u]);
                    }
                }
                open &= __ballot_sync(0xffffffffu, have && cnt < min_pts);
            }
            return open != 0;
        };
        if (open) for_stream_cells(v, rg, p0, p1, scan);
        bool decide = true;
        if (SPILL) {
            // the last window of the chunk decides its rows from the summed counts
            __threadfence();
            __syncwarp();
            uint32_t left = 0;
            if (lane == 0) left = atomicSub(v.sp_pending + t, 1u);
            decide = __shfl_sync(0xffffffffu, left, 0) == 1u;
            __threadfence();
            if (decide && have) cnt = __ldcg(v.sp_val + p);
        } else if (open && p1 < total) {
            if (have) v.sp_val[p] = cnt;
            decide = !spill_push(v, 0, t, p1, total);
            if (decide) for_stream_cells(v, rg, p1, total, scan);
        }
        if (decide) {
            const bool is_core = have && cnt >= min_pts;
            if (have) v.core[p] = is_core ? 1 : 0;
            if (have) v.nl_cnt[p] = cnt;
            if (__any_sync(0xffffffffu, is_core) && lane == 0) v.cell_core[A] = 1;
        }
        __syncwarp();
    }
    add_counter(&v.ctr->work[0], lane == 0 ? chunks : 0u);
}

// Four list entries of point p from entry i on.
template <typename V>
__device__ __forceinline__ uint4 list4(const V &v, uint32_t p, uint32_t i) {
    return ld(reinterpret_cast<const uint4 *>(v.nl + (uint64_t)p * v.nl_k + i));
}

// Union-find over points: every core point starts below the smallest core point on its list (an
// edge of the core graph to a smaller index, so the links form a forest inside the clusters),
// every other point is its own root.  With tc_hook = 0 only in the cells whose unions run on the
// CUDA cores.
template <typename T, int DP>
__global__ void __launch_bounds__(256) k_list_link(HdView<T, DP> v) {
    pdl_enter();
    // (the cells' trees and odd counts are cleared here too)
    const uint32_t C = unless_failed(v.ctr, v.ctr->n_cells);
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < C; c += gridDim.x * blockDim.x) {
        v.cell_root[c] = kNoRoot;
        v.odd_cnt[c] = 0u;
    }
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < v.g.n; j += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t p = (uint32_t)j;
        uint32_t m = p;
        bool use = v.core[p];
        if (use && v.tc_min[1] && !v.tc_hook) {
            const uint32_t A = v.cell_of[p];
            use = v.cx[v.cell_start[A + 1]] - v.cx[v.cell_start[A]] < v.tc_min[1];
        }
        if (use) {
            const uint32_t len = min(v.nl_cnt[p], v.nl_k);
            for (uint32_t i = 0; i < len; i += 4) {
                const uint4 e4 = list4(v, p, i);
                const uint32_t e[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)  // (a flagged entry is above every index)
                    if (i + u < len && e[u] < m && v.core[e[u]]) m = e[u];
            }
        }
        v.parent[p] = m;
        v.comp_min[p] = kNoLabel;
    }
}

// parent[p] = root of every core point (nothing hooks meanwhile).
template <typename T, int DP>
__global__ void __launch_bounds__(256) k_flatten_hd(HdView<T, DP> v) {
    pdl_enter();
    bool open = true;
    for (uint32_t round = 0; open; ++round) {
        open = false;
        for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < v.g.n; j += (int64_t)gridDim.x * blockDim.x)
            if (v.core[j] && !uf_shorten(v.parent, (uint32_t)j)) open = true;
        if (round > kLoopLimit) { set_error(v.ctr, kErrLoop); return; }
    }
}

// Four list entries of one point and its tree against theirs (k_list_hook, k_list_join): the tree
// nodes of the point (rp) and of the entries (r[u], rp itself where there is no edge).
template <typename V>
__device__ __forceinline__ void load_edges(const V &v, int64_t j, int64_t m, uint32_t &rp, uint32_t (&r)[4]) {
    const uint32_t quads = v.nl_k / 4;
    const uint32_t p = (uint32_t)(min(j, m - 1) / quads), i = 4u * (uint32_t)(j % quads);
    uint32_t len = j < m && v.core[p] ? min(v.nl_cnt[p], v.nl_k) : 0u;
    if (len > i && v.tc_min[1] && !v.tc_hook) {
        const uint32_t A = v.cell_of[p];
        if (v.cx[v.cell_start[A + 1]] - v.cx[v.cell_start[A]] >= v.tc_min[1]) len = 0u;
    }
    const uint4 e4 = len > i ? list4(v, p, i) : make_uint4(p, p, p, p);
    const uint32_t e[4] = {e4.x, e4.y, e4.z, e4.w};
    rp = __ldcg(v.parent + p);
    bool c[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const bool ok = i + u < len && !(e[u] & kListNear);
        const uint32_t q = ok ? e[u] : p;
        c[u] = ok && v.core[q];
        r[u] = __ldcg(v.parent + q);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (!c[u]) r[u] = rp;
}

// The other edges of the lists, one thread per four entries, in two passes.  The first puts every
// tree below the smallest tree that one of its edges leads to: one minimum per edge between two
// trees, nothing waited for, and of two minima on one root the larger is lost.  The second
// joins what that left.  Joining at once is bound by the roots that everybody wants: when it
// starts, the large trees have thousands of edges between them, and every one of them tries to
// hook the same root.
template <typename T, int DP>
__global__ void __launch_bounds__(256) k_list_hook(HdView<T, DP> v) {
    pdl_enter();
    const int64_t m = v.g.n * (v.nl_k / 4);
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        uint32_t rp, r[4];
        load_edges(v, j, m, rp, r);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t lo = min(rp, r[u]), hi = max(rp, r[u]);
            if (lo != hi && __ldcg(v.parent + hi) > lo) atomicMin(v.parent + hi, lo);
        }
    }
}

template <typename T, int DP>
__global__ void __launch_bounds__(256) k_list_join(HdView<T, DP> v) {
    pdl_enter();
    const uint32_t lane = lane_id();
    const int64_t m = v.g.n * (v.nl_k / 4);
    for (int64_t jb = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); jb < m; jb += (int64_t)gridDim.x * blockDim.x) {
        uint32_t rp, r[4];
        load_edges(v, jb + lane, m, rp, r);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            bool need = r[u] != rp;
            if (!__any_sync(0xffffffffu, need)) continue;
            if (need) {
                rp = uf_root_readonly(v.parent, rp, v.ctr);
                r[u] = uf_root_readonly(v.parent, r[u], v.ctr);
                need = r[u] != rp;
            }
            // the lanes with the same two roots leave the join to one of them
            const unsigned active = __ballot_sync(0xffffffffu, need);
            if (!need) continue;
            const uint32_t lo = min(rp, r[u]), hi = max(rp, r[u]);
            const unsigned same = __match_any_sync(active, (unsigned long long)hi << 32 | lo);
            if ((int)lane == __ffs(same) - 1) uf_join_readonly(v.parent, lo, hi, v.ctr);
        }
    }
}

// One edge for every pair of neighbouring cells (upper half) whose first core points are in
// different trees: the first 32 points of one against the first 32 of the other.  The lists
// of a dense cluster hold the first points of the stream, so they join its points along each
// pencil but hardly across pencils; between dense cells nearly every such sample has an edge.
template <typename T, int DP, bool FILTER>
__global__ void __launch_bounds__(32 * kHdMaxWarps) k_cell_link(HdView<T, DP> v) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typedef Candidate<T, DP, FILTER> Cand;
    typedef typename Cand::Row R;
    R *rows = reinterpret_cast<R *>(smem_raw) + (threadIdx.x >> 5) * 32 * DP;
    const int lane = lane_id();
    const uint64_t N = (uint64_t)unless_failed(v.ctr, v.ctr->n_cells) * v.n_half;  // one warp per cell and neighbour pencil
    for (uint64_t w = global_warp(); w < N; w += total_warps()) {
        const uint32_t A = (uint32_t)(w / v.n_half);
        const int kk = (int)(w % v.n_half);
        if (!v.cell_core[A]) continue;
        const uint2 rg = v.ranges[(uint64_t)A * v.n_all + kk];
        const uint32_t lo = kk == 0 ? A + 1 : rg.x;
        if (lo >= rg.y) continue;
        const uint32_t s = v.cell_start[A], e = min(v.cell_start[A + 1], s + 32u), p = s + lane;
        const bool pc = p < e && v.core[p];
        const unsigned amask = __ballot_sync(0xffffffffu, pc);
        if (!amask) continue;
        const uint32_t a0 = s + (uint32_t)__ffs(amask) - 1u;
        const GridParams &G = params_of(v, set_of_key(v, v.cell_key[A]));
        bool staged = false;
        for (uint32_t B = lo; B < rg.y; ++B) {
            if (!v.cell_core[B]) continue;
            const uint32_t q = v.cell_start[B] + lane;
            const bool qc = q < v.cell_start[B + 1] && v.core[q];
            const unsigned bmask = __ballot_sync(0xffffffffu, qc);
            if (!bmask) continue;
            uint32_t r = 0;  // the roots of the two first core points
            if (lane == 0) r = uf_find(v.parent, a0, v.ctr);
            if (lane == 1) r = uf_find(v.parent, v.cell_start[B] + (uint32_t)__ffs(bmask) - 1u, v.ctr);
            if (__shfl_sync(0xffffffffu, r, 0) == __shfl_sync(0xffffffffu, r, 1)) continue;
            if (!staged) stage_rows<R, DP>(rows, Cand::src(v), s, e);
            staged = true;
            Cand qv;
            qv.load(v, q, qc);
            unsigned rem = amask;
            while (rem) {
                const int jj = __ffs(rem) - 1;
                rem &= rem - 1;
                const unsigned hm = __ballot_sync(0xffffffffu, qc && qv.within(v, rows + jj * DP, s + jj, G));
                if (!hm) continue;
                if (lane == __ffs(hm) - 1) uf_union(v.parent, s + jj, q, v.ctr);
                break;
            }
        }
        __syncwarp();
    }
}

// The tree of a cell: the smallest root among its core points.  A tree's root is its smallest
// index, so the tree that spans a cluster has a smaller root than the small trees that the lists
// left over in the cluster's cells, and nearly all core points of a cell have this one; the
// others are the cell's odd points.
template <typename T, int DP>
__global__ void __launch_bounds__(256) k_cell_root(HdView<T, DP> v) {
    pdl_enter();
    const int lane = lane_id();
    const int64_t n = v.g.n;
    for (int64_t jb = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); jb < n; jb += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = jb + lane;
        const bool isc = j < n && v.core[j];
        const uint32_t r = isc ? v.parent[j] : 0xffffffffu, c = isc ? v.cell_of[j] : 0xffffffffu;
        // one atomic per cell of the warp's 32 consecutive points
        const unsigned peers = __match_any_sync(0xffffffffu, c);
        const uint32_t m = __reduce_min_sync(peers, r);
        if (isc && lane == __ffs(peers) - 1) atomicMin(v.cell_root + c, m);
    }
}

template <typename T, int DP>
__global__ void __launch_bounds__(256) k_cell_odd(HdView<T, DP> v) {
    pdl_enter();
    const int lane = lane_id();
    const uint32_t C = v.ctr->n_cells, NC = unless_failed(v.ctr, v.ctr->n_chunks), warps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < NC; t += warps) {
        const uint32_t A = chunk_cell(v.chunk_off, C, t);
        const uint32_t e = v.cell_start[A + 1], p = v.cell_start[A] + 32u * (t - v.chunk_off[A]) + lane;
        const unsigned m = __ballot_sync(0xffffffffu, p < e && v.core[p] && v.parent[p] != v.cell_root[A]);
        if (lane == 0) {
            v.odd_mask[t] = m;
            if (m) atomicAdd(v.odd_cnt + A, (uint32_t)__popc(m));
        }
    }
}

// A cell with more odd points than this has no tree of its own: its core points are all compared
// with those of every neighbour cell (the union kernels) instead of one odd point at a time.
constexpr uint32_t kOddMin = 8;
template <typename T, int DP>
__global__ void __launch_bounds__(256) k_cell_mixed(HdView<T, DP> v) {
    pdl_enter();
    const uint32_t C = unless_failed(v.ctr, v.ctr->n_cells);
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < C; c += gridDim.x * blockDim.x) {
        const uint32_t odd = v.odd_cnt[c];
        if (odd > kOddMin && odd > (v.cell_start[c + 1] - v.cell_start[c]) / 4u) v.cell_root[c] = kMixedRoot;
    }
}

// Has a pair of cells anything left for the union kernels?  Not when both have one tree and it is
// the same: then a pair of core points in different trees has an odd point, and those were
// compared with their whole neighbourhood.
__device__ __forceinline__ bool cells_to_join(uint32_t ra, uint32_t rb) {
    return rb != kNoRoot && (ra != rb || ra == kMixedRoot);
}

// Odd points against every core point of the 27 neighbour cells, joining the pairs within eps
// whose trees differ.  One warp per chunk with odd points; long streams in windows as in the
// counts (SPILL = true: the second launch).
template <typename T, int DP, bool SPILL, bool FILTER>
__global__ void __launch_bounds__(32 * kHdMaxWarps) k_odd_hd(HdView<T, DP> v) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typedef Candidate<T, DP, FILTER> Cand;
    typedef typename Cand::Row R;
    R *rows = reinterpret_cast<R *>(smem_raw) + (threadIdx.x >> 5) * 32 * DP;
    const int lane = lane_id();
    uint32_t chunks = 0;
    const uint32_t C = v.ctr->n_cells, N = unless_failed(v.ctr, SPILL ? min(v.ctr->hd_spill[2], v.sp_cap) : v.ctr->n_chunks);
    ItemQueue items(SPILL ? &v.ctr->hd_spill_next[2] : &v.ctr->hd_next[1], N);
    while (items.next()) {
        const uint32_t item = items.cur;
        const uint2 entry = SPILL ? v.sp_queue[item] : make_uint2(item, 0u);
        if (SPILL && entry.x == 0xffffffffu) continue;
        const uint32_t t = entry.x;
        const unsigned omask = v.odd_mask[t];
        if (!omask) continue;
        const uint32_t A = chunk_cell(v.chunk_off, C, t);
        if (v.cell_root[A] == kMixedRoot) continue;  // mixed: left to the union kernels
        const uint32_t e = v.cell_start[A + 1], base = v.cell_start[A] + 32u * (t - v.chunk_off[A]), p = base + lane;
        const GridParams &G = params_of(v, set_of_key(v, v.cell_key[A]));
        const uint2 rg = stream_span(v, A, lane);
        const uint32_t total = stream_length(v, rg);
        uint32_t p0 = 0, p1 = min(kSpillWin, total);
        if (SPILL) spill_window(entry.y, p1, total, p0, p1);
        stage_rows<R, DP>(rows, Cand::src(v), base, e);
        const bool mine = (omask >> lane) & 1u;
        uint32_t rp = mine ? uf_find(v.parent, p, v.ctr) : 0xffffffffu;
        auto scan = [&](uint32_t B, uint32_t q0, uint32_t q1) -> bool {
            // nothing to join with a cell without core points, nor for a row in the tree of the cell:
            // the cell's other core points are in that tree too, but for its odd ones, and those
            // come to the row's cell themselves (or, where the row's cell has another tree, the
            // two cells are left to the union kernels)
            uint32_t rb = v.cell_root[B];
            if (rb == kNoRoot) return true;
            if (rb != kMixedRoot) rb = uf_root_readonly(v.parent, rb, v.ctr);
            unsigned near = __ballot_sync(0xffffffffu, mine && rp != rb);
            if (!near) return true;
            near &= __ballot_sync(0xffffffffu, !cell_far<FILTER, DP>(v, rows + lane * DP, B, G));
            if (!near) return true;
            for (uint32_t qb = q0; qb < q1; qb += 32) {
                const uint32_t q = qb + lane;
                const bool qc = q < q1 && v.core[q];
                if (!__any_sync(0xffffffffu, qc)) continue;
                uint32_t rq = qc ? uf_find(v.parent, q, v.ctr) : 0xfffffffeu;
                Cand qv;
                qv.load(v, q, qc);
                ++chunks;
                unsigned rem = near;
                while (rem) {
                    const int jj = __ffs(rem) - 1;
                    rem &= rem - 1;
                    const uint32_t rj = __shfl_sync(0xffffffffu, rp, jj);
                    const bool hit = qc && rq != rj && qv.within(v, rows + jj * DP, base + jj, G);
                    if (hit) uf_union(v.parent, base + jj, q, v.ctr);
                    if (__any_sync(0xffffffffu, hit)) {
                        rq = qc ? uf_find(v.parent, q, v.ctr) : 0xfffffffeu;
                        if (mine) rp = uf_find(v.parent, p, v.ctr);
                    }
                }
            }
            return true;
        };
        for_stream_cells(v, rg, p0, p1, scan);
        if (!SPILL && p1 < total && !spill_push(v, 2, t, p1, total)) for_stream_cells(v, rg, p1, total, scan);
        __syncwarp();
    }
    add_counter(&v.ctr->work[1], lane == 0 ? chunks : 0u);
}

// Labels from complete lists (nl_k >= MINPTS - 1): a non-core point takes the smallest cluster id
// among its listed core points, a core point its cluster id.  One thread per point: at most nl_k scattered loads of a byte, a tree
// and an id instead of the comparison with the whole neighbourhood (9-D call of 200,003 points
// 3.50 -> 2.18 ms for the labels and unions from lists together).
template <typename T, int DP>
__global__ void __launch_bounds__(256) k_list_labels(HdView<T, DP> v) {
    pdl_enter();
    uint32_t noise = 0;
    const bool failed = look_failed(v.ctr);
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < v.g.n; j += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t p = (uint32_t)j;
        const bool isc = v.core[p];
        if (failed) continue;
        const uint32_t set = v.gtab ? set_of_key(v, v.cell_key[v.cell_of[p]]) : 0u;
        uint32_t best = kNoLabel;
        if (isc) {
            best = v.comp_min[v.parent[p]];
        } else {
            const uint32_t len = min(v.nl_cnt[p], v.nl_k);
            for (uint32_t i = 0; i < len; i += 4) {
                const uint4 e4 = list4(v, p, i);
                const uint32_t e[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t q = e[u] & ~kListNear;
                    if (i + u >= len || !v.core[q]) continue;
                    const uint32_t lq = v.comp_min[v.parent[q]];
                    if (lq >= best) continue;
                    if ((e[u] & kListNear) && !hd_exact<T, DP>(v.pts, p, q, params_of(v, set).eps2)) continue;
                    best = lq;
                }
            }
        }
        const uint32_t base_label = v.gtab ? (uint32_t)v.set_off[set] : 0u;
        const int32_t lab = best == kNoLabel ? -1 : (int32_t)(best - base_label);
        const uint32_t o = v.perm[p];
        v.labels[o] = lab;
        if (v.core_out) v.core_out[o] = isc ? 1 : 0;
        noise += lab < 0;
    }
    noise = __reduce_add_sync(0xffffffffu, noise);
    if (lane_id() == 0 && noise) atomicAdd(&v.ctr->n_noise, noise);
}

// Definitions 3-5, remaining edges: every pair of core points within eps of the upper half of
// the neighbourhood (the own pencil from this chunk on) whose trees differ is joined
// (lock-free union-find, root = smallest index).  A 32 x 32 tile whose core points all share
// one root is skipped without loading coordinates.
template <typename T, int DP, bool FILTER>
__global__ void __launch_bounds__(32 * kHdMaxWarps) k_merge_hd(HdView<T, DP> v) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typedef Candidate<T, DP, FILTER> Cand;
    typedef typename Cand::Row R;
    R *rows = reinterpret_cast<R *>(smem_raw) + (threadIdx.x >> 5) * 32 * DP;
    const int lane = lane_id();
    uint32_t chunks = 0, tests = 0, skipped = 0;
    HD_FOR_EACH_CHUNK(v, A, base, e, 2) {
        if (!v.cell_core[A]) continue;
        if (v.tc_min[1] && v.cx[e] - v.cx[v.cell_start[A]] >= v.tc_min[1]) continue;  // tensor-core cell
        const uint32_t p = base + lane;
        const bool pc = p < e && v.core[p];
        const unsigned amask = __ballot_sync(0xffffffffu, pc);
        if (!amask) continue;
        // the neighbour cells of the upper half that still have something to join
        const uint32_t ra = v.cell_root[A];
        const uint2 mine = lane < v.n_half ? v.ranges[(uint64_t)A * v.n_all + lane] : make_uint2(0u, 0u);
        bool any = false;
        for (uint32_t B = lane == 0 ? A : mine.x; B < mine.y; ++B) any |= cells_to_join(ra, v.cell_root[B]);
        if (!__any_sync(0xffffffffu, any)) continue;
        const GridParams &G = params_of(v, set_of_key(v, v.cell_key[A]));
        stage_rows<R, DP>(rows, Cand::src(v), base, e);
        uint32_t rp = pc ? uf_find(v.parent, p, v.ctr) : 0xffffffffu;
        for (int kk = 0; kk < v.n_half; ++kk) {
            const uint32_t lo = kk == 0 ? A : __shfl_sync(0xffffffffu, mine.x, kk);  // own pencil: this cell on
            const uint32_t hi = __shfl_sync(0xffffffffu, mine.y, kk);
            for (uint32_t B = lo; B < hi; ++B) {
                if (!cells_to_join(ra, v.cell_root[B])) continue;
                // own cell: start at this chunk (earlier points pair with it from their side)
                const uint32_t q0 = B == A ? base : v.cell_start[B];
                const uint32_t q1 = v.cell_start[B + 1];
                for (uint32_t qb = q0; qb < q1; qb += 32) {
                    const uint32_t q = qb + lane;
                    const bool qc = q < q1 && v.core[q];
                    if (!__any_sync(0xffffffffu, qc)) continue;
                    uint32_t rq = qc ? uf_find(v.parent, q, v.ctr) : 0xfffffffeu;
                    const uint32_t r0 = __shfl_sync(0xffffffffu, rp, __ffs(amask) - 1);
                    if (__all_sync(0xffffffffu, (!pc || rp == r0) && (!qc || rq == r0))) {
                        ++skipped;
                        continue;
                    }
                    Cand qv;
                    qv.load(v, q, qc);
                    ++chunks;
                    unsigned rem = amask;
                    while (rem) {
                        const int jj = __ffs(rem) - 1;
                        rem &= rem - 1;
                        const uint32_t pj = base + jj;
                        const uint32_t rj = __shfl_sync(0xffffffffu, rp, jj);
                        const bool need = qc && q > pj && rq != rj;
                        if (!__any_sync(0xffffffffu, need)) continue;
                        ++tests;
                        const bool hit = need && qv.within(v, rows + jj * DP, pj, G);
                        if (hit) uf_union(v.parent, pj, q, v.ctr);
                        if (__any_sync(0xffffffffu, hit)) {
                            // roots moved: refresh every lane so later pairs of the tile skip
                            rq = qc ? uf_find(v.parent, q, v.ctr) : 0xfffffffeu;
                            rp = pc ? uf_find(v.parent, p, v.ctr) : 0xffffffffu;
                        }
                    }
                }
            }
        }
        __syncwarp();
    }
    add_counter(&v.ctr->work[4], lane == 0 ? chunks : 0u);
    add_counter(&v.ctr->work[3], lane == 0 ? tests : 0u);
    add_counter(&v.ctr->work[2], lane == 0 ? skipped : 0u);
}

// Flatten the point union-find (read-only finds; the only writes are parent[j] = root), count the
// roots and the core points, canonical ids.
template <typename T, int DP>
__global__ void __launch_bounds__(256) k_comp_min_hd(HdView<T, DP> v) {
    pdl_enter();
    const int64_t n = v.g.n;
    const int lane = lane_id();
    uint32_t ncore = 0, roots = 0;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = base + lane;
        const bool valid = j < n && v.core[j];
        const uint32_t r = valid ? uf_root_readonly(v.parent, (uint32_t)j, v.ctr) : 0xffffffffu;
        if (valid) v.parent[j] = r;
        roots += (valid && r == (uint32_t)j) ? 1u : 0u;
        uint32_t val = valid ? v.perm[j] : kNoLabel;
        const unsigned vm = __ballot_sync(0xffffffffu, valid);
        if (!vm) continue;
        ncore += (lane == 0) ? __popc(vm) : 0u;
        const uint32_t r0 = __shfl_sync(0xffffffffu, r, __ffs(vm) - 1);
        if (__all_sync(0xffffffffu, !valid || r == r0)) {
            val = __reduce_min_sync(0xffffffffu, val);
            if (lane == 0) atomicMin(&v.comp_min[r0], val);
        } else if (valid) {
            atomicMin(&v.comp_min[r], val);
        }
    }
    if (lane == 0 && ncore) atomicAdd(&v.ctr->n_core, ncore);
    roots = __reduce_add_sync(0xffffffffu, roots);
    if (lane == 0 && roots) atomicAdd(&v.ctr->n_clusters, roots);
}

// Algorithm 4 / Definition 5 with the canonical rule, over points: core points take their
// cluster id, a non-core point the smallest id among its core neighbours, else -1.  For MINPTS
// beyond the lists.  Long streams are split into windows as in k_count_hd (SPILL = true: the
// second launch).
template <typename T, int DP, bool SPILL, bool FILTER>
__global__ void __launch_bounds__(32 * kHdMaxWarps) k_labels_hd(HdView<T, DP> v) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typedef Candidate<T, DP, FILTER> Cand;
    typedef typename Cand::Row R;
    R *rows = reinterpret_cast<R *>(smem_raw) + (threadIdx.x >> 5) * 32 * DP;
    const int lane = lane_id();
    uint32_t noise = 0, chunks = 0;
    const uint32_t C = v.ctr->n_cells, N = unless_failed(v.ctr, SPILL ? min(v.ctr->hd_spill[1], v.sp_cap) : v.ctr->n_chunks);
    ItemQueue items(SPILL ? &v.ctr->hd_spill_next[1] : &v.ctr->hd_next[3], N);
    while (items.next()) {
        const uint32_t item = items.cur;
        const uint2 entry = SPILL ? v.sp_queue[item] : make_uint2(item, 0u);
        if (SPILL && entry.x == 0xffffffffu) continue;
        const uint32_t t = entry.x, A = chunk_cell(v.chunk_off, C, t);
        const uint32_t s0 = v.cell_start[A], e = v.cell_start[A + 1], base = s0 + 32u * (t - v.chunk_off[A]);
        if (v.tc_min[2] && e - s0 - (v.cx[e] - v.cx[s0]) >= v.tc_min[2])
            continue;  // non-core rows of a tensor-core cell: labelled there
        const uint32_t aset = set_of_key(v, v.cell_key[A]);
        const GridParams &G = params_of(v, aset);
        const uint32_t base_label = v.gtab ? (uint32_t)v.set_off[aset] : 0u;
        const uint32_t p = base + lane;
        const bool have = p < e;
        const bool isc = have && v.core[p];
        uint32_t best = isc ? v.comp_min[v.parent[p]] : SPILL && have ? __ldcg(v.sp_val + p) : kNoLabel;
        const unsigned smask = __ballot_sync(0xffffffffu, have && !isc);
        bool decide = true;
        if (smask) {
            const uint2 rg = stream_span(v, A, lane);
            const uint32_t total = stream_length(v, rg);
            uint32_t p0 = 0, p1 = min(kSpillWin, total);
            if (SPILL) spill_window(entry.y, p1, total, p0, p1);
            stage_rows<R, DP>(rows, Cand::src(v), base, e);
            auto scan = [&](uint32_t B, uint32_t q0, uint32_t q1) -> bool {
                // a cell whose box is farther than eps from every row is passed over
                const unsigned near = smask & __ballot_sync(0xffffffffu,
                    !cell_far<FILTER, DP>(v, rows + lane * DP, B, G));
                if (!near) return true;
                for (uint32_t qb = q0; qb < q1; qb += 32) {
                    const uint32_t q = qb + lane;
                    const bool qc = q < q1 && v.core[q];
                    if (!__any_sync(0xffffffffu, qc)) continue;
                    const uint32_t lq = qc ? v.comp_min[v.parent[q]] : kNoLabel;
                    Cand qv;
                    qv.load(v, q, qc);
                    ++chunks;
                    unsigned rem = near;
                    while (rem) {
                        const int jj = __ffs(rem) - 1;
                        rem &= rem - 1;
                        const uint32_t bj = __shfl_sync(0xffffffffu, best, jj);
                        const bool need = qc && lq < bj;
                        if (!__any_sync(0xffffffffu, need)) continue;
                        uint32_t cand = (need && qv.within(v, rows + jj * DP, base + jj, G)) ? lq : kNoLabel;
                        cand = __reduce_min_sync(0xffffffffu, cand);
                        if (lane == jj && cand < best) best = cand;
                    }
                }
                return true;
            };
            for_stream_cells(v, rg, p0, p1, scan);
            if (SPILL) {
                // the last window of the chunk writes its labels from the smallest ids
                if (have && !isc) atomicMin(v.sp_val + p, best);
                __threadfence();
                __syncwarp();
                uint32_t left = 0;
                if (lane == 0) left = atomicSub(v.sp_pending + t, 1u);
                decide = __shfl_sync(0xffffffffu, left, 0) == 1u;
                __threadfence();
                if (decide && have && !isc) best = __ldcg(v.sp_val + p);
            } else if (p1 < total) {
                if (have) v.sp_val[p] = best;
                decide = !spill_push(v, 1, t, p1, total);
                if (decide) for_stream_cells(v, rg, p1, total, scan);
            }
            __syncwarp();
        }
        if (decide && have) {
            const int32_t lab = best == kNoLabel ? -1 : (int32_t)(best - base_label);
            const uint32_t o = v.perm[p];
            v.labels[o] = lab;
            if (v.core_out) v.core_out[o] = isc ? 1 : 0;
            noise += lab < 0;
        }
    }
    noise = __reduce_add_sync(0xffffffffu, noise);
    if (lane == 0 && noise) atomicAdd(&v.ctr->n_noise, noise);
    add_counter(&v.ctr->work[5], lane == 0 ? chunks : 0u);
}


// Batched calls: per-set min / max of every dimension (mm[set * 64 + i] complements of the min
// encodings, mm[(nsets + set) * 64 + i] max encodings), by seg_minmax.
template <typename T>
__global__ void __launch_bounds__(256) k_minmax_rt_seg(const T *__restrict__ in, int64_t n, int d,
                                                      const int64_t *set_off, int nsets,
                                                      unsigned long long *mm, DevCounters *ctr) {
    pdl_enter();
    seg_minmax<T>(in, n, d, set_off, nsets, mm, 64, ctr);
}

// Batched calls: coarse cell keys with the set id above them; each set projects on its own
// three dimensions (GridParams::sel).
template <typename T, typename K>
__global__ void __launch_bounds__(256) k_bin_proj_seg(const T *__restrict__ in, int64_t n, int d,
                                                     const int64_t *set_off, int nsets, const GridParams *gtab,
                                                     int key_bits, K *__restrict__ keys,
                                                     uint32_t *__restrict__ digit_counts, int total_bits, FillList fill) {
    pdl_enter();
    __shared__ uint32_t h[8][256];
    fill_regions(fill);
    count_digits_begin(h);
    const int passes = (total_bits + 7) / 8;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n;
         j += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t set = set_of_point(set_off, nsets, j);
        const GridParams &g = gtab[set];
        uint64_t key = (uint64_t)set << key_bits;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double t = __dmul_rn(__dsub_rn((double)ld_old(in + j * d + g.sel[i]), g.origin[i]), g.inv_side);
            uint32_t c = (uint32_t)floor(t);
            if (c > g.ncell[i] - 1) c = g.ncell[i] - 1;
            key |= (uint64_t)c << g.shift[i];
        }
        keys[j] = (K)key;
        count_digits(h, key, passes);
    }
    count_digits_end(h, passes, digit_counts);
}

}  // namespace hca
