// Internal declarations shared by the CUDA translation units of the HCA-DBSCAN library.
// Nothing here is part of the public ABI (include/hca_dbscan.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/hca_dbscan.h"

namespace hca {

constexpr int kMaxD = 4;            // dimensions handled by the hypercube-stencil path
constexpr int kMaxPencils = 512;    // neighbour pencil offsets per cell (d = 4 needs 179)
constexpr int kWarp = 32;
constexpr uint64_t kEmptyKey = ~0ull;
constexpr uint32_t kNoLabel = 0x7fffffffu;
constexpr uint32_t kLoopLimit = 1u << 22;  // cap of every loop that reads concurrently written data

// device-side status word bits (HCA_EDEVICE when non-zero)
constexpr uint32_t kErrHashFull = 1u;
constexpr uint32_t kErrLoop = 2u;
constexpr uint32_t kErrLook = 4u;  // a tile's wait for the earlier tiles ran out (sort, scans, cells)
constexpr uint32_t kErrBox = 8u;   // a point lies outside the extents a plan declared

// Base tuning (include/hca_dbscan.h): dimension-chosen neighbour search; tensor-core tiles
// from 8 rows (counts, unions) and 2 non-core rows (labels); hand-off at 32 open count rows;
// list edges joined in every cell.  The defaults per d (tune.cu) adjust the split from it.
constexpr hca_tuning kDefaultTuning = {0, 8, 8, 2, 32, 1, 4};

// Device counters and status, one struct per call in the workspace.
struct DevCounters {
    uint32_t n_cells;      // C: non-empty cells
    uint32_t n_pencils;    // P: non-empty pencils (cells sharing all but the last coordinate)
    uint32_t hash_mask;    // capacity - 1 of the pencil hash table
    uint32_t status;       // kErr* bits
    uint32_t n_dense;
    uint32_t n_core;
    uint32_t n_clusters;
    uint32_t n_noise;
    uint32_t n_core_cells;  // cells holding a core point (hypercube path)
    uint32_t n_list[3];     // hypercube path: cells to count, cells with core points, cells to label
    uint64_t minmax_enc[2 * kMaxD];  // order-preserving encodings per dim: complement of the min's (first
                                     // kMaxD; so that both halves start at 0 and grow) and the max's
    uint32_t nan_seen;
    uint32_t n_chunks;     // 32-point chunks of the coarse cells (high-dimensional path)
    uint32_t n_tc_chunks[4];  // work items of the tensor-core phases: counts, unions (the first window of
                              // every 128-row chunk), labels; [3]: the unions' other windows
    uint32_t tc_next[3];      // next unclaimed item of each tensor-core phase
    uint32_t n_tc_recount;    // chunks of the tensor-core recount of handed-over rows
    uint32_t tc_next_recount;
    uint32_t hd_next[4];      // next unclaimed 32-point chunk: counts, odd rows, unions, labels
    uint32_t hd_spill[3];     // windows queued by the CUDA-core chunks: counts, labels, odd rows
    uint32_t hd_spill_next[3];  // next unclaimed window of each queue
    uint32_t lowd_next;       // next unclaimed cell of k_labels
    // (lines of their own: beside the queue heads above, the work counters' atomics took k_labels of
    // 250,000 points in 2-D 27.6 -> 29.1 us; digit counts that straddle sectors took k_bin 14.6 -> 16.5)
    alignas(128) unsigned long long work[8];  // work counters (see hca_stats)
    unsigned long long tc_pairs;  // point pairs of the tensor-core tiles computed
    alignas(128) uint32_t digit_counts[8 * 256];  // radix digit counts per pass, filled while binning
};

// After kErrLook the tables that a sort or scan left are incomplete: permutations, offsets and counts
// of memory that nobody wrote.  The kernels that follow find nothing to do: every count that they take
// from such a table is read through unless_failed (one more word of the counters' first line, read
// along with the count), and sorts and scans return at their start.
__device__ __forceinline__ bool look_failed(const DevCounters *ctr) { return (ctr->status & kErrLook) != 0u; }
__device__ __forceinline__ uint32_t unless_failed(const DevCounters *ctr, uint32_t count) {
    const uint32_t status = ctr->status;
    return (status & kErrLook) ? 0u : count;
}

// Polls of one word after which a tile's wait for an earlier tile gives up.
#ifndef HCA_LOOK_SPINS
#define HCA_LOOK_SPINS (1u << 24)
#endif

// Grid of hypercubes (Algorithm 1) and everything a kernel needs to bin, pack and compare.
struct GridParams {
    int d;
    int64_t n;
    double origin[kMaxD];        // per-dimension minimum (origin shift, Sec. 2)
    float origin_f[kMaxD];
    double inv_side;             // 1 / cell side (cells per unit length)
    float inv_side_f;
    uint32_t ncell[kMaxD];       // cells per dimension
    uint32_t shift[kMaxD];       // bit offset of each coordinate in the packed key
    uint32_t bits[kMaxD];
    int key_bits;
    int prefix_shift;            // key >> prefix_shift = pencil key (all but the last coordinate)
    uint32_t min_pts;
    double eps2;                 // fl64(eps * eps): the exact predicate's threshold
    float lo32, hi32;            // FP32 filter: s < lo32 => within, s > hi32 => outside
    int bin_fp64;                // bin FP32 input in double precision
    int box_ok;                  // band coordinates exact enough in FP32 for cell-box tests
    float tau_box;               // widening of a cell box, band units
    float box_full, box_none;    // eps^2 in band units^2 times (1 -/+ 2^-12)
    int sel[3];                  // coarse-grid path: the three projected input dimensions
};

// Neighbour pencils: offsets of the first d-1 coordinates and the reach along the last one.
// Full list (every neighbour) and the upper half (pairs counted once) share the table:
// entries [0, n_half) are the offsets that are lexicographically >= 0.
struct Stencil {
    int n_all;
    int n_half;
    int8_t off[kMaxPencils][kMaxD - 1 > 0 ? kMaxD - 1 : 1];
    int8_t reach[kMaxPencils];   // max |delta_last| that can hold a point within eps
    uint16_t near[kMaxPencils];  // all pencils, nearest offsets first (counting order)
};

template <typename T, int D>
struct PadDim {
    static constexpr int value = (D == 3) ? 4 : D;
};

template <typename T, int D>
struct alignas(sizeof(T) * PadDim<T, D>::value) Pt {
    T x[PadDim<T, D>::value];
};

// Workspace carved out of one pool allocation per call.
struct Workspace {
    void *base;
    size_t bytes;
};

// A call's stream, and whether its kernels are put on the GPU early: while the one before in the
// stream still runs (programmatic stream serialisation; every kernel launched this way starts with
// pdl_enter, which waits until that one and its writes are complete).  Short kernels gain the
// launch: a call of 16 of them (2-D, 10,000 points) 197 -> 167 us, one of 34 (8-D, 3,001 points)
// 362 -> 298 us.  Long ones lose: a block that comes early finds its SM divided into shared memory
// and L1 as the kernel before needed it, the SM never drains in between, and the passes after
// the sort run on what L1 the sort left.  Never -> always early:
//   single 3-D sets of 100,000 points 336 -> 299 us, 500,000 402 -> 366, two million 634 -> 599, three
//   million 752 -> 736, four million 978 -> 1175, 16 million 3.38 -> 4.49 ms; 2-D, five million 1437 ->
//   1422 us; 4-D double, 500,000 942 -> 919: up to two million (the crossing lies between three and
//   four million in 3-D and above five in 2-D)
//   coarse grid: 9-D sets of 100,000 points 1061 -> 1004 us, 300,000 3.00 -> 3.01 ms, 600,000 6.41 -> 6.48,
//   a million 13.56 -> 13.80; 16-D, a million 2.64 -> 2.60: up to a million
//   64 sets in a call, 250,000 points in all: 2-D 368 -> 349 us, 3-D 603 -> 589, 8-D 791 -> 756; a million
//   527 -> 488, 1003 -> 992, 1942 -> 1933; one and a half million 635 -> 604, 1153 -> 1176, 2712 -> 2797:
//   up to a million
constexpr int64_t kEarlyMax = 1 << 21, kEarlyMaxBatched = 1 << 20;
struct Lane {
    cudaStream_t s;
    bool early;
    Lane(cudaStream_t stream = nullptr, bool e = false) : s(stream), early(e) {}
    operator cudaStream_t() const { return s; }
};

template <typename... P, typename... A>
inline void launch(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, Lane lane, A &&...args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = lane.s;
    cfg.attrs = &attr;
    cfg.numAttrs = lane.early ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// First statement of those kernels: wait for the kernel before, then let the next one be put in
// place behind this one (it waits in turn).
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Loads in these kernels.  A kernel put in place early is there while the one before it still writes, so
// what that one writes is not constant over its lifetime: the read-only path (__ldg, or a const pointer
// with __restrict__, which also lets the compiler move a load above the wait) is not for it, and ld is
// a plain load.  What was written two or more kernels before is constant: the kernel before lets
// this one in only after its own wait, when everything earlier is complete and visible.  The
// input and the tables copied from the host are older still (a memset comes before the first
// kernel of a call).  ld_old reads such data, and the input's pointer has its __restrict__; plain
// loads, which the compiler keeps behind earlier stores, took k_cells of 10,000 points 9.5 -> 11.4 us,
// the 7-D double call 623 -> 658.
template <typename T>
__device__ __forceinline__ T ld(const T *p) { return *p; }
template <typename T>
__device__ __forceinline__ T ld_old(const T *p) { return __ldg(p); }

// ---------------------------------------------------------------------------------------
// Primitives implemented in sort.cu / scan.cu
// ---------------------------------------------------------------------------------------

// Scratch words of cells_from_flags for m_max elements.
size_t scan_partials_size(int64_t m_max);

// Elements per tile of the scan (the tile sums in `partials` are per this many elements).
constexpr int kScanTileElems = 2048;

// Run-length cells from first-of-cell flags (1 on the first point of every cell, points in
// cell order).  The kernel that wrote the flags also wrote the sum of every kScanTileElems-flag
// tile into partials[tile] (tiles = ceil(n / kScanTileElems)).  Scans those sums (the total,
// the cell count, into *n_cells), then per point replaces the flag by the point's cell id and
// writes the first point and the key of every cell, and cell_start[n_cells] = n.
// partials: scan_partials_size(n) uint32.  Two launches.
template <typename K>
void cells_from_flags(const K *keys, uint32_t *flags_cell_of, int64_t n, uint32_t *partials, uint32_t *n_cells,
                      uint32_t *cell_start, uint64_t *cell_key, cudaStream_t s, int *launches);

// Geometry of the onesweep radix sort (sort.cu): keys per tile, digits per pass, and the
// most passes a call can make.  The scratch of a sort of n pairs is sort_hist_elems(n)
// uint32: two words per tile and digit for the look-back, the digit counts of every pass,
// one ticket per pass and a status word.
constexpr int kSortThreads = 1024;
constexpr int kSortRadix = 256;
constexpr int kSortMaxPasses = 8;
// Keys per thread of a tile: 13 for large sorts, and up to 1,228,800 keys the fewest of 2, 4 and 8
// that still leave 150 tiles or less (one per SM, with two SMs to spare), so that the passes of a
// small sort are spread over the chip and each tile ranks fewer keys in turn.
constexpr int sort_items_for(int64_t n) {
    return n <= 150 * kSortThreads * 2 ? 2 : n <= 150 * kSortThreads * 4 ? 4 : n <= 150 * kSortThreads * 8 ? 8 : 13;
}
// Threads of a tile: half as many, two tiles on an SM at a time, for more than four million keys.
constexpr int sort_threads_for(int64_t n) { return n > 4000000 ? kSortThreads / 2 : kSortThreads; }
constexpr int64_t sort_tiles_for(int64_t n) {
    const int64_t tile = (int64_t)sort_items_for(n) * sort_threads_for(n);
    return n <= tile ? 1 : (n + tile - 1) / tile;
}
constexpr size_t sort_hist_elems(int64_t n) {
    // (where the tiles grow their number drops; the scratch keeps growing with n)
    int64_t tiles = sort_tiles_for(n);
    if (n > 150 * kSortThreads * 2 && tiles < 150) tiles = 150;
    return (size_t)(2 * tiles * kSortRadix + kSortMaxPasses * kSortRadix + kSortMaxPasses + 2);
}

// LSD radix sort of (key, value) pairs by bits [begin_bit, end_bit), 8 bits per pass.
// Ping-pongs between (keys, vals) and (keys_alt, vals_alt); returns true when the sorted
// result ends up in the alternate buffers.  hist: sort_hist_size(n) uint32 of scratch
// (8-byte aligned; cleared by the sort itself).  A bounded look-back wait that ran out sets
// kErrLook in *err_out (device word; NULL: the status word inside hist, sort_status_word); the
// passes after it return at once.
inline size_t sort_hist_size(int64_t n) { return sort_hist_elems(n); }
uint32_t *sort_status_word(uint32_t *hist, int64_t n);
// digit_counts (optional, device): counts of every 8-bit digit of every pass, [pass][256],
// already computed by the caller.  hist_cleared: the caller has cleared hist.  identity: the values
// are 0 .. n - 1 and vals need not hold them.
template <typename K>
bool radix_sort_pairs(K *keys, uint32_t *vals, K *keys_alt, uint32_t *vals_alt, int64_t n,
                      int begin_bit, int end_bit, uint32_t *hist, Lane s, int *launches,
                      uint32_t *err_out = nullptr, const uint32_t *digit_counts = nullptr,
                      bool hist_cleared = false, bool identity = false);

// Pool allocation (stream ordered) used by api.cu and the pipelines.
cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t s);
cudaError_t pool_free(void *p, cudaStream_t s);

int device_sm_count();

// Host orchestration of one clustering call, instantiated per (T, D) in lowd_*.cu.
struct RunArgs {
    const void *d_points = nullptr;
    int64_t n = 0;
    int d = 0;
    double eps = 0.0;
    int min_pts = 0;
    int32_t *d_labels = nullptr;
    uint8_t *d_core = nullptr;
    cudaStream_t stream = nullptr;
    hca_stats *stats = nullptr;
    int flags = 0;
    // batched calls (n_sets > 0): sets of consecutive points, each with its own eps and MINPTS
    int nsets = 0;
    const int64_t *h_off = nullptr;      // host, nsets + 1 point offsets
    const double *h_eps = nullptr;       // host, nsets
    const int32_t *h_minpts = nullptr;   // host, nsets
    hca_tuning tune = kDefaultTuning;    // neighbour search and tensor-core split of this call
    // Plans (d <= 4): declared extents box_mn / box_mx (host, D values per set, set-major) size
    // the grids instead of the measured ones, so nothing in the call waits for the host; a
    // device kernel flags a point outside its box (status kErrBox).
    const double *box_mn = nullptr, *box_mx = nullptr;
    size_t *ws_query = nullptr;          // set: store the workspace bytes needed, launch nothing
    void *ws_ext = nullptr;              // caller-owned workspace (nullptr: the call allocates)
    size_t ws_ext_bytes = 0;
    DevCounters *h_ext = nullptr;        // pinned host copy of the counters (nullptr: the thread's)
    void *h_stage = nullptr;             // pinned staging of the batched tables (deferred calls)
    bool deferred = false;               // no host synchronisation: the caller checks the status
    bool short_lists = false;            // coarse grid: neighbour lists no longer than the table space holds
    // optional outputs: the measured extents of a single-set call without declared extents
    // (host, 2 d values: d minima then d maxima), and the launch count and key bits of the call
    double *ext_out = nullptr;
    int *launches_out = nullptr;
    int *key_bits_out = nullptr;
};

// The tuning in effect for dimension d (tune.cu).
hca_tuning tuning_for(int d);

// The unique id of the calling thread's current CUDA context, 0 when there is none or the
// driver cannot say (sort_static.cu).
unsigned long long current_context_id();

// A plan of one set with the given flags (plan.cu; hca_plan_create is this with flags 0).  Without
// memory for whole neighbour lists it takes short ones, or with whole_lists fails.
int plan_create_single(hca_plan **out, const void *d_points, int32_t dtype, int64_t n, int32_t d, double eps,
                       int32_t min_pts, const double *box_min, const double *box_max, int32_t *d_labels,
                       uint8_t *d_core, int32_t flags, bool whole_lists = false);

// The workspace bound of hca_workspace_bytes for calls of at most min_pts; with short_lists, what a
// call takes without memory for its whole neighbour lists (api.cu).
int workspace_bound(int64_t n, int32_t d, int32_t dtype, int32_t flags, int32_t min_pts, bool short_lists,
                    int64_t *bytes);

// api.cu: argument checks, dispatch to the pipelines, and the clustering calls with an
// explicit tuning.
int dispatch(const RunArgs &a, int32_t dtype);
int check_common(const void *pts, int32_t dtype, int64_t n, int32_t d, double eps, int32_t min_pts,
                 const void *labels);
int device_ex_tuned(const void *d_points, int32_t dtype, int64_t n, int32_t d, double eps, int32_t min_pts,
                    int32_t *d_labels, uint8_t *d_core, void *stream, hca_stats *stats, int32_t flags,
                    const hca_tuning &tune, double *ext_out = nullptr);
int batched_tuned(const void *d_points, int32_t dtype, int32_t n_sets, const int64_t *offsets, int32_t d,
                  const double *eps, const int32_t *min_pts, int32_t *d_labels, uint8_t *d_core, void *stream,
                  hca_stats *stats, int32_t flags, const hca_tuning &tune, bool short_lists = false);
// multi.cu: batched calls with one d per set.  The sets are grouped by d (increasing d); a
// group whose sets are consecutive in the caller's buffers runs in place, any other group is
// gathered into a compact copy (points, labels, core flags, segment table) and scattered back.
struct SetGroup {
    int d = 0;
    std::vector<int32_t> sets;            // the call's set indices, increasing
    std::vector<int64_t> off;             // group-local point offsets (sets + 1)
    std::vector<double> eps;
    std::vector<int32_t> min_pts;
    std::vector<double> box_mn, box_mx;   // declared boxes of the sets, d values each (plans)
    std::vector<int64_t> far_pts;         // element offset of each set in the caller's points
    std::vector<int64_t> far_lab;         // point offset of each set in the caller's labels
    int64_t n = 0;                        // points of the group
    bool gather = false;                  // sets not consecutive: run on a compact copy
    int64_t first_point = 0;              // in place: first set's point offset
    size_t first_elem = 0;                // in place: first set's element offset
};
struct GroupBuffers {
    void *points;
    int32_t *labels;
    uint8_t *core;
    int64_t *table;
};
int group_sets(int32_t n_sets, const int64_t *offsets, const int32_t *d_per_set, const double *eps,
               const int32_t *min_pts, const double *box_mn, const double *box_mx, std::vector<SetGroup> &out);
size_t group_gather_bytes(const SetGroup &g, int32_t dtype, bool with_core);
void group_gather_layout(const SetGroup &g, int32_t dtype, bool with_core, void *buf, GroupBuffers &gb);
void group_table(const SetGroup &g, std::vector<int64_t> &t);
void group_gather(const SetGroup &g, int32_t dtype, const void *d_points, const GroupBuffers &gb, cudaStream_t s);
void group_scatter(const SetGroup &g, const GroupBuffers &gb, int32_t *d_labels, uint8_t *d_core, cudaStream_t s);
void add_stats(hca_stats &acc, const hca_stats &x);
int run_group(const SetGroup &g, const void *d_points, int32_t dtype, int32_t *d_labels, uint8_t *d_core,
              cudaStream_t s, hca_stats *stats, int32_t flags, const hca_tuning &tune, bool short_lists = false);
// tune_by_d: nullable, 64 tunings indexed by d - 1 (NULL: the table of tune.cu)
int batched_mixed(const void *d_points, int32_t dtype, int32_t n_sets, const int64_t *offsets,
                  const int32_t *d_per_set, const double *eps, const int32_t *min_pts, int32_t *d_labels,
                  uint8_t *d_core, void *stream, hca_stats *stats, int32_t flags, const hca_tuning *tune_by_d,
                  bool short_lists = false);

template <typename T, int D>
int run_lowd(const RunArgs &a);
template <typename T, int DP>
int run_hd(const RunArgs &a);

}  // namespace hca

#define HCA_CUDA_TRY(expr)                                    \
    do {                                                      \
        cudaError_t _e = (expr);                              \
        if (_e != cudaSuccess) return HCA_ECUDA;              \
    } while (0)
