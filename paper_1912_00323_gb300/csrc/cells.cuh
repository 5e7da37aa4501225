// One-pass prefix sums over tiles (decoupled look-back) and what is built on them: the scan of a
// function's values with a callback per element, and the cells and pencils of sorted keys.
//
// At every size the steps between the sort and the neighbour ranges are launches of a few
// microseconds on data that the previous launch just wrote: flags, tile sums, the scan of the
// sums, the applied scan.  Here a tile computes its values, publishes their sum, adds up the
// earlier tiles' and writes its results, so a scan is one launch instead of four, and cells and
// pencils together one instead of seven.
//
// Look-back: a tile's word holds a state and a value, its own sum (AGG) and then the sum of all
// tiles up to it (PREFIX), written and read as one 64-bit word.  Tiles are numbered by a ticket
// in the order they start, so a tile only waits for running ones; the wait is bounded.  The scans
// of a call share one array of words, told apart by an epoch; the cells and pencils have
// another, whose words hold two counts of 31 bits.
#pragma once

#include "block_scan.cuh"
#include "hca_internal.cuh"

namespace hca {

constexpr uint32_t kLookSpins = HCA_LOOK_SPINS;
constexpr int kTileThreads = 256;
constexpr int kTileItems = kScanTileElems / kTileThreads;
constexpr int kMaxScans = 16;  // scans (epochs 1 .. kMaxScans - 1) of one call; epoch 0: cleared words, the cells

// Scratch of the scans of one call over at most n elements (or of its cells): a ticket per epoch,
// then the words.  Cleared once per call (fill_regions).
inline size_t look_bytes(int64_t n) {
    return sizeof(uint32_t) * kMaxScans + sizeof(uint64_t) * ((size_t)(n + kScanTileElems - 1) / kScanTileElems + 1);
}
struct LookBack {
    uint32_t *tickets;
    unsigned long long *words;
    static LookBack at(void *p) {
        LookBack l;
        l.tickets = (uint32_t *)p;
        l.words = (unsigned long long *)((char *)p + sizeof(uint32_t) * kMaxScans);
        return l;
    }
};

// Up to four regions of words that a kernel sets to a value (instead of a memset launch each).
struct FillList {
    uint32_t *p[4];
    uint64_t words[4];
    uint32_t value[4];
    int n;
    // bytes set to 1 (any alignment): the core flags.  Most points are core, and their flags in the
    // input's order are one scattered byte each; written in a stream here, only the other points'
    // zeros are scattered later (labels stage of two million points in 3-D 50 -> 38 us, of 16 million
    // 329 -> 248)
    uint8_t *ones;
    uint64_t n_ones;
    void add(void *ptr, size_t bytes, uint32_t v) {
        p[n] = (uint32_t *)ptr;
        words[n] = bytes / 4;
        value[n] = v;
        ++n;
    }
};
__device__ __forceinline__ void fill_regions(const FillList &f) {
    const uint64_t t0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, step = (uint64_t)gridDim.x * blockDim.x;
    for (int r = 0; r < f.n; ++r) {
        const uint64_t quads = f.words[r] / 4;  // (regions start on 256-byte boundaries)
        const uint32_t x = f.value[r];
        for (uint64_t i = t0; i < quads; i += step) reinterpret_cast<uint4 *>(f.p[r])[i] = make_uint4(x, x, x, x);
        for (uint64_t i = 4 * quads + t0; i < f.words[r]; i += step) f.p[r][i] = x;
    }
    if (f.ones) {
        const uint64_t to_quad = (16u - ((uintptr_t)f.ones & 15u)) & 15u;
        const uint64_t head = to_quad < f.n_ones ? to_quad : f.n_ones, quads = (f.n_ones - head) / 16;
        const uint32_t x = 0x01010101u;
        for (uint64_t i = t0; i < quads; i += step) reinterpret_cast<uint4 *>(f.ones + head)[i] = make_uint4(x, x, x, x);
        if (t0 < head) f.ones[t0] = 1;
        const uint64_t tail = head + 16 * quads + t0;
        if (tail < f.n_ones) f.ones[tail] = 1;
    }
}

// A tile's own value (PAIR: the cells' words, two counts of 31 bits; else 32 bits and the epoch).
template <bool PAIR>
__device__ __forceinline__ void look_publish(const LookBack &l, uint32_t epoch, uint32_t tile, unsigned long long own) {
    constexpr int kShift = PAIR ? 62 : 56;
    const unsigned long long tag = PAIR ? 0ull : (unsigned long long)epoch << 58;
    ((volatile unsigned long long *)l.words)[tile] = tag | (tile == 0 ? 2ull : 1ull) << kShift | own;
}

// Sum of the earlier tiles' values, and the sum with this tile's published.  One full warp calls it
// after look_publish; every lane returns the result.  When the wait runs out kErrLook is set, ok is
// false, nothing is published, and the tile writes nothing; so the later ones, which wait for it.
template <bool PAIR>
__device__ __forceinline__ unsigned long long look_back(const LookBack &l, uint32_t epoch, uint32_t tile,
                                                        unsigned long long own, uint32_t *err, bool &ok_all) {
    const int lane = threadIdx.x & 31;
    volatile unsigned long long *st = l.words;
    constexpr int kShift = PAIR ? 62 : 56;
    constexpr unsigned long long kAgg = 1ull << kShift, kPrefix = 2ull << kShift;
    constexpr unsigned long long kValue = PAIR ? kAgg - 1ull : 0xffffffffull;
    const unsigned long long tag = PAIR ? 0ull : (unsigned long long)epoch << 58;
    unsigned long long sum = 0;
    int64_t base = (int64_t)tile - 1;
    uint32_t spins = 0;
    ok_all = true;
    while (base >= 0) {
        const int64_t i = base - lane;
        const unsigned long long w = i >= 0 ? st[i] : (tag | kPrefix);
        const bool ok = (PAIR || (w >> 58) == epoch) && (w & (kAgg | kPrefix)) != 0ull;
        const unsigned okm = __ballot_sync(0xffffffffu, ok), pm = __ballot_sync(0xffffffffu, ok && (w & kPrefix));
        const int first = pm ? __ffs(pm) - 1 : 31;
        const unsigned take = first == 31 ? 0xffffffffu : (2u << first) - 1u;
        if ((okm & take) != take) {  // wait for the nearest ones
            if (++spins > kLookSpins) {
                if (lane == 0) atomicOr(err, kErrLook);
                ok_all = false;
                break;
            }
            continue;
        }
        unsigned long long x = (take >> lane) & 1u ? (w & kValue) : 0ull;
#pragma unroll
        for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        sum += x;
        if (pm) break;
        base -= 32;
    }
    if (lane == 0 && tile > 0 && ok_all) st[tile] = tag | kPrefix | ((sum + own) & kValue);
    return sum;
}

// The next tile, for the whole block; ok is false once a wait has run out (here or before).
__device__ __forceinline__ uint32_t take_tile(const LookBack &l, uint32_t epoch, const uint32_t *err, bool &ok) {
    __shared__ uint32_t s_tile, s_failed;
    if (threadIdx.x == 0) s_tile = atomicAdd(l.tickets + epoch, 1u);
    if (threadIdx.x == 32) s_failed = *(const volatile uint32_t *)err & kErrLook;  // (beside the ticket)
    __syncthreads();
    ok = s_failed == 0u;
    return s_tile;
}

// out[i] = sum of f(0 .. i - 1) for i < m = min(*m_dev, m_max) (m_max without m_dev), emit(i, f(i),
// out[i]) for each, and the sum of all into *total (nullable).  out nullable.  The grid has one
// block per tile of m_max; tiles past m only keep the total right when m is 0.
template <typename F, typename E>
__global__ void __launch_bounds__(kTileThreads) k_scan_fn(F f, E emit, uint32_t *out, int64_t m_max,
                                                         const uint32_t *m_dev, uint32_t *total, LookBack l,
                                                         uint32_t epoch, uint32_t *err) {
    pdl_enter();
    __shared__ uint32_t s_val[kScanTileElems];
    __shared__ uint32_t s_base, s_ok;
    const int64_t m = m_dev ? min((int64_t)*m_dev, m_max) : m_max;
    bool ok;
    const uint32_t tile = take_tile(l, epoch, err, ok);
    if (!ok) return;
    const int64_t base = (int64_t)tile * kScanTileElems;
    if (base >= m) {
        if (m == 0 && tile == 0 && threadIdx.x == 0 && total) *total = 0u;
        return;
    }
    uint32_t mine[kTileItems];
#pragma unroll
    for (int k = 0; k < kTileItems; ++k) {
        const int64_t i = base + k * kTileThreads + threadIdx.x;
        mine[k] = i < m ? f(i) : 0u;
        s_val[k * kTileThreads + threadIdx.x] = mine[k];
    }
    __syncthreads();
    uint32_t v[kTileItems], sum = 0;
#pragma unroll
    for (int k = 0; k < kTileItems; ++k) {
        v[k] = s_val[threadIdx.x * kTileItems + k];
        sum += v[k];
    }
    uint32_t all;
    uint32_t run = block_exclusive_scan<kTileThreads>(sum, &all);
    if (threadIdx.x < 32) {
        if (threadIdx.x == 0) look_publish<false>(l, epoch, tile, all);
        bool found;
        const uint32_t b = (uint32_t)look_back<false>(l, epoch, tile, all, err, found);
        if (threadIdx.x == 0) {
            s_base = b;
            s_ok = found;
            if (found && total && base + kScanTileElems >= m) *total = b + all;
        }
    }
    __syncthreads();
    if (!s_ok) return;
    run += s_base;
#pragma unroll
    for (int k = 0; k < kTileItems; ++k) {
        s_val[threadIdx.x * kTileItems + k] = run;
        run += v[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kTileItems; ++k) {
        const int64_t i = base + k * kTileThreads + threadIdx.x;
        if (i >= m) continue;
        const uint32_t x = s_val[k * kTileThreads + threadIdx.x];
        if (out) out[i] = x;
        emit(i, mine[k], x);
    }
}

// The scans of one call, numbered.
struct Scans {
    LookBack l;
    uint32_t *err;
    uint32_t epoch;
    Lane s;
    int *launches;
    template <typename F, typename E>
    void run(F f, E emit, uint32_t *out, int64_t m_max, const uint32_t *m_dev, uint32_t *total) {
        const unsigned tiles = (unsigned)((m_max + kScanTileElems - 1) / kScanTileElems);
        launch(k_scan_fn<F, E>, tiles ? tiles : 1u, kTileThreads, 0, s, f, emit, out, m_max, m_dev, total, l, epoch++, err);
        *launches += 1;
    }
};

// Cells (runs of equal keys) and pencils (runs of cells that share key >> prefix_shift) of n
// sorted keys: the cell of every point, first point and key of every cell, first cell of every
// pencil, the ends, the two counts.  With ptab the pencils also go into a direct table indexed by
// their key (cleared to ~0 beforehand).
template <typename K>
struct CellsArgs {
    const K *keys;
    const uint32_t *idx;
    int64_t n;
    int prefix_shift;
    uint32_t *cell_of, *cell_start;
    uint64_t *cell_key;
    uint32_t *pencil_start, *ptab;
    LookBack l;
    DevCounters *ctr;
};

// One tile (all 256 threads of the block): `between` runs after the tile's counts are published and
// before the earlier tiles' are read, so that its loads cover the wait; on_cell(c) for every
// first point of a cell.
template <typename K, typename B, typename F>
__device__ __forceinline__ void cells_tile(const CellsArgs<K> &a, uint32_t tile, B between, F on_cell) {
    constexpr int kWarps = kTileThreads / 32, kGroups = kTileItems * kWarps;  // 32-point groups
    static_assert(kGroups == 64, "two groups per lane of the scanning warp");
    __shared__ uint32_t s_cnt[kGroups];  // pencils << 16 | cells, then their exclusive sums
    __shared__ uint32_t s_cells, s_pencils;  // (s_cells ~0: the look-back failed)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)tile * kScanTileElems;
    unsigned cb[kTileItems], pb[kTileItems];
    {
        K key[kTileItems];
#pragma unroll
        for (int k = 0; k < kTileItems; ++k) {
            const int64_t j = base + k * kTileThreads + threadIdx.x;
            key[k] = j < a.n ? a.keys[j] : K(0);
        }
#pragma unroll
        for (int k = 0; k < kTileItems; ++k) {
            const int64_t j = base + k * kTileThreads + threadIdx.x;
            K prev = __shfl_up_sync(0xffffffffu, key[k], 1);
            if (lane == 0 && j > 0 && j < a.n) prev = a.keys[j - 1];
            const bool c = j < a.n && (j == 0 || key[k] != prev);
            const bool p = c && (j == 0 || ((uint64_t)key[k] >> a.prefix_shift) != ((uint64_t)prev >> a.prefix_shift));
            cb[k] = __ballot_sync(0xffffffffu, c);
            pb[k] = __ballot_sync(0xffffffffu, p);
            if (lane == 0) s_cnt[k * kWarps + warp] = (uint32_t)__popc(pb[k]) << 16 | (uint32_t)__popc(cb[k]);
        }
    }
    __syncthreads();
    unsigned long long own = 0;
    if (warp == 0) {
        const uint32_t x0 = s_cnt[2 * lane], x1 = s_cnt[2 * lane + 1];  // (a tile has at most 2048 of each)
        const uint32_t incl = warp_inclusive_scan(x0 + x1);
        const uint32_t all = __shfl_sync(0xffffffffu, incl, 31);
        s_cnt[2 * lane] = incl - x0 - x1;
        s_cnt[2 * lane + 1] = incl - x1;
        // (fewer than 2^31 points: either count fits its 31 bits)
        own = (unsigned long long)(all >> 16) << 31 | (all & 0xffffu);
        if (lane == 0) look_publish<true>(a.l, 0u, tile, own);
    }
    between();
    if (warp == 0) {
        bool found;
        const unsigned long long b = look_back<true>(a.l, 0u, tile, own, &a.ctr->status, found);
        if (lane == 0) {
            s_cells = found ? (uint32_t)(b & 0x7fffffffull) : 0xffffffffu;
            s_pencils = (uint32_t)(b >> 31);
        }
    }
    __syncthreads();
    const uint32_t c0 = s_cells, p0 = s_pencils;
    if (c0 == 0xffffffffu) return;
#pragma unroll
    for (int k = 0; k < kTileItems; ++k) {
        const int64_t j = base + k * kTileThreads + threadIdx.x;
        if (j >= a.n) continue;
        const uint32_t off = s_cnt[k * kWarps + warp];
        const unsigned upto = lane == 31 ? 0xffffffffu : (2u << lane) - 1u;
        const uint32_t c = c0 + (off & 0xffffu) + (uint32_t)__popc(cb[k] & upto) - 1u;
        a.cell_of[j] = c;
        const uint32_t p = p0 + (off >> 16) + (uint32_t)__popc(pb[k] & upto) - 1u;
        if ((cb[k] >> lane) & 1u) {
            const uint64_t key = (uint64_t)a.keys[j];
            a.cell_start[c] = (uint32_t)j;
            a.cell_key[c] = key;
            on_cell(c);
            if ((pb[k] >> lane) & 1u) {
                a.pencil_start[p] = c;
                if (a.ptab) a.ptab[key >> a.prefix_shift] = p;
            }
        }
        if (j == a.n - 1) {
            a.cell_start[c + 1] = (uint32_t)a.n;
            a.pencil_start[p + 1] = c + 1;
            a.ctr->n_cells = c + 1;
            a.ctr->n_pencils = p + 1;
        }
    }
}

}  // namespace hca
