// LSD radix sort of (key, uint32 value) pairs, 8 bits per pass, one kernel per pass.
//
// A first kernel counts the digits of every pass over all keys (the counts do not depend on
// the order, so one read of the keys serves all passes); a caller that produced the keys may
// pass these counts in instead.  Each pass kernel then takes a tile of 1024 threads x 2, 4, 8
// or 13 keys or 512 threads x 13 keys (sort_items_for, sort_threads_for), ranks every key stably
// among the keys of its tile with the same digit (the lanes of a warp with one digit found by a
// match instruction or by shared-memory OR masks, per-warp digit counters, an exclusive scan across warps), publishes the tile's digit
// counts, scatters the tile through shared memory in digit order, learns how many keys of each
// digit the earlier tiles hold by decoupled look-back, and writes the digit runs out with
// coalesced stores.
//
// Tile size.  A tile is one CTA per SM (its shared memory holds the whole tile), so at two
// million keys the ~150 tiles of 13,312 all run at once.  A smaller sort takes smaller tiles, so
// that it spreads over as many SMs and each ranks fewer keys in turn: four passes over 300,001
// keys 70 -> 46 us, two over 10,000 28 -> 19 us (one tile of 13,312 before).  Two CTAs of 512
// threads per SM instead were slower (two million keys 76 -> 109 us); above four million keys, with
// many tiles per SM, one of the two loads or stores while the other ranks (five passes over 64-bit
// keys: 3.4 million 186 -> 191 us, five million 273 -> 261, 16 million 759 -> 734).  With every tile running together a published
// prefix reaches the later tiles only through their own reads, so the look-back reads 64
// predecessors per round trip (four thread quarters of 16 words per digit): the last tile of
// two million keys needs three round trips instead of the dozens that a 4096-key tile with a
// few words per trip needed.
//
// A pass is bound by the wavefronts of shared memory: 13,312 keys take an SM some 37,000 cycles, 7,000
// to rank, 5,500 to scatter, 7,000 to write out, 3,000 for the digit starts, the rest for the
// loads and the look-back.  So whole tiles (all but the last) test no bounds, the digit's place in
// the tile is folded into the per-warp offsets and into the global offset, and both digit scans
// are one (16 million keys as above 786 -> 759 us; four passes over 32-bit keys, two million 70 -> 66 us,
// 600,000 45 -> 41, 50,000 28 -> 25).  One vote per digit bit instead of the shared
// OR was slower (759 -> 857 us).
//
// Up to kFullSumTiles tiles (about 3.4 million keys) a tile instead sums the published counts
// of all earlier tiles (eight loads in flight per thread, no prefix published): with every
// tile running at once no prefix would be there to shorten the look-back anyway.
//
// Look-back: a tile publishes, per digit, first its own count (state AGG) and then the count of
// all tiles up to and including itself (state PREFIX).  A tile reads its predecessors'
// words from the nearest one backwards, adding AGG values until it meets a PREFIX.  Tiles take
// their index from an atomic ticket in the order they start, so a tile only ever waits on
// tiles that are already running; every wait is bounded (kSpinLimit), and a wait that runs
// out sets the caller's status word instead of hanging.  Each status word packs
// (epoch, state, count) into 64 bits so flag and value are read and written together; the
// epoch (pass number + 1) makes words left by an earlier pass invisible.  Words are tile-major
// (the 256 digits of one tile are consecutive), so a warp reads 32 digits of a tile in one
// coalesced 256-byte access.
#include <type_traits>

#include "block_scan.cuh"
#include "hca_internal.cuh"

namespace hca {

namespace {

constexpr int kRadix = kSortRadix;
constexpr int kMaxPasses = kSortMaxPasses;
constexpr int kLbWords = 16;                      // predecessors per thread per round trip
constexpr int kHistThreads = 256;
constexpr uint32_t kSpinLimit = HCA_LOOK_SPINS;
// Up to this many tiles a tile sums the counts of all earlier tiles instead of the decoupled
// look-back (at two million keys all ~150 tiles run at once, so the look-back finds no
// published prefix and reads the same words over three round trips)
constexpr int kFullSumTiles = 256;
constexpr uint64_t kStateAgg = 1, kStatePrefix = 2;

__device__ __forceinline__ uint64_t os_pack(uint32_t epoch, uint64_t state, uint32_t value) {
    return ((uint64_t)(epoch * 4u + (uint32_t)state) << 32) | value;
}

// Digit counts of every pass: ghist[p * 256 + digit].
template <typename K>
__global__ void __launch_bounds__(kHistThreads) k_os_hist(const K *keys, int64_t n, int begin_bit,
                                                         int end_bit, uint32_t *__restrict__ ghist) {
    pdl_enter();
    __shared__ uint32_t h[kMaxPasses][kRadix];
    for (int i = threadIdx.x; i < kMaxPasses * kRadix; i += kHistThreads) (&h[0][0])[i] = 0;
    __syncthreads();
    const int passes = (end_bit - begin_bit + 7) / 8;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = base + threadIdx.x;
        const bool valid = i < n;
        const K key = valid ? keys[i] : K(0);
        if (valid) {
            for (int p = 0; p < passes; ++p) {
                const int shift = begin_bit + 8 * p;
                const int bits = min(8, end_bit - shift);
                atomicAdd(&h[p][(uint32_t)(key >> shift) & ((1u << bits) - 1u)], 1u);
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * kRadix; i += kHistThreads) {
        const uint32_t c = (&h[0][0])[i];
        if (c) atomicAdd(&ghist[i], c);
    }
}

// Shared memory of a pass (dynamic, 16-byte aligned).
template <typename K, int ITEMS, int NT>
struct PassSmem {
    // (quarters: the groups of one thread per digit, four of 1024 threads, two of 512)
    static constexpr int tile = ITEMS * NT, kSortWarps = NT / 32, kQuarters = NT / kRadix;
    static_assert(kQuarters * kRadix == NT, "whole groups of digits");
    uint32_t whist[kSortWarps][kRadix];       // per-warp digit counts, then per-warp digit offsets
    uint32_t part[kQuarters][kRadix];     // counts of a quarter's warps, per digit
    uint32_t lstart[kRadix];                // first position of each digit in the tile
    uint32_t goff[kRadix];                  // global position of the tile's first key of each digit
    uint32_t lb_sum[kQuarters][kRadix];   // look-back: AGG sum of a quarter's window
    uint32_t lb_used[kQuarters][kRadix];  // predecessors the quarter consumed
    uint32_t lb_kind[kQuarters][kRadix];  // 0 window read through, 1 met a PREFIX, 2 met an unpublished word
    int32_t lb_next[kRadix];                // nearest predecessor not yet added, per digit (-1: done)
    uint2 wsum[kRadix / 32];                // digit starts: the warps' sums of the tile's and all counts
    uint32_t tile_id, failed, pad[2];
    union {
        uint32_t wmask[kSortWarps][kRadix];   // ranking: per-warp lane masks of each digit
        K keys[tile];                       // then: the tile in digit order
    };
    uint32_t vals[tile];
};

// A pass in which a wait ran out leaves places of its output unwritten, with digits that were never
// counted, so the passes after it are closed: their tickets start at kClosed, and every tile that takes
// one returns.
constexpr uint32_t kClosed = 0x80000000u;
__device__ __forceinline__ void pass_failed(uint32_t *err, uint32_t *ticket, uint32_t epoch) {
    atomicOr(err, kErrLook);
    for (uint32_t q = epoch; q < (uint32_t)kMaxPasses; ++q) atomicOr(ticket + (q - epoch + 1u), kClosed);
}

// One pass: rank within the tile, publish the tile's digit counts, scatter the tile into
// shared memory in digit order, look back for the counts of the earlier tiles, write out.
// IDENT: the values are the positions (first pass of a sort of indices; vals_in is not read).
template <typename K, int ITEMS, int NT, bool IDENT>
__global__ void __launch_bounds__(NT, kSortThreads / NT) k_os_pass(
    const K *keys_in, const uint32_t *vals_in, K *__restrict__ keys_out,
    uint32_t *__restrict__ vals_out, int64_t n, int shift, int mask_bits,
    const uint32_t *ghist_pass, unsigned long long *status, uint32_t *ticket, uint32_t epoch,
    uint32_t *err, bool full_sum) {
    pdl_enter();
    constexpr int kSortItems = ITEMS, kSortTile = ITEMS * NT;
    constexpr int kSortWarps = NT / 32, kQuarters = NT / kRadix;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    PassSmem<K, ITEMS, NT> &S = *reinterpret_cast<PassSmem<K, ITEMS, NT> *>(sm_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int dg = threadIdx.x & (kRadix - 1), q = threadIdx.x / kRadix;
    const uint32_t mask = (1u << mask_bits) - 1u;
    for (int i = threadIdx.x; i < kSortWarps * kRadix; i += NT) {
        (&S.whist[0][0])[i] = 0;
        (&S.wmask[0][0])[i] = 0;
    }
    if (threadIdx.x == 0) {
        S.tile_id = atomicAdd(ticket, 1u);
        S.failed = 0u;
    }
    __syncthreads();
    const uint32_t tile = S.tile_id;
    if (tile >= kClosed) return;

    const int64_t tbase = (int64_t)tile * kSortTile;
    const int64_t wbase = tbase + (int64_t)warp * (32 * kSortItems);
    const bool full = tbase + kSortTile <= n;  // every tile but the last
    const uint32_t tile_count = full ? (uint32_t)kSortTile : (uint32_t)(n - tbase);
    const uint32_t gcount = q == 0 ? ghist_pass[dg] : 0u;
    K k[kSortItems];
    uint32_t v[kSortItems];
    uint32_t rank2[(kSortItems + 1) / 2];  // rank within the warp's digit run, two 16-bit ranks per word
    static_assert(32 * kSortItems < 65536, "16-bit ranks");
    const K *kin = keys_in + wbase + lane;
    const uint32_t *vin = vals_in + wbase + lane;
    const int left = full ? kSortTile : (int)(n - tbase) - warp * (32 * kSortItems);  // from the warp's first key
    auto load = [&](auto whole) {
#pragma unroll
        for (int r = 0; r < kSortItems; ++r) k[r] = decltype(whole)::value || r * 32 + lane < left ? kin[r * 32] : K(0);
#pragma unroll
        for (int r = 0; r < kSortItems; ++r)
            v[r] = IDENT ? (uint32_t)(wbase + r * 32 + lane)
                         : decltype(whole)::value || r * 32 + lane < left ? vin[r * 32] : 0u;
    };
    if (full) load(std::true_type());
    else load(std::false_type());
    // ranks within the warp: the lanes holding the same digit by a match instruction when a digit
    // recurs often (few distinct digits; judged by the first and the last keys), else by one
    // shared-memory OR per lane into the warp's digit masks (many distinct digits, where the
    // match instruction is slow)
    uint32_t *const wh = S.whist[warp], *const wm = S.wmask[warp];
    const uint32_t below = (1u << lane) - 1u;
    auto rank = [&](auto whole, auto by_match) {
        constexpr bool WHOLE = decltype(whole)::value, MATCH = decltype(by_match)::value;
#pragma unroll
        for (int r = 0; r < kSortItems; ++r) {
            const bool valid = WHOLE || r * 32 + lane < left;
            const uint32_t d = (uint32_t)(k[r] >> shift) & mask;
            unsigned peers = 0u;
            if (MATCH) {
                peers = __match_any_sync(0xffffffffu, valid ? d : (uint32_t)kRadix);
            } else {
                if (valid) atomicOr(wm + d, 1u << lane);
                __syncwarp();
                if (valid) peers = wm[d];
            }
            const uint32_t before = valid ? wh[d] : 0u;
            const uint32_t lower = peers & below;
            __syncwarp();
            if (valid && lower == 0u) {
                wh[d] = before + __popc(peers);
                if (!MATCH) wm[d] = 0u;  // clean for the next key
            }
            __syncwarp();
            const uint32_t rk = before + __popc(lower);
            if (r & 1) rank2[r >> 1] |= rk << 16;
            else rank2[r >> 1] = rk;
        }
    };
    {
        const uint32_t d0 = (uint32_t)(k[0] >> shift) & mask, d1 = (uint32_t)(k[kSortItems - 1] >> shift) & mask;
        const int same = __popc(__ballot_sync(0xffffffffu, d0 == __shfl_sync(0xffffffffu, d0, 0))) +
                         __popc(__ballot_sync(0xffffffffu, d1 == __shfl_sync(0xffffffffu, d1, 0)));
        if (full) {
            if (same >= 8) rank(std::true_type(), std::true_type());
            else rank(std::true_type(), std::false_type());
        } else {
            rank(std::false_type(), std::true_type());
        }
    }
    __syncthreads();
    // per digit: the count of each quarter's eight warps, then per-warp exclusive offsets
    {
        uint32_t c = 0;
#pragma unroll
        for (int w = 0; w < kSortWarps / kQuarters; ++w) c += S.whist[q * (kSortWarps / kQuarters) + w][dg];
        S.part[q][dg] = c;
    }
    __syncthreads();
    uint32_t count = 0, base = 0;  // the tile's count of digit dg; that of the quarters before q
#pragma unroll
    for (int qq = 0; qq < kQuarters; ++qq) {
        const uint32_t c = S.part[qq][dg];
        base += qq < q ? c : 0u;
        count += c;
    }
    // publish this tile's count of the digit at once, so later tiles can read past it
    volatile unsigned long long *st = status;
    if (q == 0) st[(uint64_t)tile * kRadix + dg] = os_pack(epoch, tile == 0 ? kStatePrefix : kStateAgg, count);
    // local and global digit starts (the global one from the pass's digit counts)
    uint32_t lst = 0, gdig = 0;
    if (q == 0) {  // the first eight warps
        lst = warp_inclusive_scan(count);
        gdig = warp_inclusive_scan(gcount);
        if (lane == 31) S.wsum[warp] = make_uint2(lst, gdig);
        lst -= count;
        gdig -= gcount;
    }
    __syncthreads();
    if (q == 0) {
        for (int w = 0; w < warp; ++w) {
            lst += S.wsum[w].x;
            gdig += S.wsum[w].y;
        }
        S.lstart[dg] = lst;
        S.lb_next[dg] = (int32_t)tile - 1;
    }
    __syncthreads();
    // per warp and digit: the place in the tile of the warp's first key of that digit
    base += S.lstart[dg];
#pragma unroll
    for (int w = 0; w < kSortWarps / kQuarters; ++w) {
        uint32_t &h = S.whist[q * (kSortWarps / kQuarters) + w][dg];
        const uint32_t t = h;
        h = base;
        base += t;
    }
    __syncthreads();
    // the tile in digit order in shared memory (frees the key registers before the look-back)
    auto scatter = [&](auto whole) {
#pragma unroll
        for (int r = 0; r < kSortItems; ++r) {
            if (!decltype(whole)::value && r * 32 + lane >= left) continue;
            const uint32_t d = (uint32_t)(k[r] >> shift) & mask;
            const uint32_t lpos = wh[d] + ((rank2[r >> 1] >> (16 * (r & 1))) & 0xffffu);
            S.keys[lpos] = k[r];
            S.vals[lpos] = v[r];
        }
    };
    if (full) scatter(std::true_type());
    else scatter(std::false_type());
    // decoupled look-back over the earlier tiles: per round trip, quarter q of digit dg reads
    // the 16 predecessors [j - 16 q - 15, j - 16 q] (j = nearest not yet added), adds the AGG
    // counts from its nearest down to the first PREFIX (included) or unpublished word
    // (excluded); the quarter-0 thread then joins the quarters in order.  Bounded wait.
    uint32_t excl = 0, spins = 0;
    int32_t next = (int32_t)tile - 1;  // quarter 0: nearest predecessor not yet added (-1: done)
    if (full_sum) {
        // few tiles: sum every earlier tile's own count (quarter q takes the tiles q, q + 4, ...,
        // eight loads in flight); no inclusive prefix is published or read.  Bounded waits.
        uint32_t sum = 0;
        for (int32_t i0 = q; i0 < (int32_t)tile; i0 += kQuarters * 8) {
            unsigned long long w[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int32_t i = i0 + kQuarters * u;
                w[u] = i < (int32_t)tile ? st[(uint64_t)i * kRadix + dg] : os_pack(epoch, kStateAgg, 0u);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int32_t i = i0 + kQuarters * u;
                uint32_t tries = 0;
                while (((uint32_t)(w[u] >> 34)) != epoch || ((uint32_t)(w[u] >> 32) & 3u) == 0u) {
                    if (++tries > kSpinLimit) {
                        S.failed = 1u;
                        break;
                    }
                    w[u] = st[(uint64_t)i * kRadix + dg];
                }
                sum += (uint32_t)w[u];
            }
        }
        S.lb_sum[q][dg] = sum;
        __syncthreads();
        if (q == 0)
#pragma unroll
            for (int qq = 0; qq < kQuarters; ++qq) excl += S.lb_sum[qq][dg];
        next = -1;
    }
    while (!full_sum) {
        const int32_t j = S.lb_next[dg];
        if (j >= 0) {
            const int32_t hi = j - kLbWords * q;
            unsigned long long w[kLbWords];
#pragma unroll
            for (int u = 0; u < kLbWords; ++u)
                w[u] = hi - u >= 0 ? st[(uint64_t)(hi - u) * kRadix + dg] : 0ull;
            uint32_t sum = 0, used = 0, kind = 0;
#pragma unroll
            for (int u = 0; u < kLbWords; ++u) {
                if (kind != 0 || hi - u < 0) continue;
                const uint32_t h32 = (uint32_t)(w[u] >> 32);
                if ((h32 >> 2) != epoch || (h32 & 3u) == 0u) {
                    kind = 2;
                    continue;
                }
                sum += (uint32_t)w[u];
                ++used;
                if ((h32 & 3u) == kStatePrefix) kind = 1;
            }
            S.lb_sum[q][dg] = sum;
            S.lb_used[q][dg] = used;
            S.lb_kind[q][dg] = kind;
        }
        __syncthreads();
        if (q == 0 && j >= 0) {
            int32_t nj = j;
            bool done = false, stalled = false;
#pragma unroll
            for (int qq = 0; qq < kQuarters; ++qq) {
                if (done || stalled) continue;
                excl += S.lb_sum[qq][dg];
                nj -= (int32_t)S.lb_used[qq][dg];
                const uint32_t kind = S.lb_kind[qq][dg];
                if (kind == 1 || nj < 0) done = true;
                else if (kind == 2) stalled = true;
            }
            if (stalled && ++spins > kSpinLimit) {
                S.failed = 1u;
                done = true;
            }
            next = done ? -1 : nj;
            S.lb_next[dg] = next;
        }
        // every digit done: the quarter-0 threads decide, read after this barrier
        if (__syncthreads_and(q != 0 || next < 0)) break;
    }
    if (q == 0) {
        if (tile > 0 && !full_sum) st[(uint64_t)tile * kRadix + dg] = os_pack(epoch, kStatePrefix, excl + count);
        S.goff[dg] = gdig + excl - lst;  // (plus the place in the tile; modulo 2^32)
    }
    __syncthreads();
    if (S.failed) {  // no places for this tile's keys
        if (threadIdx.x == 0) pass_failed(err, ticket, epoch);
        return;
    }
    auto put = [&](uint32_t i) {
        const K key = S.keys[i];
        const uint32_t gpos = S.goff[(uint32_t)(key >> shift) & mask] + i;
        keys_out[gpos] = key;
        vals_out[gpos] = S.vals[i];
    };
    if (full) {
#pragma unroll
        for (int r = 0; r < kSortItems; ++r) put(r * NT + threadIdx.x);
    } else {
        for (uint32_t i = threadIdx.x; i < tile_count; i += NT) put(i);
    }
}

// The passes of one sort.
template <typename K, int ITEMS, int NT>
bool run_passes(K *keys, uint32_t *vals, K *keys_alt, uint32_t *vals_alt, int64_t n, int begin_bit, int end_bit,
                const uint32_t *ghist, unsigned long long *status, uint32_t *tickets, uint32_t *err, bool identity,
                Lane s) {
    const int nb = (int)((n + (int64_t)ITEMS * NT - 1) / ((int64_t)ITEMS * NT));
    const int passes = (end_bit - begin_bit + 7) / 8;
    const size_t smem = sizeof(PassSmem<K, ITEMS, NT>);
    cudaFuncSetAttribute(k_os_pass<K, ITEMS, NT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_os_pass<K, ITEMS, NT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    bool flipped = false;
    K *kin = keys, *kout = keys_alt;
    uint32_t *vin = vals, *vout = vals_alt;
    for (int p = 0; p < passes; ++p) {
        const int shift = begin_bit + 8 * p;
        const int bits = (end_bit - shift) < 8 ? (end_bit - shift) : 8;
        auto kern = p == 0 && identity ? k_os_pass<K, ITEMS, NT, true> : k_os_pass<K, ITEMS, NT, false>;
        launch(kern, nb, NT, smem, s, kin, vin, kout, vout, n, shift, bits, ghist + p * kRadix, status, tickets + p,
                                            (uint32_t)(p + 1), err, nb <= kFullSumTiles);
        K *tk = kin; kin = kout; kout = tk;
        uint32_t *tv = vin; vin = vout; vout = tv;
        flipped = !flipped;
    }
    return flipped;
}

}  // namespace

uint32_t *sort_status_word(uint32_t *hist, int64_t n) {
    return hist + 2 * sort_tiles_for(n) * kRadix + kMaxPasses * kRadix + kMaxPasses;
}

template <typename K>
bool radix_sort_pairs(K *keys, uint32_t *vals, K *keys_alt, uint32_t *vals_alt, int64_t n,
                      int begin_bit, int end_bit, uint32_t *hist, Lane s, int *launches,
                      uint32_t *err_out, const uint32_t *digit_counts, bool hist_cleared, bool identity) {
    if (n <= 1 || end_bit <= begin_bit) {
        if (identity && n == 1) cudaMemsetAsync(vals, 0, sizeof(uint32_t), s);
        return false;
    }
    const int64_t nb = sort_tiles_for(n);
    unsigned long long *status = reinterpret_cast<unsigned long long *>(hist);  // 8-byte aligned
    uint32_t *ghist = hist + 2 * (size_t)nb * kRadix;
    uint32_t *tickets = ghist + kMaxPasses * kRadix;
    uint32_t *err = err_out ? err_out : sort_status_word(hist, n);
    if (!hist_cleared) cudaMemsetAsync(hist, 0, sizeof(uint32_t) * sort_hist_size(n), s);
    if (digit_counts) {
        ghist = const_cast<uint32_t *>(digit_counts);
    } else {
        const int64_t hb = (n + kHistThreads - 1) / kHistThreads;
        launch(k_os_hist<K>, hb < 1216 ? (int)hb : 1216, kHistThreads, 0, s, keys, n, begin_bit, end_bit, ghist);
        if (launches) *launches += 1;
    }
    if (launches) *launches += (end_bit - begin_bit + 7) / 8;
    auto run = [&](auto items, auto threads) {
        return run_passes<K, decltype(items)::value, decltype(threads)::value>(keys, vals, keys_alt, vals_alt, n, begin_bit, end_bit, ghist, status,
                                                     tickets, err, identity, s);
    };
    const std::integral_constant<int, kSortThreads> whole;
    switch (sort_items_for(n)) {
        case 2: return run(std::integral_constant<int, 2>(), whole);
        case 4: return run(std::integral_constant<int, 4>(), whole);
        case 8: return run(std::integral_constant<int, 8>(), whole);
    }
    if (sort_threads_for(n) == kSortThreads) return run(std::integral_constant<int, 13>(), whole);
    return run(std::integral_constant<int, 13>(), std::integral_constant<int, kSortThreads / 2>());
}

template bool radix_sort_pairs<uint32_t>(uint32_t *, uint32_t *, uint32_t *, uint32_t *, int64_t,
                                         int, int, uint32_t *, Lane, int *, uint32_t *,
                                         const uint32_t *, bool, bool);
template bool radix_sort_pairs<uint64_t>(uint64_t *, uint32_t *, uint64_t *, uint32_t *, int64_t,
                                         int, int, uint32_t *, Lane, int *, uint32_t *,
                                         const uint32_t *, bool, bool);

}  // namespace hca
