// Waits of sorts and scans that run out, with the limit at 256 polls: a tile that nobody takes (its ticket
// is spent beforehand) is what the later tiles wait for.  Prints one line per check, "ok" or "FAIL".
#define HCA_LOOK_SPINS 256u
#include <stdio.h>

#include <functional>
#include <string>
#include <vector>

#include "sort.cu"
#include "tc_kernels.cuh"

using namespace hca;

static int g_bad = 0;
static void check(bool ok, const std::string &what) {
    printf("%s %s\n", ok ? "ok" : "FAIL", what.c_str());
    g_bad += ok ? 0 : 1;
}

template <typename T>
struct Dev {
    T *p = nullptr;
    size_t n;
    explicit Dev(size_t count, int byte = 0) : n(count) {
        cudaMalloc((void **)&p, n * sizeof(T));
        cudaMemset(p, byte, n * sizeof(T));
    }
    explicit Dev(const std::vector<T> &v) : n(v.size()) {
        cudaMalloc((void **)&p, n * sizeof(T));
        put(v);
    }
    void put(const std::vector<T> &v) { cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice); }
    std::vector<T> get() const {
        std::vector<T> v(n);
        cudaDeviceSynchronize();
        cudaMemcpy(v.data(), p, n * sizeof(T), cudaMemcpyDeviceToHost);
        return v;
    }
    ~Dev() { cudaFree(p); }
};

constexpr uint32_t kGuard = 0x0b0b0b0bu;
constexpr int kPast = 64;  // guarded words behind every output

struct One {
    __device__ uint32_t operator()(int64_t) const { return 1u; }
};
struct Nothing {
    __device__ void operator()(int64_t, uint32_t, uint32_t) const {}
};

static void scans() {
    const int64_t m = 4 * kScanTileElems + 7;
    Dev<unsigned char> look(look_bytes(m));
    Dev<uint32_t> out(m + kPast, 0x0b), out2(m + kPast, 0x0b), total(2, 0x0b), err(1);
    LookBack l = LookBack::at(look.p);
    const uint32_t one = 1;
    cudaMemcpy(l.tickets + 1, &one, 4, cudaMemcpyHostToDevice);  // tile 0 of the first scan is never taken
    k_scan_fn<One, Nothing><<<5, kTileThreads>>>(One(), Nothing(), out.p, m, nullptr, total.p, l, 1u, err.p);
    check(err.get()[0] == kErrLook, "scan: the status word");
    const std::vector<uint32_t> o = out.get();
    bool none = total.get()[0] == kGuard;
    for (uint32_t x : o) none &= x == kGuard;
    check(none, "scan: the tiles that waited write nothing");
    k_scan_fn<One, Nothing><<<5, kTileThreads>>>(One(), Nothing(), out2.p, m, nullptr, total.p + 1, l, 2u, err.p);
    none = total.get()[1] == kGuard;
    for (uint32_t x : out2.get()) none &= x == kGuard;
    check(none, "scan: the next one does nothing");
}

static void cells() {
    const int64_t n = 3 * kScanTileElems + 5;
    std::vector<uint32_t> keys(n), idx(n);
    for (int64_t i = 0; i < n; ++i) keys[i] = (uint32_t)i / 3, idx[i] = (uint32_t)i;
    Dev<uint32_t> dk(keys), di(idx), cell_of(n + kPast, 0x0b), start(n + 1 + kPast, 0x0b), pencil(n + 1 + kPast, 0x0b);
    Dev<uint64_t> ckey(n + kPast, 0x0b);
    Dev<float> in(2 * n);
    Dev<Pt<float, 2>> pts(n);
    Dev<unsigned char> look(look_bytes(n));
    Dev<DevCounters> ctr(1);
    CellsArgs<uint32_t> a;
    a.keys = dk.p;
    a.idx = di.p;
    a.n = n;
    a.prefix_shift = 2;
    a.cell_of = cell_of.p;
    a.cell_start = start.p;
    a.cell_key = ckey.p;
    a.pencil_start = pencil.p;
    a.ptab = nullptr;
    a.l = LookBack::at(look.p);
    a.ctr = ctr.p;
    const uint32_t one = 1;
    cudaMemcpy(a.l.tickets, &one, 4, cudaMemcpyHostToDevice);
    k_cells<float, 2, uint32_t><<<4, kTileThreads>>>(in.p, a, pts.p);
    check(ctr.get()[0].status == kErrLook, "cells: the status word");
    bool none = ctr.get()[0].n_cells == 0 && ctr.get()[0].n_pencils == 0;
    for (auto *b : {&cell_of, &start, &pencil})
        for (uint32_t x : b->get()) none &= x == kGuard;
    check(none, "cells: the tiles that waited write nothing");
}

// Two passes, the first with one block less than it has tiles (the blocks take the tiles from 1 on).
template <typename K, int ITEMS, int NT>
static void sort_of(int64_t n, bool full_sum, const char *what) {
    std::vector<K> keys(n);
    std::vector<uint32_t> vals(n);
    uint32_t x = 12345;
    for (int64_t i = 0; i < n; ++i) {
        x = x * 1664525u + 1013904223u;
        keys[i] = (K)(x >> 16);
        vals[i] = (uint32_t)i;
    }
    const int nb = (int)((n + (int64_t)ITEMS * NT - 1) / ((int64_t)ITEMS * NT));
    Dev<K> k(keys), ka(n + kPast, 0x0b);
    Dev<uint32_t> v(vals), va(n + kPast, 0x0b), ghist(kMaxPasses * kRadix), tickets(kMaxPasses), err(1);
    Dev<unsigned long long> status((size_t)nb * kRadix);
    std::vector<uint32_t> t(kMaxPasses, 0u);
    t[0] = 1;
    tickets.put(t);
    k_os_hist<K><<<64, kHistThreads>>>(k.p, n, 0, 16, ghist.p);
    const size_t smem = sizeof(PassSmem<K, ITEMS, NT>);
    auto kern = k_os_pass<K, ITEMS, NT, false>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<nb - 1, NT, smem>>>(k.p, v.p, ka.p, va.p, n, 0, 8, ghist.p, status.p, tickets.p, 1u, err.p, full_sum);
    check(err.get()[0] == kErrLook, std::string(what) + ": the status word");
    const std::vector<K> g = ka.get();
    const std::vector<uint32_t> gv = va.get();
    bool past = true, in = true;
    for (int i = 0; i < kPast; ++i) past &= gv[n + i] == kGuard && (uint32_t)g[n + i] == kGuard;
    for (int64_t i = 0; i < n; ++i) in &= gv[i] == kGuard || gv[i] < (uint32_t)n;
    check(past && in, std::string(what) + ": nothing behind the output");
    kern<<<nb, NT, smem>>>(ka.p, va.p, k.p, v.p, n, 8, 8, ghist.p + kRadix, status.p, tickets.p + 1, 2u, err.p, full_sum);
    check(k.get() == keys && v.get() == vals, std::string(what) + ": the second pass does nothing");
}

// The kernels after a failure: valid small tables that they would work on, and the status word set.
template <int D>
struct Views {
    static constexpr int n = 1000, C = 100, NA = 9;
    std::vector<uint32_t> zero, tens, ones, ident;
    Dev<unsigned char> ws;
    Dev<DevCounters> ctr;
    size_t at = 0;
    std::vector<unsigned char> before;
    LowdView<float, D> v;
    HdView<float, 16> h;
    tc::Tables tt;

    template <typename T>
    T *take(size_t count, const std::vector<T> *init = nullptr, int byte = 0) {
        T *p = (T *)(ws.p + at);
        cudaMemset(p, byte, count * sizeof(T));
        if (init) cudaMemcpy(p, init->data(), init->size() * sizeof(T), cudaMemcpyHostToDevice);
        at += (count * sizeof(T) + 511) & ~(size_t)255;
        return p;
    }
    Views() : ws(1 << 22), ctr(1) {
        std::vector<uint32_t> start(C + 1), chunk(C + 1), perm(n), cell(n);
        std::vector<uint64_t> key(C);
        for (int c = 0; c <= C; ++c) start[c] = 10u * c, chunk[c] = c;
        for (int c = 0; c < C; ++c) key[c] = c;
        for (int j = 0; j < n; ++j) perm[j] = j, cell[j] = j / 10;
        memset(&v, 0, sizeof(v));
        memset(&h, 0, sizeof(h));
        v.g.n = n;
        v.g.min_pts = 5;
        v.g.eps2 = 1.0;
        v.g.hi32 = INFINITY;
        v.g.inv_side = v.g.inv_side_f = 1.f;
        for (int i = 0; i < kMaxD; ++i) v.g.ncell[i] = 1000, v.g.bits[i] = i == D - 1 ? 10 : 4;
        v.g.prefix_shift = 10;
        for (int i = 0; i < D - 1; ++i) v.g.shift[i] = 10 + 4 * (D - 2 - i);
        v.pts = take<Pt<float, D>>(n);
        v.perm = take<uint32_t>(n, &perm);
        v.cell_of = take<uint32_t>(n, &cell);
        v.cell_start = take<uint32_t>(C + 1, &start);
        v.cell_key = take<uint64_t>(C, &key);
        std::vector<uint32_t> ps = {0u, (uint32_t)C};
        v.pencil_start = take<uint32_t>(C + 1, &ps);
        v.hkeys = take<uint64_t>(64, nullptr, 0xff);
        v.hvals = take<uint32_t>(64);
        v.ptab = take<uint32_t>(1 << 12);
        v.core = take<uint8_t>(n, nullptr, 1);
        v.cell_core = take<uint8_t>(C, nullptr, 1);
        v.parent = take<uint32_t>(n);
        v.reps = take<uint64_t>((size_t)n * 26, nullptr, 0);
        v.rep_pts = take<Pt<float, D>>((size_t)n * 26, nullptr, 7);
        v.comp_min = take<uint32_t>(n);
        v.ranges = take<uint2>((size_t)n * 16);
        v.list_count = take<uint32_t>(n, nullptr, 7);
        v.list_core = take<uint32_t>(n, nullptr, 7);
        v.list_label = take<uint32_t>(n, nullptr, 7);
        v.labels = take<int32_t>(n, nullptr, 7);
        v.core_out = take<uint8_t>(n, nullptr, 7);
        v.ctr = ctr.p;
        h.g = v.g;
        h.d = 16;
        h.n_all = NA;
        h.n_half = 5;
        for (int k = 0; k < NA; ++k) h.near[k] = (uint8_t)k;
        h.pts = take<float>((size_t)n * 16);
        h.fpts = h.pts;
        h.perm = v.perm;
        h.cell_of = v.cell_of;
        h.cell_start = v.cell_start;
        h.chunk_off = take<uint32_t>(C + 1, &chunk);
        h.cell_key = v.cell_key;
        h.ranges = v.ranges;
        h.core = v.core;
        h.cell_core = v.cell_core;
        h.parent = v.parent;
        h.comp_min = v.comp_min;
        h.labels = v.labels;
        h.core_out = v.core_out;
        h.ctr = ctr.p;
        h.box_lo = take<float>((size_t)n * 16, nullptr, 7);
        h.box_hi = take<float>((size_t)n * 16, nullptr, 7);
        h.sp_queue = take<uint2>(n);
        h.sp_pending = take<uint32_t>(n);
        h.sp_val = take<uint32_t>(n);
        h.sp_cap = n;
        h.nl = take<uint32_t>((size_t)n * 8);
        h.nl_cnt = take<uint32_t>(n, nullptr, 7);
        h.nl_k = 8;
        h.cell_root = take<uint32_t>(C);
        std::vector<uint32_t> many(C, 9u);
        h.odd_cnt = take<uint32_t>(C, &many);
        h.odd_mask = take<uint32_t>(n, nullptr, 7);
        std::vector<uint32_t> cx(n + 1);
        for (int j = 0; j <= n; ++j) cx[j] = j;
        h.cx = take<uint32_t>(n + 1, &cx);
        h.tc_cnt = take<uint32_t>(n);
        h.tc_pos = take<uint32_t>(n);
        tt = tc::Tables{h.chunk_off, h.cx, v.perm, v.perm, take<uint32_t>(n), h.chunk_off};
        DevCounters c;
        memset(&c, 0, sizeof(c));
        c.n_cells = C;
        c.n_pencils = 1;
        c.hash_mask = 63;
        c.n_chunks = C;
        for (int i = 0; i < 4; ++i) c.n_tc_chunks[i] = C;
        c.n_tc_recount = C;
        c.status = kErrLook;
        cudaMemcpy(ctr.p, &c, sizeof(c), cudaMemcpyHostToDevice);
        before = ws.get();
    }
    bool same() { return ws.get() == before; }
};

static void after_failure() {
    Views<2> w;
    Stencil st;
    memset(&st, 0, sizeof(st));
    st.n_all = st.n_half = 1;
    st.reach[0] = 1;
    auto run = [&](const char *what, std::function<void()> f) {
        f();
        const bool ran = cudaDeviceSynchronize() == cudaSuccess;
        check(ran && w.same(), std::string("after a failure: ") + what);
    };
    const int64_t n = w.n;
    run("k_hash_init clears no more than its least part", [&] { k_hash_init<<<1, 256>>>(w.v.hkeys, w.ctr.p); });
    run("k_pencils", [&] { k_pencils<<<1, 256>>>(w.v.cell_key, 10, w.v.pencil_start, w.v.hkeys, w.v.hvals, w.ctr.p); });
    run("k_ranges", [&] { k_ranges<float, 2><<<1, 256>>>(w.v, st); });
    {
        k_triage<float, 2><<<1, 256>>>(w.v, 1);
        cudaDeviceSynchronize();
        std::vector<uint8_t> core(n);
        cudaMemcpy(core.data(), w.v.core, n, cudaMemcpyDeviceToHost);
        bool clear = true;
        for (uint8_t x : core) clear &= x == 0;
        memcpy(w.before.data() + ((unsigned char *)w.v.core - w.ws.p), core.data(), n);
        check(clear && w.same(), "after a failure: k_triage leaves no core point and nothing else");
    }
    run("k_reps", [&] { k_reps<float, 2, 32><<<8, 32 * kRepWarps>>>(w.v, n); });
    run("k_rep_fix", [&] { k_rep_fix<float, 2, 32><<<8, 256>>>(w.v, n); });
    run("k_label_core", [&] { k_label_core<float, 2><<<4, 256>>>(w.v); });
    const size_t smem = 4 * 32 * 16 * sizeof(float);
    run("k_cell_box_hd", [&] { k_cell_box_hd<float, 16, float><<<4, 256>>>(w.h); });
    run("k_cell_box_decode", [&] { k_cell_box_decode<float, 16, float><<<4, 256>>>(w.h); });
    run("k_count_hd", [&] { k_count_hd<float, 16, false, true><<<4, 128, smem>>>(w.h); });
    run("k_cell_link", [&] { k_cell_link<float, 16, true><<<4, 128, smem>>>(w.h); });
    run("k_cell_odd", [&] { k_cell_odd<float, 16><<<4, 256>>>(w.h); });
    run("k_cell_mixed", [&] { k_cell_mixed<float, 16><<<4, 256>>>(w.h); });
    run("k_odd_hd", [&] { k_odd_hd<float, 16, false, true><<<4, 128, smem>>>(w.h); });
    run("k_merge_hd", [&] { k_merge_hd<float, 16, true><<<4, 128, smem>>>(w.h); });
    run("k_list_labels", [&] { k_list_labels<float, 16><<<4, 256>>>(w.h); });
    run("k_labels_hd", [&] { k_labels_hd<float, 16, false, true><<<4, 128, smem>>>(w.h); });
    run("k_tc_core_labels", [&] { tc::k_tc_core_labels<16><<<4, 256>>>(w.h, w.tt, 0, (uint32_t *)w.tt.core_lab); });
    const size_t tsm = tc::smem_bytes<16>();
    cudaFuncSetAttribute(tc::k_tc_hd<16, tc::kCount>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tsm);
    cudaFuncSetAttribute(tc::k_tc_hd<16, tc::kMerge>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tsm);
    cudaFuncSetAttribute(tc::k_tc_hd<16, tc::kLabels>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tsm);
    run("k_tc_hd counts", [&] { tc::k_tc_hd<16, tc::kCount><<<4, tc::kTile, tsm>>>(w.h, w.tt); });
    run("k_tc_hd unions", [&] { tc::k_tc_hd<16, tc::kMerge><<<4, tc::kTile, tsm>>>(w.h, w.tt); });
    run("k_tc_hd labels", [&] { tc::k_tc_hd<16, tc::kLabels><<<4, tc::kTile, tsm>>>(w.h, w.tt); });
    // (the same tables without the failure are worked on)
    const uint32_t none = 0;
    cudaMemcpy(&w.ctr.p->status, &none, 4, cudaMemcpyHostToDevice);
    k_triage<float, 2><<<1, 256>>>(w.v, 1);
    check(!w.same(), "without a failure: k_triage");
}

int main() {
    scans();
    cells();
    sort_of<uint32_t, 2, 1024>(10000, true, "sort, sums of all tiles");
    sort_of<uint64_t, 13, 512>(100000, false, "sort, look-back");
    after_failure();
    return g_bad != 0 || cudaDeviceSynchronize() != cudaSuccess;
}
