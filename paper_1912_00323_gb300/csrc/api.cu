// C ABI entry points (include/hca_dbscan.h): argument checks, the library's device memory
// pool, and dispatch to the per-(type, dimension) pipelines.
#include <math.h>
#include <string.h>

#include <mutex>
#include <vector>

#include "hca_internal.cuh"

namespace hca {

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_pool_mu;
cudaMemPool_t g_pools[kMaxDevices] = {};
int g_sms[kMaxDevices] = {};

cudaError_t get_pool(cudaMemPool_t *out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (!g_pools[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p;
        e = cudaMemPoolCreate(&p, &props);
        if (e != cudaSuccess) return e;
        uint64_t keep = ~0ull;  // keep freed blocks for reuse by later calls
        cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
        g_pools[dev] = p;
    }
    *out = g_pools[dev];
    return cudaSuccess;
}

bool finite_positive(double x) { return isfinite(x) && x > 0.0; }

}  // namespace

cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t s) {
    cudaMemPool_t pool;
    cudaError_t e = get_pool(&pool);
    if (e != cudaSuccess) return e;
    if (bytes == 0) bytes = 256;
    return cudaMallocFromPoolAsync(p, bytes, pool, s);
}

cudaError_t pool_free(void *p, cudaStream_t s) {
    if (!p) return cudaSuccess;
    return cudaFreeAsync(p, s);
}

int device_sm_count() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -1;
    if (g_sms[dev] <= 0) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
        g_sms[dev] = v;
    }
    return g_sms[dev];
}

int check_common(const void *pts, int32_t dtype, int64_t n, int32_t d, double eps,
                        int32_t min_pts, const void *labels) {
    if (n < 0 || n >= ((int64_t)1 << 31)) return HCA_EINVAL;
    if (d < 1 || d > 64) return HCA_EINVAL;
    if (dtype != HCA_F32 && dtype != HCA_F64) return HCA_EINVAL;
    if (!finite_positive(eps) || min_pts < 1) return HCA_EINVAL;
    if (n > 0 && (!pts || !labels)) return HCA_EINVAL;
    return HCA_OK;
}

template <typename T>
static int dispatch_t(const RunArgs &a) {
    // the hypercube stencil path exists for d <= 4, the coarse grid for d >= 3
    const int path = a.tune.path == 0 ? (a.d <= 4 ? 1 : 2) : a.tune.path;
    if (path == 1) {
        switch (a.d) {
            case 1: return run_lowd<T, 1>(a);
            case 2: return run_lowd<T, 2>(a);
            case 3: return run_lowd<T, 3>(a);
            case 4: return run_lowd<T, 4>(a);
        }
        return HCA_EINVAL;
    }
    if (path == 2 && a.d >= 3) {
        if (a.d <= 8) return run_hd<T, 8>(a);
        if (a.d <= 16) return run_hd<T, 16>(a);
        if (a.d <= 32) return run_hd<T, 32>(a);
        if (a.d <= 64) return run_hd<T, 64>(a);
    }
    return HCA_EINVAL;
}

int dispatch(const RunArgs &a, int32_t dtype) {
    return dtype == HCA_F32 ? dispatch_t<float>(a) : dispatch_t<double>(a);
}

int device_ex_tuned(const void *d_points, int32_t dtype, int64_t n, int32_t d, double eps, int32_t min_pts,
                    int32_t *d_labels, uint8_t *d_core, void *stream, hca_stats *stats, int32_t flags,
                    const hca_tuning &tune, double *ext_out) {
    int rc = check_common(d_points, dtype, n, d, eps, min_pts, d_labels);
    if (rc) return rc;
    if (stats) {
        hca_stats z = {};
        *stats = z;
    }
    if (n == 0) return HCA_OK;
    const size_t esz = dtype == HCA_F32 ? 4 : 8;
    if (((uintptr_t)d_points) % esz || ((uintptr_t)d_labels) % 4) return HCA_EINVAL;
    RunArgs a;
    a.d_points = d_points;
    a.n = n;
    a.d = d;
    a.eps = eps;
    a.min_pts = min_pts;
    a.d_labels = d_labels;
    a.d_core = d_core;
    a.stream = (cudaStream_t)stream;
    a.stats = stats;
    a.flags = flags;
    a.tune = tune;
    a.ext_out = ext_out;
    return dispatch(a, dtype);
}

int batched_tuned(const void *d_points, int32_t dtype, int32_t n_sets, const int64_t *offsets, int32_t d,
                  const double *eps, const int32_t *min_pts, int32_t *d_labels, uint8_t *d_core, void *stream,
                  hca_stats *stats, int32_t flags, const hca_tuning &tune, bool short_lists) {
    if (n_sets < 1 || !offsets || !eps || !min_pts) return HCA_EINVAL;
    if (offsets[0] != 0) return HCA_EINVAL;
    for (int32_t i = 0; i < n_sets; ++i) {
        if (offsets[i + 1] < offsets[i]) return HCA_EINVAL;
        if (!finite_positive(eps[i]) || min_pts[i] < 1) return HCA_EINVAL;
    }
    const int64_t n = offsets[n_sets];
    int rc = check_common(d_points, dtype, n, d, 1.0, 1, d_labels);
    if (rc) return rc;
    if (stats) {
        hca_stats z = {};
        *stats = z;
    }
    if (n == 0) return HCA_OK;
    const size_t esz = dtype == HCA_F32 ? 4 : 8;
    if (((uintptr_t)d_points) % esz || ((uintptr_t)d_labels) % 4) return HCA_EINVAL;
    RunArgs a;
    a.d_points = d_points;
    a.n = n;
    a.d = d;
    a.eps = eps[0];
    a.min_pts = min_pts[0];
    a.d_labels = d_labels;
    a.d_core = d_core;
    a.stream = (cudaStream_t)stream;
    a.stats = stats;
    a.flags = flags;
    a.nsets = n_sets;
    a.h_off = offsets;
    a.h_eps = eps;
    a.h_minpts = min_pts;
    a.tune = tune;
    a.short_lists = short_lists;
    return dispatch(a, dtype);
}

namespace {

// The graph a host thread keeps for repeated identical calls of hca_dbscan_device_ex: the key
// of its last call and, once that call repeated, a plan captured with the extents it measured.
struct CallKey {
    int dev = -1;
    unsigned long long ctx = 0;
    const void *pts = nullptr;
    int32_t *lab = nullptr;
    uint8_t *core = nullptr;
    int64_t n = 0;
    int32_t d = 0, dtype = 0, min_pts = 0, flags = 0;
    double eps = 0.0;
    hca_tuning tune = kDefaultTuning;
    bool operator==(const CallKey &o) const {
        return dev == o.dev && ctx == o.ctx && pts == o.pts && lab == o.lab && core == o.core && n == o.n &&
               d == o.d && dtype == o.dtype && min_pts == o.min_pts && flags == o.flags && eps == o.eps &&
               memcmp(&tune, &o.tune, sizeof(tune)) == 0;
    }
};

struct RepeatCache {
    bool have = false;  // key holds the thread's last call
    CallKey key;
    hca_plan *plan = nullptr;
    void drop() {
        if (plan) hca_plan_destroy(plan);
        plan = nullptr;
    }
};

thread_local RepeatCache t_repeat;

}  // namespace

}  // namespace hca

using namespace hca;

extern "C" int hca_dbscan_device_ex(const void *d_points, int32_t dtype, int64_t n, int32_t d,
                                    double eps, int32_t min_pts, int32_t *d_labels, uint8_t *d_core,
                                    void *stream, hca_stats *stats, int32_t flags) {
    const hca_tuning tune = tuning_for(d);
    if ((flags & (HCA_FLAG_TIMING | HCA_FLAG_NO_GRAPH_CACHE)) || n <= 0 ||
        check_common(d_points, dtype, n, d, eps, min_pts, d_labels) != HCA_OK)
        return device_ex_tuned(d_points, dtype, n, d, eps, min_pts, d_labels, d_core, stream, stats, flags, tune);
    CallKey k;
    if (cudaGetDevice(&k.dev) != cudaSuccess) return HCA_ECUDA;
    k.ctx = current_context_id();
    k.pts = d_points;
    k.lab = d_labels;
    k.core = d_core;
    k.n = n;
    k.d = d;
    k.dtype = dtype;
    k.min_pts = min_pts;
    k.flags = flags;
    k.eps = eps;
    k.tune = tune;
    RepeatCache &c = t_repeat;
    const bool same = c.have && k.ctx != 0 && c.key == k;
    if (same && c.plan) {
        int rc = hca_plan_launch(c.plan, stream);
        if (rc == HCA_OK) rc = hca_plan_wait(c.plan, stream, stats);
        if (rc != HCA_ERANGE) return rc;
        c.drop();  // points outside the captured extents: run the call afresh
    }
    std::vector<double> ext((size_t)2 * d, 0.0);
    const int rc = device_ex_tuned(d_points, dtype, n, d, eps, min_pts, d_labels, d_core, stream, stats, flags,
                                   tune, ext.data());
    if (rc != HCA_OK) return rc;
    if (same && !c.plan) {
        // the call repeated: capture it with the extents it measured (a failure, e.g. no memory
        // for a second workspace, only leaves the calls uncached; a graph with shorter neighbour
        // lists than the direct call has would be slower than it)
        hca_plan *p = nullptr;
        if (plan_create_single(&p, d_points, dtype, n, d, eps, min_pts, ext.data(), ext.data() + d, d_labels,
                               d_core, flags, true) == HCA_OK)
            c.plan = p;
        cudaGetLastError();
    } else if (!same) {
        c.drop();
        c.key = k;
        c.have = true;
    }
    return HCA_OK;
}

extern "C" int hca_graph_cache_release(void) {
    t_repeat.drop();
    t_repeat.have = false;
    return HCA_OK;
}

extern "C" int hca_dbscan_batched(const void *d_points, int32_t dtype, int32_t n_sets, const int64_t *offsets,
                                  const int32_t *d_per_set, const double *eps, const int32_t *min_pts,
                                  int32_t *d_labels, uint8_t *d_core, void *stream, hca_stats *stats, int32_t flags) {
    return batched_mixed(d_points, dtype, n_sets, offsets, d_per_set, eps, min_pts, d_labels, d_core, stream,
                         stats, flags, nullptr);
}

extern "C" int hca_dbscan_device(const void *d_points, int32_t dtype, int64_t n, int32_t d, double eps,
                                 int32_t min_pts, int32_t *d_labels, void *stream) {
    return hca_dbscan_device_ex(d_points, dtype, n, d, eps, min_pts, d_labels, nullptr, stream, nullptr, 0);
}

extern "C" int hca_dbscan(const void *points, int32_t dtype, int64_t n, int32_t d, double eps,
                          int32_t min_pts, int32_t *labels) {
    int rc = check_common(points, dtype, n, d, eps, min_pts, labels);
    if (rc) return rc;
    if (n == 0) return HCA_OK;
    // one non-blocking stream per host thread and device, created on first use and kept
    thread_local cudaStream_t streams[kMaxDevices] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return HCA_ECUDA;
    if (!streams[dev] && cudaStreamCreateWithFlags(&streams[dev], cudaStreamNonBlocking) != cudaSuccess) {
        streams[dev] = nullptr;
        return HCA_ECUDA;
    }
    cudaStream_t s = streams[dev];
    const size_t in_bytes = (size_t)n * d * (dtype == HCA_F32 ? 4 : 8);
    void *dp = nullptr, *dl = nullptr;
    if (pool_alloc(&dp, in_bytes, s) != cudaSuccess || pool_alloc(&dl, (size_t)n * 4, s) != cudaSuccess) {
        pool_free(dp, s);
        cudaStreamSynchronize(s);
        return HCA_ENOMEM;
    }
    rc = HCA_OK;
    if (cudaMemcpyAsync(dp, points, in_bytes, cudaMemcpyHostToDevice, s) != cudaSuccess) rc = HCA_ECUDA;
    if (rc == HCA_OK) rc = hca_dbscan_device(dp, dtype, n, d, eps, min_pts, (int32_t *)dl, (void *)s);
    if (rc == HCA_OK &&
        (cudaMemcpyAsync(labels, dl, (size_t)n * 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
         cudaStreamSynchronize(s) != cudaSuccess))
        rc = HCA_ECUDA;
    pool_free(dp, s);
    pool_free(dl, s);
    cudaStreamSynchronize(s);
    return rc;
}

namespace hca {

int workspace_bound(int64_t n, int32_t d, int32_t dtype, int32_t flags, int32_t min_pts, bool short_lists,
                    int64_t *bytes) {
    if (!bytes) return HCA_EINVAL;
    if (n < 0 || n >= ((int64_t)1 << 31) || d < 1 || d > 64) return HCA_EINVAL;
    if (dtype != HCA_F32 && dtype != HCA_F64) return HCA_EINVAL;
    *bytes = 0;
    if (n == 0) return HCA_OK;
    RunArgs a;
    a.d_points = nullptr;
    a.n = n;
    a.d = d;
    a.eps = 1.0;
    a.min_pts = min_pts;
    a.short_lists = short_lists;
    a.d_labels = nullptr;
    a.d_core = nullptr;
    a.stream = nullptr;
    a.stats = nullptr;
    a.flags = flags;
    a.tune = tuning_for(d);
    size_t b = 0;
    a.ws_query = &b;
    const int rc = dispatch(a, dtype);
    if (rc == HCA_OK) *bytes = (int64_t)b;
    return rc;
}

}  // namespace hca

extern "C" int hca_workspace_bytes(int64_t n, int32_t d, int32_t dtype, int32_t flags, int64_t *bytes) {
    return workspace_bound(n, d, dtype, flags, INT32_MAX, false, bytes);  // (the bound of any MINPTS)
}

extern "C" int hca_radix_sort_pairs(void *d_keys, uint32_t *d_vals, int64_t n, int32_t key_bytes,
                                    int32_t begin_bit, int32_t end_bit, void *stream) {
    if (n < 0 || n >= ((int64_t)1 << 31)) return HCA_EINVAL;
    if (key_bytes != 4 && key_bytes != 8) return HCA_EINVAL;
    if (begin_bit < 0 || end_bit <= begin_bit || end_bit > 8 * key_bytes) return HCA_EINVAL;
    if (n > 0 && (!d_keys || !d_vals)) return HCA_EINVAL;
    if (((uintptr_t)d_keys) % key_bytes || ((uintptr_t)d_vals) % 4) return HCA_EINVAL;
    if (n <= 1) return HCA_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t hist = sort_hist_size(n);
    const size_t bytes = (size_t)n * key_bytes + (size_t)n * 4 + 4 * hist + 512;
    void *ws = nullptr;
    if (pool_alloc(&ws, bytes, s) != cudaSuccess) return HCA_ENOMEM;
    char *b = (char *)ws;
    void *kalt = b;
    uint32_t *valt = (uint32_t *)(b + (((size_t)n * key_bytes + 255) & ~(size_t)255));
    uint32_t *h = (uint32_t *)((char *)valt + (((size_t)n * 4 + 255) & ~(size_t)255));
    bool flipped;
    if (key_bytes == 4)
        flipped = radix_sort_pairs<uint32_t>((uint32_t *)d_keys, d_vals, (uint32_t *)kalt, valt, n,
                                             begin_bit, end_bit, h, s, nullptr);
    else
        flipped = radix_sort_pairs<uint64_t>((uint64_t *)d_keys, d_vals, (uint64_t *)kalt, valt, n,
                                             begin_bit, end_bit, h, s, nullptr);
    int rc = HCA_OK;
    if (flipped) {
        if (cudaMemcpyAsync(d_keys, kalt, (size_t)n * key_bytes, cudaMemcpyDeviceToDevice, s) != cudaSuccess ||
            cudaMemcpyAsync(d_vals, valt, (size_t)n * 4, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
            rc = HCA_ECUDA;
    }
    uint32_t status = 0;
    if (cudaMemcpyAsync(&status, sort_status_word(h, n), sizeof(status), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        rc = HCA_ECUDA;
    if (cudaGetLastError() != cudaSuccess) rc = HCA_ECUDA;
    pool_free(ws, s);
    if (cudaStreamSynchronize(s) != cudaSuccess) rc = HCA_ECUDA;
    if (rc == HCA_OK && status) rc = HCA_EDEVICE;
    return rc;
}

extern "C" const char *hca_strerror(int code) {
    switch (code) {
        case HCA_OK: return "success";
        case HCA_EINVAL: return "invalid argument";
        case HCA_ENOMEM: return "device workspace allocation failed";
        case HCA_ECUDA: return "CUDA runtime error";
        case HCA_ERANGE: return "coordinate extent too large for the cell grid at this eps";
        case HCA_ENOTIMPL: return "not implemented in this build";
        case HCA_EDEVICE: return "device-side consistency check failed";
        case HCA_ETOOLARGE: return "input larger than the fixed scratch of the no-allocation entry point";
        case HCA_ETIMEDOUT: return "timed out";
        case HCA_ECANCELED: return "cancelled";
        case HCA_EBUSY: return "busy";
    }
    return "unknown error";
}

extern "C" int32_t hca_version(void) { return 101; }
