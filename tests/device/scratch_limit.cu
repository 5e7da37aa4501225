// Coarse-grid calls whose workspace does not fit: the library's objects linked with a pool_alloc that
// refuses what is above a limit.  Prints one line per check, "ok" or "FAIL".
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include <string>
#include <vector>

#include "hca_internal.cuh"

// (the linker's --wrap sends the library's calls of hca::pool_alloc here)
extern "C" cudaError_t __real__ZN3hca10pool_allocEPPvmP11CUstream_st(void **p, size_t bytes, cudaStream_t s);
static size_t g_limit = ~(size_t)0;   // refuse allocations above it ...
static int g_refuse = -1;             // ... all of them, or only this one of them
static int g_above = 0;
extern "C" cudaError_t __wrap__ZN3hca10pool_allocEPPvmP11CUstream_st(void **p, size_t bytes, cudaStream_t s) {
    if (bytes > g_limit && (g_refuse < 0 || g_above++ == g_refuse)) return cudaErrorMemoryAllocation;
    return __real__ZN3hca10pool_allocEPPvmP11CUstream_st(p, bytes, s);
}

static int g_bad = 0;
static void check(bool ok, const std::string &what) {
    printf("%s %s\n", ok ? "ok" : "FAIL", what.c_str());
    g_bad += ok ? 0 : 1;
}

static double uniform() { return rand() / (RAND_MAX + 1.0); }

// Clumps of 3 to 300 points in the box [0, 40]^d, noise between them, on a 1/64 lattice.
template <typename T>
static std::vector<T> clumps(int n, int d) {
    std::vector<T> x((size_t)n * d);
    srand(100 * d + (int)sizeof(T));
    for (int i = 0; i < n;) {
        const int m = 3 + rand() % 300;
        std::vector<double> c(d);
        for (double &v : c) v = 40 * uniform();
        const double w = rand() % 4 ? 0.5 + uniform() : 20.0;
        for (int k = 0; k < m && i < n; ++k, ++i)
            for (int j = 0; j < d; ++j) x[(size_t)i * d + j] = (T)(floor(64 * (c[j] + w * (2 * uniform() - 1))) / 64);
    }
    return x;
}

template <typename T>
static void run(int n, int d, int min_pts) {
    const int32_t dtype = sizeof(T) == 4 ? HCA_F32 : HCA_F64;
    const double eps = 0.25 * floor(4 * 0.75 * sqrt((double)d));
    const std::string what = "d " + std::to_string(d) + (sizeof(T) == 4 ? " float" : " double") + " MINPTS " + std::to_string(min_pts) + ": ";
    const std::vector<T> x = clumps<T>(n, d);
    T *dx;
    int32_t *dl;
    cudaMalloc((void **)&dx, x.size() * sizeof(T));
    cudaMalloc((void **)&dl, 4 * (size_t)n);
    cudaMemcpy(dx, x.data(), x.size() * sizeof(T), cudaMemcpyHostToDevice);
    auto labels = [&]() {
        std::vector<int32_t> l(n);
        cudaDeviceSynchronize();
        cudaMemcpy(l.data(), dl, 4 * (size_t)n, cudaMemcpyDeviceToHost);
        cudaMemset(dl, 0x55, 4 * (size_t)n);
        return l;
    };
    auto call = [&](int32_t flags, hca_stats &st) {
        return hca_dbscan_device_ex(dx, dtype, n, d, eps, min_pts, dl, nullptr, nullptr, &st, flags);
    };
    hca_stats st = {}, small = {};
    g_limit = ~(size_t)0;
    int rc = call(HCA_FLAG_NO_GRAPH_CACHE, st);
    const std::vector<int32_t> want = labels();
    const size_t whole = (size_t)st.workspace_bytes;
    check(rc == HCA_OK && st.n_clusters > 0 && st.n_noise > 5, what + "a call with memory");
    g_limit = whole - 1;
    rc = call(HCA_FLAG_NO_GRAPH_CACHE, small);
    // lists that the table's space (12 bytes a slot, a power of two of at least 2 n slots) holds whole are
    // not shortened: then nothing fits
    int64_t slots = 64;
    while (slots < 2 * (int64_t)n) slots <<= 1;
    const int entries = min_pts <= 9 ? 8 : min_pts <= 13 ? 12 : 20;
    const bool longer = 4ll * entries * n > 12 * slots;
    check(rc == (longer ? HCA_OK : HCA_ENOMEM), what + "a call without memory for its lists");
    check(!longer || (small.workspace_bytes > 0 && (size_t)small.workspace_bytes < whole), what + "its workspace");
    if (rc == HCA_OK) check(labels() == want, what + "its labels");
    // a plan (its box: the points' own)
    std::vector<double> mn(d, 1e300), mx(d, -1e300);
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < d; ++j) {
            const double v = (double)x[(size_t)i * d + j];
            mn[j] = v < mn[j] ? v : mn[j];
            mx[j] = v > mx[j] ? v : mx[j];
        }
    hca_plan *p = nullptr;
    rc = hca_plan_create(&p, dx, dtype, n, d, eps, min_pts, mn.data(), mx.data(), dl, nullptr);
    check(rc == (longer ? HCA_OK : HCA_ENOMEM), what + "a plan without memory for its lists");
    if (rc == HCA_OK) {
        check(hca_plan_launch(p, nullptr) == HCA_OK && hca_plan_wait(p, nullptr, nullptr) == HCA_OK && labels() == want,
              what + "its labels");
        hca_plan_destroy(p);
    }
    if (longer) {
        // the repeated call: the first two run directly with whole lists, the graph's workspace is refused,
        // and the third runs directly again
        hca_graph_cache_release();
        g_refuse = 2;
        g_above = 0;
        bool all = true;
        for (int k = 0; k < 3; ++k) {
            rc = call(0, st);
            all &= rc == HCA_OK && (size_t)st.workspace_bytes == whole && labels() == want;
        }
        check(all, what + "repeated calls without memory for a graph's lists");
        g_refuse = -1;
        hca_graph_cache_release();
    }
    cudaFree(dx);
    cudaFree(dl);
}

int main() {
    for (int min_pts : {2, 5, 6, 12, 21, 30, 200}) {
        run<float>(16384, 5, min_pts);  // (a slot table with no slack: lists of four)
        run<float>(12000, 9, min_pts);
        run<float>(5000, 24, min_pts);
        run<double>(12000, 7, min_pts);
        run<double>(5000, 16, min_pts);
    }
    return g_bad != 0 || cudaDeviceSynchronize() != cudaSuccess;
}
