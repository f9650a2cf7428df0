// Host checks of plan.cpp and plan_sums.cpp without a GPU: the program links
// them with a CUDA runtime of its own (host memory; allocation number g_refuse
// fails) and is built with the undefined-behaviour sanitizer.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <ctime>
#include <string>

#include "../paper_2606_27262_gb300/csrc/sp_internal.h"

static int64_t g_refuse = -1, g_asked = 0, g_live = 0;  // g_live: allocations not freed

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) {
    if (g_asked++ == g_refuse) return cudaErrorMemoryAllocation;
    *p = std::malloc(n);
    ++g_live;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    g_live -= p != nullptr;
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 227 * 1024;
    return cudaSuccess;
}
int sp_autotune_dedisperse(const double *, int32_t, double, const double *, int32_t, int64_t, int32_t, float *,
                           int32_t *, void *) {
    return SP_EINVAL;
}
}
namespace sp {
int dedisp_configure(const sp_plan *) { return SP_OK; }
int sums_configure() { return SP_OK; }
int64_t dedisp_time_tiles(const sp_plan *p, int64_t n_out) { return (n_out + p->time_tile - 1) / p->time_tile; }
}  // namespace sp

// Every piece of 0 .. n - 1 once, no other, with n near the end of 32 bits.
static int blocks() {
    const int64_t n = INT32_MAX - 10;
    std::atomic<int64_t> pieces{0}, bad{0};
    sp::blocks_on_cores(n, 1 << 20, [&](int64_t first, int64_t end) {
        if (first < 0 || first >= end || end > n) {
            ++bad;
            return false;
        }
        pieces += end - first;
        return true;
    });
    std::printf("pieces %lld of %lld, bad %lld\n", (long long)pieces, (long long)n, (long long)bad);
    return bad || pieces != n;
}

static std::vector<double> band(int nchan) {
    std::vector<double> f((size_t)nchan);
    for (int c = 0; c < nchan; ++c) f[(size_t)c] = 500.0 - 200.0 * c / nchan;
    return f;
}

// Device memory runs out at each allocation of a plan in turn: at the shared-sum
// tables (the last) the plan goes without them, earlier it is refused.
static int no_room() {
    const std::vector<double> f = band(1024);
    std::vector<double> dms;
    for (int d = 0; d < 128; ++d) dms.push_back(0.1 * d);
    sp_plan *p = nullptr;
    auto create = [&]() { return sp_plan_create(f.data(), 1024, 1.31072e-3, dms.data(), 128, &p); };
    int bad = create() != SP_OK || !p->d_sums;
    const int64_t n = g_asked;
    sp_plan_destroy(p);
    for (int64_t i = 0; i < n; ++i) {
        g_asked = 0;
        g_refuse = i;
        const int rc = create();
        std::printf("allocation %lld of %lld refused: %d\n", (long long)i, (long long)n, rc);
        if (i < n - 1) {
            bad += rc != SP_ENOMEM || p;
            continue;
        }
        if (rc != SP_OK || p->d_sums) return 1;
        const int64_t n_out = 1 << 20;
        bad += sp::sums_pay(&p, &n_out, 1);
        sp_plan_destroy(p);
    }
    return bad || g_live;
}

// Two bands of 16 almost equal channels, the lower one up to 8e8 samples late: no
// group of it fits a slot until a tile is a few trials (apart: one trial).
static int late_band(bool apart) {
    std::vector<double> f, dms;
    for (int c = 0; c < 16; ++c) f.push_back(1000.0 - 1e-7 * c);
    for (int c = 0; c < 16; ++c) f.push_back(100.0 - 3e-7 * c);
    for (int d = 0; d < 64; ++d) dms.push_back(apart ? 2000.0 * (d & 1) : 2000.0 / 63 * d);
    int64_t report[8];
    const int rc = sp_plan_check_tables(f.data(), 32, 1e-6, dms.data(), 64, 0, 1000, report);
    const double seconds = (double)std::clock() / CLOCKS_PER_SEC;  // 5 s and more with a path for every pass, else 0.01
    std::printf("rc %d, violations %lld, largest delay %lld, %.2f s\n", rc, (long long)report[5], (long long)report[6],
                seconds);
    return rc || report[5] || report[6] < 800000000 || seconds > 2.0;
}

// Which kernel launches of a plan go to (1: shared sums), and their modelled clocks: channels, first
// trial, step, trials, then lengths.
static int clocks(int argc, char **argv) {
    const int nchan = std::atoi(argv[2]), ndm = std::atoi(argv[5]);
    const double first = std::atof(argv[3]), step = std::atof(argv[4]);
    const std::vector<double> f = band(nchan);
    std::vector<double> dms;
    for (int d = 0; d < ndm; ++d) dms.push_back(first + step * d);
    sp_plan *p = nullptr;
    if (sp_plan_create(f.data(), nchan, 1.31072e-3, dms.data(), ndm, &p)) return 1;
    for (int i = 6; i < argc; ++i) {
        const int64_t n_out = std::atoll(argv[i]);
        const sp::DedispClocks c = sp::dedisp_clocks(&p, &n_out, 1);
        std::printf("%lld %d %d %.0f %.0f\n", (long long)n_out, p->d_sums != nullptr, sp::sums_pay(&p, &n_out, 1),
                    c.sums, c.direct);
    }
    sp_plan_destroy(p);
    return 0;
}

int main(int argc, char **argv) {
    const std::string what = argc > 1 ? argv[1] : "";
    if (what == "blocks") return blocks();
    if (what == "no_room") return no_room();
    if (what == "late_band") return late_band(argc > 2);
    if (what == "clocks" && argc > 6) return clocks(argc, argv);
    return 2;
}
