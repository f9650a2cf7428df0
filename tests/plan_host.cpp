// Host checks of plan.cpp and plan_sums.cpp without a GPU: the driver links
// them with a CUDA runtime of its own (host memory; allocations of g_refuse_from bytes
// or more fail) and is built with the undefined-behaviour sanitizer.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>

#include "../paper_2606_27262_gb300/csrc/sp_internal.h"

static size_t g_refuse_from = SIZE_MAX;
static int64_t g_live = 0;  // allocations not freed

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) {
    if (n >= g_refuse_from) return cudaErrorMemoryAllocation;
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
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
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

int main(int argc, char **argv) {
    const std::string what = argc > 1 ? argv[1] : "";
    if (what == "blocks") return blocks();
    return 2;
}
