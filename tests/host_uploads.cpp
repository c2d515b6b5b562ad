// Host side of the propagation calls against a CUDA runtime that copies as late
// as it may: a host-to-device copy takes its bytes when the stream is
// synchronised.  Prints how many copies find other bytes at their source by
// then than when they were asked for, and how many copies there were.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <fstream>
#include <iterator>
#include <vector>

#include "kete_adjoint.h"
#include "kete_order.h"

struct Copy {
    const void *src;
    std::vector<char> asked;
};
static std::vector<Copy> g_pending;
static long g_stale, g_copies;

static void settle()
{
    for (const Copy &c : g_pending) g_stale += std::memcmp(c.src, c.asked.data(), c.asked.size()) != 0;
    g_pending.clear();
}

extern "C" {
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind kind, cudaStream_t)
{
    std::memcpy(dst, src, n);
    if (kind == cudaMemcpyHostToDevice) {
        g_pending.push_back({src, {(const char *)src, (const char *)src + n}});
        g_copies++;
    }
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { settle(); return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { settle(); return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaFree(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { settle(); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return ""; }
}

namespace kete {
void upload_radau_tables(cudaStream_t) {}
cudaError_t upload_adjoint_tables(cudaStream_t) { return cudaSuccess; }
cudaError_t upload_warp_tables(cudaStream_t) { return cudaSuccess; }
bool warp_model(const EphemDev &, const ForceDev &, WarpModel &) { return true; }
size_t order_hist_elems(int64_t) { return 16; }
int order_launches(int64_t, const kete_nongrav *) { return 1; }
int64_t scan_tmp_elems(int64_t) { return 16; }
cudaError_t order_by_cost(const EphemDev &, const double *, int64_t, const double *, int64_t, double,
                          const double *, const kete_nongrav *, OrderScratch, int32_t *, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t launch_chain_init(ChainState, const double *, const double *, const ForceDev &, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t launch_chain_finish(ChainState, double *, double *, int32_t *, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t launch_grid_rows(const EphemDev &, const GridDev &, double *, float *, uint8_t *, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t launch_gather_bodies(const double *, const double *, int64_t, int64_t, double *, double *,
                                 cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t launch_propagate(const EphemDev &, const ForceDev &, ChainState, const double *,
                             const int32_t *, int, double *, int64_t, bool, DevCounters *, cudaStream_t,
                             const GridDev *, PropVariant, unsigned long long *, PropDefer *,
                             const int32_t *, const unsigned long long *, bool)
{
    return cudaSuccess;
}
cudaError_t launch_propagate_warp(const EphemDev &, const ForceDev &, const WarpModel &, ChainState,
                                  const double *, const int32_t *, int, double *, int64_t, bool,
                                  DevCounters *, cudaStream_t, PropQueue, bool)
{
    return cudaSuccess;
}
}  // namespace kete

int main(int, char **argv)
{
    std::ifstream f(argv[1], std::ios::binary);
    const std::vector<char> table((std::istreambuf_iterator<char>(f)), std::istreambuf_iterator<char>());
    const double t0 = std::atof(argv[2]);
    kete_ctx *ctx;
    if (kete_create(&ctx, 0, nullptr) || kete_load_ephem(ctx, table.data(), table.size())) return 1;
    const long stale0 = g_stale, copies0 = g_copies;
    const double stops[3] = {t0 + 3.0, t0 + 700.0, t0 + 701.0};
    int rc = 0;
    for (int64_t n : {12, 20000}) {
        std::vector<double> st(6 * n), ep(n, t0), out(18 * n);
        std::vector<int32_t> status(n);
        rc |= kete_propagate(ctx, st.data(), ep.data(), n, t0 + 900.0, nullptr, status.data());
        rc |= kete_propagate_legs(ctx, st.data(), ep.data(), n, t0 + 900.0, 1.0, nullptr, status.data());
        rc |= kete_propagate_stops(ctx, st.data(), ep.data(), n, stops, 3, nullptr, out.data(), status.data());
        rc |= kete_autotune(ctx, st.data(), ep.data(), n, stops, 3, nullptr, 1000, nullptr, nullptr,
                            nullptr, nullptr, nullptr);
    }
    settle();
    std::printf("%d %ld %ld\n", rc, g_stale - stale0, g_copies - copies0);
    return 0;
}
