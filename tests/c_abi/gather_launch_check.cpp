// launch_host_gather() against a runtime of a few lines: it reports its own launch, whatever earlier calls of the thread left behind.
#include <cstdio>

#include "desloc_hostcopy.cuh"

static cudaError_t left_behind = cudaSuccess, launch_says = cudaSuccess;
static dim3 grid, threads;
static cudaStream_t stream;
static int launches = 0;

static cudaError_t launched(dim3 g, dim3 t, cudaStream_t s) {
    grid = g, threads = t, stream = s, ++launches;
    if (launch_says != cudaSuccess) left_behind = launch_says;
    return launch_says;
}

extern "C" {
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *lc, const void *, void **) { return launched(lc->gridDim, lc->blockDim, lc->stream); }
cudaError_t cudaLaunchKernel(const void *, dim3 g, dim3 t, void **, size_t, cudaStream_t s) { return launched(g, t, s); }
cudaError_t cudaGetLastError() {
    const cudaError_t e = left_behind;
    left_behind = cudaSuccess;
    return e;
}
cudaError_t cudaGetDriverEntryPoint(const char *, void **, unsigned long long, cudaDriverEntryPointQueryResult *) { return cudaErrorNotSupported; }
static struct { dim3 g, t; size_t smem; void *s; } pushed;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 t, size_t smem, void *s) {
    pushed.g = g, pushed.t = t, pushed.smem = smem, pushed.s = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *t, size_t *smem, void *s) {
    *g = pushed.g, *t = pushed.t, *smem = pushed.smem, *static_cast<void **>(s) = pushed.s;
    return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
}

#define CHECK(cond) if (!(cond)) { std::printf("failed: %s (line %d)\n", #cond, __LINE__); return 1; }

int main() {
    const cudaStream_t st = reinterpret_cast<cudaStream_t>(0x40);
    desloc::HostGather a{};
    a.first = 3, a.last = 5, a.M = 3;
    left_behind = cudaErrorNotReady;
    CHECK(desloc::launch_host_gather(a, st) == cudaSuccess);
    CHECK(launches == 1 && grid.x == 2 && grid.y == 1 && threads.x == 128 && stream == st);   // a warp for each of six chunks
    CHECK(cudaGetLastError() == cudaErrorNotReady);                                         // (still the caller's to find)
    a.last = 100000;
    CHECK(desloc::launch_host_gather(a, st) == cudaSuccess && launches == 2 && grid.x == 64);
    launch_says = cudaErrorInvalidConfiguration;
    CHECK(desloc::launch_host_gather(a, st) == cudaErrorInvalidConfiguration);
    std::printf("gather_launch_check: ok\n");
    return 0;
}
