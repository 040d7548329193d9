// Gradients of a small problem from pinned host memory to the device in one launch.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace desloc {

constexpr int HOST_RUNS = 64;                       // pieces that are contiguous on both sides, in a launch's parameters
constexpr int64_t HOST_KERNEL_BYTES = 4 << 20;      // most bytes that are worth it

struct HostRuns {
    const char *src[HOST_RUNS];
    char *dst[HOST_RUNS];
    uint32_t bytes[HOST_RUNS];
    int n = 0;
    uint32_t longest = 0;
    // false: full
    bool add(const char *from, char *to, size_t len) {
        if (n == HOST_RUNS || len > HOST_KERNEL_BYTES) return false;
        src[n] = from;
        dst[n] = to;
        bytes[n++] = static_cast<uint32_t>(len);
        if (len > longest) longest = static_cast<uint32_t>(len);
        return true;
    }
};

// Can a kernel read all of these bytes at the addresses the host uses?  (Every byte page-locked host memory that is mapped there.)
bool device_reads_host(const void *p, size_t bytes);

// One thread block per HOST_SLICE bytes of a run.
cudaError_t launch_host_copy(const HostRuns &runs, cudaStream_t stream);

}  // namespace desloc
