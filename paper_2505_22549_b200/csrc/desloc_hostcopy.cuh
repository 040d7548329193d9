// Gradients from pinned host memory to the device by kernels that read it there.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace desloc {

struct Chunk;

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

// host[i], dev[i]: n pieces of numel[i mod nt] elements, merged where they follow one another on both sides.  readable(from, bytes)
// is asked once per run, and only when all of them have found room: asked as they came, a list of 72 pieces put 64 questions
// to the driver at every step before it went by copies all the same (time of the calling thread alone: the copies' 290 us hide it).
template <typename Readable>
bool gather_host_runs(const void *const *host, const void *const *dev, int64_t n, const int64_t *numel, int32_t nt, size_t elem_bytes,
                      HostRuns &runs, const Readable &readable) {
    const char *from = nullptr;
    char *to = nullptr;
    size_t bytes = 0;
    for (int64_t i = 0; i < n; ++i) {
        const char *hp = static_cast<const char *>(host[i]);
        char *dp = static_cast<char *>(const_cast<void *>(dev[i]));
        const size_t len = static_cast<size_t>(numel[i % nt]) * elem_bytes;
        if (bytes != 0 && hp == from + bytes && dp == to + bytes) {
            bytes += len;
            continue;
        }
        if (bytes != 0 && !runs.add(from, to, bytes)) return false;
        from = hp;
        to = dp;
        bytes = len;
    }
    if (bytes != 0 && !runs.add(from, to, bytes)) return false;
    for (int i = 0; i < runs.n; ++i)
        if (!readable(runs.src[i], runs.bytes[i])) return false;
    return true;
}

// Can a kernel read all of these bytes at the addresses the host uses?  (Every byte page-locked host memory that is mapped there.)
// known: what the driver has said yes to last, for the next question of the same call.
struct HostRange {
    uintptr_t begin = 0, end = 0;
};
bool device_reads_host(const void *p, size_t bytes, HostRange &known);

// One thread block per HOST_SLICE bytes of a run.
cudaError_t launch_host_copy(const HostRuns &runs, cudaStream_t stream);

// Reduction chunks [first, last) of every worker, from element e0 of tensor k0 to element e1 of tensor k1.
struct HostGather {
    const Chunk *chunks;
    long long first, last;
    const void *const *src;   // tables on the device, [M * nt]: addresses of host memory,
    const void *const *dst;   // and of the device's
    int nt, M, k0, k1;
    long long e0, e1;
    int elem_bytes;
};
cudaError_t launch_host_gather(const HostGather &a, cudaStream_t stream);

// Pieces that a kernel brings sooner than copies do: 4.3 us for each of them against the 7 % by which the copy engine is faster on long ones, and
// 20 us for the launch, the table of addresses and the questions to the driver.  Measured, the whole call (before, copies): two workers x 22 M
// parameters, bf16, 92 tensors 1775 us (2487); two x 6.5 M in 47 550 (965); three x 593 K, fp32, in 56 161 (928); eight x 37 K in 38 32 (1217).
// One rate for pieces that lie alike on both sides and for others: off by 2, 4 or 8 bytes the kernel took 0.16 to 0.19 of the copies' time in pieces of 32
// KB, 0.32 to 0.51 of 128 KB, 0.47 to 0.88 of 512 KB and 0.54 to 0.87 of 1 MB.
inline bool gather_pays(int64_t pieces, int64_t bytes) { return 4300 * pieces > bytes / 685 + 20000; }

}  // namespace desloc
