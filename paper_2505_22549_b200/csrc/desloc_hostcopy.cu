// Gradients from pinned host memory to the device by kernels that read it: small problems in one launch, lists of many pieces group by group.
//
// Bound: PCIe.  A copy by the copy engine costs 4.3 us beside its bytes where others are behind it, 6 us by itself, one per worker and contiguous
// piece at best, and the step waits for it through two events on two streams.  Here one kernel in the step's own stream reads the host's
// memory directly, every byte requested at once, and the step kernel may begin behind it without a gap.
// Measured on B200, the whole call of step_host (before, copies): two workers x 4096 parameters, fp32, 17.1 us (24.9); eight x 20 K 19.2
// (50.2), x 100 K 69.2 (100.1); four x 189 K in 21 tensors, bf16, 36.0 (69.1), eight x 260 K 91.0 (123.5).  47 GB/s; large
// copies by the copy engine reach 49 to 55, so that beyond 4 MB, where the pieces are large, nothing is gained (one piece
// of 4 MB: 85.2 us against 86.8).
//
// Lists whose tensors do not follow one another on both sides: a copy by the engine costs 4.3 us beside its bytes at 55.1 GB/s (752 of 237 KB:
// 8.5 us each, 27.8 GB/s; on two to four streams the same), kernels read 51.0 GB/s, with 16 blocks as with 600, where the two sides lie alike
// within 16 bytes.  Else a lane brings less at a time: calls of 25 MB in pieces of 32 KB to 1 MB, SGDM step and all, 42 to 49 GB/s alike, 36 to 41
// off by 4 or 8 bytes, 35 to 38 off by 2; by copies 7 (32 KB), 17 (128 KB), 18 to 32 (512 KB, 1 MB).
#include "desloc_hostcopy.cuh"

#include <cuda.h>

#include "desloc_kernels.cuh"

namespace desloc {

namespace {

constexpr int COPY_THREADS = 128, COPY_UNITS = 4;
constexpr uint32_t HOST_SLICE = COPY_THREADS * COPY_UNITS * 16;
constexpr long long GATHER_BLOCKS = 64;   // sixteen keep the bus busy where the pieces are long; the step's blocks run beside them

// Units of U bytes from the first boundary on, what lies around them byte by byte, by THREADS threads.
template <typename U, int THREADS>
__device__ __forceinline__ void copy_slice(const char *src, char *dst, uint32_t begin, uint32_t end) {
    const uint32_t tid = threadIdx.x % THREADS;
    constexpr uint32_t S = sizeof(U);
    const uint32_t head = min(end, begin + static_cast<uint32_t>((0 - reinterpret_cast<uintptr_t>(src + begin)) & (S - 1)));
    const uint32_t body = (end - head) / S;
    const U *s = reinterpret_cast<const U *>(src + head);
    U *d = reinterpret_cast<U *>(dst + head);
    for (uint32_t i0 = tid; i0 < body; i0 += THREADS * COPY_UNITS) {
        U v[COPY_UNITS];
#pragma unroll
        for (int k = 0; k < COPY_UNITS; ++k)
            if (i0 + k * THREADS < body) v[k] = s[i0 + k * THREADS];
#pragma unroll
        for (int k = 0; k < COPY_UNITS; ++k)
            if (i0 + k * THREADS < body) d[i0 + k * THREADS] = v[k];
    }
    for (uint32_t i = begin + tid; i < head; i += THREADS) dst[i] = src[i];
    for (uint32_t i = head + body * S + tid; i < end; i += THREADS) dst[i] = src[i];
}

template <int THREADS>
__device__ __forceinline__ void copy_slice(const char *src, char *dst, uint32_t begin, uint32_t end) {
    const uintptr_t off = reinterpret_cast<uintptr_t>(src) ^ reinterpret_cast<uintptr_t>(dst);
    if ((off & 15u) == 0) copy_slice<uint4, THREADS>(src, dst, begin, end);
    else if ((off & 3u) == 0) copy_slice<uint32_t, THREADS>(src, dst, begin, end);
    else if ((off & 1u) == 0) copy_slice<uint16_t, THREADS>(src, dst, begin, end);
    else copy_slice<uint8_t, THREADS>(src, dst, begin, end);
}

__global__ void __launch_bounds__(COPY_THREADS) host_copy_kernel(const __grid_constant__ HostRuns r) {
    begin_and_let_next_begin();
    const char *src = r.src[blockIdx.y];
    char *dst = r.dst[blockIdx.y];
    const uint32_t begin = blockIdx.x * HOST_SLICE, end = min(r.bytes[blockIdx.y], begin + HOST_SLICE);
    if (begin >= end) return;
    // (the gradient buffers may still be read, and the host's memory written, by what is in front in the stream)
    wait_for_earlier_kernels();
    copy_slice<COPY_THREADS>(src, dst, begin, end);
}

// A warp per reduction chunk (4096 elements) and worker.
__global__ void __launch_bounds__(COPY_THREADS) host_gather_kernel(const __grid_constant__ HostGather a) {
    const long long n = a.last - a.first, stride = static_cast<long long>(gridDim.x) * (COPY_THREADS / 32);
    for (long long w = static_cast<long long>(blockIdx.x) * (COPY_THREADS / 32) + (threadIdx.x >> 5); w < n * a.M; w += stride) {
        const int m = static_cast<int>(w / n);
        const Chunk ch = a.chunks[a.first + (w - m * n)];
        long long from = ch.start, to = ch.start + ch.count;
        if (ch.tensor == a.k0 && from < a.e0) from = a.e0;
        if (ch.tensor == a.k1 && to > a.e1) to = a.e1;
        if (from >= to) continue;
        const long long idx = static_cast<long long>(m) * a.nt + ch.tensor;
        copy_slice<32>(static_cast<const char *>(a.src[idx]) + from * a.elem_bytes, static_cast<char *>(const_cast<void *>(a.dst[idx])) + from * a.elem_bytes,
                       0, static_cast<uint32_t>(to - from) * a.elem_bytes);
    }
}

using PointerGetAttributes = CUresult (*)(unsigned, CUpointer_attribute *, void **, CUdeviceptr);

PointerGetAttributes pointer_get_attributes() {
    static const PointerGetAttributes fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult found{};
        if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &p, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess) {
            (void)cudaGetLastError();
            p = nullptr;
        }
        return reinterpret_cast<PointerGetAttributes>(p);
    }();
    return fn;
}

}  // namespace

bool device_reads_host(const void *p, size_t bytes, HostRange &known) {
    const PointerGetAttributes get = pointer_get_attributes();
    if (!get) return false;
    // from allocation to allocation until the last byte
    for (uintptr_t at = reinterpret_cast<uintptr_t>(p), end = at + bytes; at < end;) {
        if (at >= known.begin && at < known.end) {
            at = known.end;
            continue;
        }
        unsigned type = 0;
        CUdeviceptr dev = 0, start = 0;
        size_t size = 0;
        CUpointer_attribute which[4] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                        CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
        void *values[4] = {&type, &dev, &start, &size};
        if (get(4, which, values, static_cast<CUdeviceptr>(at)) != CUDA_SUCCESS) return false;
        if (type != CU_MEMORYTYPE_HOST || dev != at || start > at || start + size <= at) return false;
        known = HostRange{at, static_cast<uintptr_t>(start + size)};
    }
    return true;
}

cudaError_t launch_host_copy(const HostRuns &runs, cudaStream_t stream) {
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3((runs.longest + HOST_SLICE - 1) / HOST_SLICE, static_cast<unsigned>(runs.n));
    lc.blockDim = dim3(COPY_THREADS);
    lc.stream = stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = &at;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, host_copy_kernel, runs);
}

cudaError_t launch_host_gather(const HostGather &a, cudaStream_t stream) {
    const long long warps = (a.last - a.first) * a.M, blocks = (warps + COPY_THREADS / 32 - 1) / (COPY_THREADS / 32);
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(static_cast<unsigned>(blocks < GATHER_BLOCKS ? blocks : GATHER_BLOCKS));
    lc.blockDim = dim3(COPY_THREADS);
    lc.stream = stream;
    return cudaLaunchKernelEx(&lc, host_gather_kernel, a);   // (its own error: an older one of the thread is not this launch's)
}

}  // namespace desloc
