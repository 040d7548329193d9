// Gradients of a small problem from pinned host memory to the device in one launch.
//
// Bound: PCIe.  A copy by the copy engine costs 6 us beside its bytes, one per worker and contiguous piece at best, and the
// step waits for it through two events on two streams.  Here one kernel in the step's own stream reads the host's
// memory directly, every byte requested at once, and the step kernel may begin behind it without a gap.
// Measured on B200, the whole call of step_host (before, copies): two workers x 4096 parameters, fp32, 17.1 us (24.9); eight x 20 K 19.2
// (50.2), x 100 K 69.2 (100.1); four x 189 K in 21 tensors, bf16, 36.0 (69.1), eight x 260 K 91.0 (123.5).  47 GB/s; large
// copies by the copy engine reach 49 to 55, so that beyond 4 MB, where the pieces are large, nothing is gained (one piece
// of 4 MB: 85.2 us against 86.8).
#include "desloc_hostcopy.cuh"

#include <cuda.h>

#include "desloc_kernels.cuh"

namespace desloc {

namespace {

constexpr int COPY_THREADS = 128, COPY_UNITS = 4;
constexpr uint32_t HOST_SLICE = COPY_THREADS * COPY_UNITS * 16;

// Units of U bytes from the first boundary on, what lies around them byte by byte.
template <typename U>
__device__ __forceinline__ void copy_slice(const char *src, char *dst, uint32_t begin, uint32_t end) {
    constexpr uint32_t S = sizeof(U);
    const uint32_t head = min(end, begin + static_cast<uint32_t>((0 - reinterpret_cast<uintptr_t>(src + begin)) & (S - 1)));
    const uint32_t body = (end - head) / S;
    const U *s = reinterpret_cast<const U *>(src + head);
    U *d = reinterpret_cast<U *>(dst + head);
    for (uint32_t i0 = threadIdx.x; i0 < body; i0 += COPY_THREADS * COPY_UNITS) {
        U v[COPY_UNITS];
#pragma unroll
        for (int k = 0; k < COPY_UNITS; ++k)
            if (i0 + k * COPY_THREADS < body) v[k] = s[i0 + k * COPY_THREADS];
#pragma unroll
        for (int k = 0; k < COPY_UNITS; ++k)
            if (i0 + k * COPY_THREADS < body) d[i0 + k * COPY_THREADS] = v[k];
    }
    for (uint32_t i = begin + threadIdx.x; i < head; i += COPY_THREADS) dst[i] = src[i];
    for (uint32_t i = head + body * S + threadIdx.x; i < end; i += COPY_THREADS) dst[i] = src[i];
}

__global__ void __launch_bounds__(COPY_THREADS) host_copy_kernel(const __grid_constant__ HostRuns r) {
    begin_and_let_next_begin();
    const char *src = r.src[blockIdx.y];
    char *dst = r.dst[blockIdx.y];
    const uint32_t begin = blockIdx.x * HOST_SLICE, end = min(r.bytes[blockIdx.y], begin + HOST_SLICE);
    if (begin >= end) return;
    // (the gradient buffers may still be read, and the host's memory written, by what is in front in the stream)
    wait_for_earlier_kernels();
    const uintptr_t off = reinterpret_cast<uintptr_t>(src) ^ reinterpret_cast<uintptr_t>(dst);
    if ((off & 15u) == 0) copy_slice<uint4>(src, dst, begin, end);
    else if ((off & 3u) == 0) copy_slice<uint32_t>(src, dst, begin, end);
    else if ((off & 1u) == 0) copy_slice<uint16_t>(src, dst, begin, end);
    else copy_slice<uint8_t>(src, dst, begin, end);
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

bool device_reads_host(const void *p, size_t bytes) {
    const PointerGetAttributes get = pointer_get_attributes();
    if (!get) return false;
    // from allocation to allocation until the last byte
    for (uintptr_t at = reinterpret_cast<uintptr_t>(p), end = at + bytes; at < end;) {
        unsigned type = 0;
        CUdeviceptr dev = 0, start = 0;
        size_t size = 0;
        CUpointer_attribute which[4] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                        CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
        void *values[4] = {&type, &dev, &start, &size};
        if (get(4, which, values, static_cast<CUdeviceptr>(at)) != CUDA_SUCCESS) return false;
        if (type != CU_MEMORYTYPE_HOST || dev != at || start > at || start + size <= at) return false;
        at = start + size;
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

}  // namespace desloc
