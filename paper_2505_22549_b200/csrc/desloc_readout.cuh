// Results that the last kernel of a call writes straight to the host's memory, each word once.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <chrono>
#include <cstddef>
#include <cstdint>

namespace desloc {

constexpr uint32_t RESULT_UNWRITTEN = 0x7fb5eed5u;   // (a NaN that no conversion or root gives)

// Before the launch: n words are to come, the last of them stored with a release at system scope by a thread of the read-out kernel, behind its
// wait for the kernels in front (release_results()).
inline void expect_results(float *v, size_t n) {
    volatile uint32_t *p = reinterpret_cast<volatile uint32_t *>(v);
    for (size_t i = 0; i < n; ++i) p[i] = RESULT_UNWRITTEN;
}

// After it: the calling thread looks for the words, and asks the driver only when they keep it waiting (20 ms, or an error).  A launch and
// cudaStreamSynchronize() take 10.6 us until the thread goes on, a launch and the look 7.1.  What is in front in the stream is complete
// for the caller then, as it would be behind the synchronisation: the acquire here stands behind the last look.  The flag of a bounded wait that
// ran out is a plain store of a kernel in front: it is read after this and not before.
template <typename Synchronise>
cudaError_t wait_for_results(const float *v, size_t n, const Synchronise &synchronise) {
    const volatile uint32_t *p = reinterpret_cast<const volatile uint32_t *>(v);
    const auto until = std::chrono::steady_clock::now() + std::chrono::milliseconds(20);
    unsigned looks = 0;
    for (size_t i = 0; i < n; ++i) {
        while (p[i] == RESULT_UNWRITTEN)
            if ((++looks & 1023u) == 0 && std::chrono::steady_clock::now() > until) return synchronise();
    }
    std::atomic_thread_fence(std::memory_order_acquire);
    return cudaSuccess;
}

}  // namespace desloc
