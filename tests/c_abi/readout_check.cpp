// wait_for_results(): the thread goes on when the last word is there, however early the values are, and sees what was stored in front of it.
#include <cstdio>
#include <thread>

#include "desloc_readout.cuh"

#define CHECK(cond) if (!(cond)) { std::printf("failed: %s (line %d)\n", #cond, __LINE__); return 1; }

static float words[5];
static int flag;   // a plain store in front of the last word's release

static void write_word(int i, float v) { *static_cast<volatile float *>(&words[i]) = v; }
static void sleep_ms(int ms) { std::this_thread::sleep_for(std::chrono::milliseconds(ms)); }

int main() {
    int asked = 0;
    const auto never = [&] { ++asked; return cudaErrorUnknown; };
    for (int late = 0; late < 50; ++late) {   // four values at once, what an earlier kernel has stored and the last word behind them
        desloc::expect_results(words, 5);
        flag = 0;
        std::thread device([&] {
            for (int i = 0; i < 4; ++i) write_word(i, 1.f + i);
            if (late % 10 == 0) sleep_ms(4);
            flag = 1;
            std::atomic_thread_fence(std::memory_order_release);
            write_word(4, 1.f);
        });
        const cudaError_t e = desloc::wait_for_results(words, 5, never);
        const int seen = flag;
        device.join();
        if (e == cudaSuccess) CHECK(seen == 1 && words[0] == 1.f && words[3] == 4.f && words[4] == 1.f);   // (a busy machine may pass the 20 ms)
    }
    asked = 0;
    {   // nothing comes: the driver is asked after a while, and its answer is the call's
        desloc::expect_results(words, 5);
        asked = 0;
        CHECK(desloc::wait_for_results(words, 5, never) == cudaErrorUnknown && asked == 1);
    }
    {   // late, but there when the driver says so
        desloc::expect_results(words, 5);
        CHECK(desloc::wait_for_results(words, 5, [&] {
            for (int i = 0; i < 5; ++i) write_word(i, 2.f);
            return cudaSuccess;
        }) == cudaSuccess && words[4] == 2.f);
    }
    std::printf("readout_check: ok\n");
    return 0;
}
