// gather_host_runs(): which pieces are merged, how many are taken, and how often the driver is asked about them.
#include <cstdio>
#include <vector>

#include "desloc_hostcopy.cuh"

static char host_mem[1 << 16], dev_mem[1 << 16];

// n pieces of len bytes, gap bytes apart on the host; the first `yes` questions are answered yes.
static bool gather(int n, int len, int gap, int yes, desloc::HostRuns &runs, int &asked) {
    std::vector<const void *> h, d;
    std::vector<int64_t> numel(n, len);
    for (int i = 0; i < n; ++i) h.push_back(host_mem + i * (len + gap)), d.push_back(dev_mem + i * len);
    asked = 0;
    return desloc::gather_host_runs(h.data(), d.data(), n, numel.data(), n, 1, runs,
                                    [&](const void *, size_t) { return asked++ < yes; });
}

#define CHECK(cond) if (!(cond)) { std::printf("failed: %s (line %d)\n", #cond, __LINE__); return 1; }

int main() {
    int asked = 0;
    { desloc::HostRuns r; CHECK(gather(72, 33, 0, 99, r, asked) && r.n == 1 && r.bytes[0] == 72 * 33 && asked == 1); }
    { desloc::HostRuns r; CHECK(gather(64, 33, 1, 99, r, asked) && r.n == 64 && r.longest == 33 && asked == 64); }
    { desloc::HostRuns r; CHECK(!gather(65, 33, 1, 99, r, asked) && asked == 0); }
    { desloc::HostRuns r; CHECK(!gather(72, 33, 1, 99, r, asked) && asked == 0); }
    { desloc::HostRuns r; CHECK(!gather(8, 33, 1, 0, r, asked) && asked == 1); }
    { desloc::HostRuns r; CHECK(!gather(8, 33, 1, 5, r, asked) && asked == 6); }
    std::printf("host_runs_check: ok\n");
    return 0;
}
