// Host side of the DES-LOC library: the C ABI of include/desloc.h, argument validation, the
// sync schedule (Algorithm 1's "t mod K = 0" tests), the multi-tensor chunk plan and the
// launcher that picks one kernel instantiation per step.  No torch types, no CPU compute path.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <limits>
#include <new>
#include <utility>
#include <vector>

#include "../../include/desloc_testing.h"
#include "desloc_hostcopy.cuh"
#include "desloc_inst.cuh"
#include "desloc_internal.cuh"
#include "desloc_norms.cuh"
#include "desloc_readout.cuh"

namespace desloc {

const void *lookup_step_kernel(int opt, bool post, bool bf16, int mt, int mask, bool diag) {
    // A local step (mask 0) has nothing to do with the other workers: it takes the one-replica
    // kernel, whose blocks move 2-3 % more bytes per second than tiles of all replicas.  It lives
    // in the pre-average units and is the same code for either ordering.
    const bool pre = !post || mask == 0;
    const int m = mask == 0 ? 1 : mt;
    if (m > MAX_MT) {
        if (post || diag || m > MAX_TILE_MT) return nullptr;
        if (opt == OPT_ADAM) return m < 13 ? lookup_adam_m9(bf16, m, mask) : lookup_adam_m13(bf16, m, mask);
        if (opt == OPT_ADOPT) return m < 13 ? lookup_adopt_m9(bf16, m, mask) : lookup_adopt_m13(bf16, m, mask);
        return m < 13 ? lookup_sgdm_m9(bf16, m, mask) : lookup_sgdm_m13(bf16, m, mask);
    }
    if (opt == OPT_ADAM) {
        if (diag) return pre ? lookup_adam_pre_diag(bf16, m, mask) : lookup_adam_post_diag(bf16, m, mask);
        return pre ? lookup_adam_pre(bf16, m, mask) : lookup_adam_post(bf16, m, mask);
    }
    if (opt == OPT_ADOPT) {
        if (diag) return pre ? lookup_adopt_pre_diag(bf16, m, mask) : lookup_adopt_post_diag(bf16, m, mask);
        return pre ? lookup_adopt_pre(bf16, m, mask) : lookup_adopt_post(bf16, m, mask);
    }
    if (opt == OPT_SGDM) {
        if (diag) return pre ? lookup_sgdm_pre_diag(bf16, m, mask) : lookup_sgdm_post_diag(bf16, m, mask);
        return pre ? lookup_sgdm_pre(bf16, m, mask) : lookup_sgdm_post(bf16, m, mask);
    }
    return nullptr;
}

}  // namespace desloc

using desloc::mask_at;
using desloc::validate_config;

namespace {

constexpr int kSlots = 8;  // staging slots for per-step gradient pointer tables
constexpr size_t kHostGroups = 8;  // most groups that desloc_step_host is pipelined in, and
constexpr int64_t kHostSplit = 1600000;   // the fewest parameters worth splitting again

struct Slot {
    void **host = nullptr;
    void **dev = nullptr;
    cudaEvent_t done = nullptr;
    bool in_flight = false;     // `done` has been recorded behind the first kernel that reads the table
};

// desloc_step_host: groups whose copies and kernels are pipelined
struct HostGroup {
    int64_t c0, c1;   // chunks [c0, c1)
    int32_t k0, k1;   // of tensors k0 .. k1,
    int64_t e0, e1;   // the first one from element e0 on, the last one up to element e1
    int64_t elems;    // in all
    int64_t r0, r1;   // the same in chunks of the reduction kernels, the first and the last one in parts
};

// Everything that depends on the worker count M (re-made by desloc_set_workers): the pointer
// tables, the tile plan (the tile length is a function of M) and the scratch sized by either.
struct WorkerRes {
    desloc::Chunk *d_chunks = nullptr;   // tiles of the step kernels
    int64_t nchunks = 0;
    desloc::ChunkSet set;                // all of them
    bool full_round = false;             // a plan for them asks how the gradients lie (full_round_of_three)
    long long *d_tstart = nullptr;       // [num_tensors + 1] first tile of every tensor, and a word for d_diag_parts
    std::vector<int64_t> heads;          // [num_tensors] elements of the short first chunk
    std::vector<HostGroup> groups;
    void **d_tables = nullptr;  // [3][nptr] x, u, v
    Slot slots[kSlots];
    void **h_slots = nullptr;   // the slots' tables, pinned, and
    void **d_slots = nullptr;   // on the device
    float *d_partial = nullptr;  // reductions: partial sums [2][M][reduce_row(nrchunks)]
    float *d_norms = nullptr;    // [2][M]: gradient norms, clip factors
    void **h_snap = nullptr;     // pinned pointer table for desloc_rel_change
    void **d_snap = nullptr;
    Slot host_slots[2];          // tables of addresses in host memory (desloc_step_host), staged on the copy stream
    // Diagnostics step: [3][M][row] sums of squares, of a chunk each or, in desloc_crowd_kernel, of a part of one.  How many a chunk
    // has is written by the step that leaves them (behind d_tstart): the host does not see when a captured step runs.
    float *d_diag = nullptr;
    int *d_diag_parts = nullptr;
    // Results the host waits for go to its memory straight from the kernels, without a copy: [3][M][num_tensors] per-tensor norms,
    // [3][M] totals; [M] relative changes; behind either a word that releases them.
    float *h_out = nullptr;      // mapped pinned memory, and
    float *d_out = nullptr;      // the same as the kernels address it
};

void free_worker_res(WorkerRes &r) {
    for (Slot &s : r.slots) {
        if (s.done) cudaEventDestroy(s.done);
        s = Slot();
    }
    for (Slot &s : r.host_slots)
        if (s.done) cudaEventDestroy(s.done);
    if (r.h_slots) cudaFreeHost(r.h_slots);
    if (r.d_slots) cudaFree(r.d_slots);
    if (r.d_chunks) cudaFree(r.d_chunks);
    if (r.d_tstart) cudaFree(r.d_tstart);
    if (r.d_tables) cudaFree(r.d_tables);
    if (r.d_partial) cudaFree(r.d_partial);
    if (r.d_norms) cudaFree(r.d_norms);
    if (r.h_snap) cudaFreeHost(r.h_snap);
    if (r.d_snap) cudaFree(r.d_snap);
    if (r.d_diag) cudaFree(r.d_diag);
    if (r.h_out) cudaFreeHost(r.h_out);
    r = WorkerRes();
}

// Groups of desloc_step_host(): three quarters of what is left, each time.  A group's kernel takes a ninth of
// its copies' time, so it hides behind the next group's even at a quarter of the size, and the last group,
// whose kernel nothing hides, is small.  A copy costs 6 us beside its bytes, one per worker and group at
// best: below 1.6 M parameters that is more than the kernel.  A group ends with a tensor where that
// makes it no longer than seven eighths of what is left, else inside one, at the end of a chunk: a list whose
// last tensor is large would otherwise be one group, with nothing hidden.  (25 M parameters x 4 workers in 29
// tensors: 3817 us with eight equal groups of whole tensors, 3774 us with three; the copies alone 3690.)
void plan_host_groups(std::vector<HostGroup> &groups, const std::vector<desloc::Chunk> &chunks, const int64_t *numel,
                      int64_t total) {
    groups.clear();
    int64_t left = total, acc = 0;
    HostGroup g{};
    int64_t rstart = 0;   // first reduction chunk of the tensor
    for (size_t c = 0; c < chunks.size(); ++c) {
        const desloc::Chunk &ch = chunks[c];
        if (c > 0 && ch.tensor != chunks[c - 1].tensor) rstart += desloc::chunks_of(numel[chunks[c - 1].tensor], desloc::REDUCE_CHUNK_ELEMS, 0);
        const int64_t end = ch.start + ch.count, rest = numel[ch.tensor] - end;
        acc += ch.count;
        const bool split = groups.size() + 1 < kHostGroups && (left > kHostSplit || (rest == 0 && groups.empty()));
        const bool enough = 4 * acc >= 3 * left && (rest == 0 || 8 * (acc + rest) > 7 * left);
        if (c + 1 < chunks.size() && !(split && enough)) continue;
        g.c1 = static_cast<int64_t>(c) + 1;
        g.k1 = ch.tensor;
        g.e1 = end;
        g.elems = acc;
        g.r1 = rstart + (end + desloc::REDUCE_CHUNK_ELEMS - 1) / desloc::REDUCE_CHUNK_ELEMS;
        groups.push_back(g);
        g.c0 = g.c1;
        g.r0 = rest > 0 ? rstart + end / desloc::REDUCE_CHUNK_ELEMS : g.r1;
        g.k0 = rest > 0 ? ch.tensor : ch.tensor + 1;
        g.e0 = rest > 0 ? end : 0;
        left -= acc;
        acc = 0;
    }
}

// Allocates and fills the M-dependent resources; the device must be current.  May throw
// std::bad_alloc (host vectors).
cudaError_t make_worker_res(WorkerRes &r, const desloc_config &cfg, int M, const int64_t *numel, int num_tensors, int64_t total,
                            int64_t nrchunks, bool has_v, float *const *x, float *const *u,
                            float *const *v) {
    // tile plan for this worker count
    const int64_t chunk_elems = desloc::chunk_elems_for(cfg, M);
    std::vector<int64_t> heads(static_cast<size_t>(num_tensors));
    for (int32_t k = 0; k < num_tensors; ++k) heads[k] = desloc::head_elems(x[k], numel[k]);
    r.set = desloc::chunk_set(numel, num_tensors, chunk_elems, heads.data());
    const int64_t nchunks = r.set.n;
    std::vector<desloc::Chunk> chunks(static_cast<size_t>(nchunks));
    desloc::fill_chunks(numel, num_tensors, chunk_elems, chunks.data(), heads.data());
    std::vector<long long> tstart(static_cast<size_t>(num_tensors) + 2, 0);   // (the last one: *d_diag_parts, 0 before any step)
    for (int32_t k = 0; k < num_tensors; ++k)
        tstart[k + 1] = tstart[k] + desloc::chunks_of(numel[k], chunk_elems, heads[k]);
    plan_host_groups(r.groups, chunks, numel, total);
    r.nchunks = nchunks;
    r.heads.swap(heads);
    cudaError_t e0 = cudaMalloc(&r.d_chunks, chunks.size() * sizeof(desloc::Chunk));
    if (e0 == cudaSuccess)
        e0 = cudaMemcpy(r.d_chunks, chunks.data(), chunks.size() * sizeof(desloc::Chunk), cudaMemcpyHostToDevice);
    if (e0 == cudaSuccess) e0 = cudaMalloc(&r.d_tstart, tstart.size() * sizeof(long long));
    if (e0 == cudaSuccess)
        e0 = cudaMemcpy(r.d_tstart, tstart.data(), tstart.size() * sizeof(long long), cudaMemcpyHostToDevice);
    if (e0 != cudaSuccess) return e0;
    r.d_diag_parts = reinterpret_cast<int *>(r.d_tstart + num_tensors + 1);

    const int64_t nptr = static_cast<int64_t>(M) * num_tensors;
    std::vector<void *> tables(static_cast<size_t>(3 * nptr), nullptr);
    for (int64_t i = 0; i < nptr; ++i) {
        tables[i] = x[i];
        tables[nptr + i] = u[i];
        tables[2 * nptr + i] = has_v ? static_cast<void *>(v[i]) : nullptr;
    }
    cudaError_t e = cudaMalloc(&r.d_tables, tables.size() * sizeof(void *));
    if (e == cudaSuccess)
        e = cudaMemcpy(r.d_tables, tables.data(), tables.size() * sizeof(void *), cudaMemcpyHostToDevice);
    const size_t npart = static_cast<size_t>(2) * M * static_cast<size_t>(desloc::reduce_row(nrchunks));
    if (e == cudaSuccess) e = cudaMalloc(&r.d_partial, npart * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&r.d_norms, static_cast<size_t>(2) * M * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(r.d_norms, 0, static_cast<size_t>(2) * M * sizeof(float));
    if (e == cudaSuccess) e = cudaMallocHost(&r.h_snap, static_cast<size_t>(nptr) * sizeof(void *));
    if (e == cudaSuccess) e = cudaMalloc(&r.d_snap, static_cast<size_t>(nptr) * sizeof(void *));
    const size_t ndiag = static_cast<size_t>(desloc::DIAG_KINDS) * M;
    // (a partial sum per chunk, or per block of a chunk where averaging steps run in desloc_crowd_kernel)
    desloc_config as = cfg;
    as.M = M;
    r.full_round = desloc::full_round_of_three(as, r.set);
    const desloc::LaunchPlan crowd = desloc::plan_launch(as, DESLOC_SYNC_X, r.set, true, false, desloc::GradLayout::FIT);
    const int64_t row = crowd.kernel == desloc::Kernel::CROWD ? nchunks * crowd.parts : nchunks;
    if (e == cudaSuccess) e = cudaMalloc(&r.d_diag, ndiag * static_cast<size_t>(row) * sizeof(float));
    if (e == cudaSuccess)
        e = cudaHostAlloc(reinterpret_cast<void **>(&r.h_out), (ndiag * (num_tensors + 1) + M + 2) * sizeof(float),
                          cudaHostAllocMapped);
    if (e == cudaSuccess) e = cudaHostGetDevicePointer(reinterpret_cast<void **>(&r.d_out), r.h_out, 0);
    const size_t room = static_cast<size_t>(nptr + 15) & ~size_t{15};   // tables on 128-byte boundaries
    constexpr int kAll = kSlots + 2;
    if (e == cudaSuccess) e = cudaMallocHost(&r.h_slots, kAll * room * sizeof(void *));
    if (e == cudaSuccess) e = cudaMalloc(&r.d_slots, kAll * room * sizeof(void *));
    for (int i = 0; i < kAll && e == cudaSuccess; ++i) {
        Slot &s = i < kSlots ? r.slots[i] : r.host_slots[i - kSlots];
        s.host = r.h_slots + i * room;
        s.dev = r.d_slots + i * room;
        e = cudaEventCreateWithFlags(&s.done, cudaEventDisableTiming);
    }
    return e;
}

}  // namespace

struct desloc_ctx {
    desloc_config cfg{};
    std::vector<int64_t> numel;
    int device = 0;
    int64_t total_elems = 0;
    int64_t nptr = 0;  // M * num_tensors
    desloc::Chunk *d_rchunks = nullptr;  // 4096-element chunks of the reduction kernels
    int64_t nrchunks = 0;
    int *h_err = nullptr;                // mapped pinned flag: a device-side wait ran out
    int *d_err = nullptr;                // the same flag as the kernels address it
    int wait_limit = desloc::DEFAULT_WAIT_LIMIT;
    WorkerRes res;
    int next_slot = 0;
    int cur_slot = -1;           // slot holding the table equal to last_grads
    int cur_host = -1;           // the same of addresses in host memory
    std::vector<const void *> last_host;
    std::vector<const void *> last_grads;
    desloc::GradLayout last_layout = desloc::GradLayout::FIT;   // of them
    cudaStream_t last_stream = nullptr;
    int64_t counters[4] = {0, 0, 0, 0};
    int64_t launches = 0;
    int64_t gathers = 0;         // groups of host gradients that a kernel has brought (not in `launches`)
    int last_cuda_error = 0;
    bool diag_valid = false;        // a diagnostics step has run since the workers last changed
    int64_t max_blocks = 0;         // test hook: cap on the grid (0 = one block per work item)
    int staging_mode = -1;          // test hook: -1 the library decides; tile kernels that 0 always stage, 1 never, 2 as decided
    std::vector<const void *> prepared;  // kernels whose shared-memory limit this context has raised
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t ev_entry = nullptr;
    cudaEvent_t ev_group[kHostGroups] = {};
};

namespace {

int cuda_fail(desloc_ctx *ctx, cudaError_t e) {
    if (ctx) ctx->last_cuda_error = static_cast<int>(e);
    (void)cudaGetLastError();  // clear the sticky per-thread error where it can be cleared
    return DESLOC_E_CUDA;
}

// A block of an earlier kernel of this context gave up waiting for its copies: what it should have
// updated or summed up is incomplete.
bool wait_ran_out(const desloc_ctx *ctx) { return *static_cast<volatile int *>(ctx->h_err) != 0; }

void free_ctx(desloc_ctx *ctx) {
    if (!ctx) return;
    free_worker_res(ctx->res);
    if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
    if (ctx->ev_entry) cudaEventDestroy(ctx->ev_entry);
    for (cudaEvent_t ev : ctx->ev_group)
        if (ev) cudaEventDestroy(ev);
    if (ctx->d_rchunks) cudaFree(ctx->d_rchunks);
    if (ctx->h_err) cudaFreeHost(ctx->h_err);
    delete ctx;
}

// Stage the gradient pointer table for this step on `stream`; returns the device table.
int stage_grads(desloc_ctx *ctx, const void *const *grads, cudaStream_t stream, void ***dev_out) {
    const size_t bytes = static_cast<size_t>(ctx->nptr) * sizeof(void *);
    if (ctx->cur_slot >= 0 && stream == ctx->last_stream &&
        std::memcmp(ctx->last_grads.data(), grads, bytes) == 0) {
        *dev_out = ctx->res.slots[ctx->cur_slot].dev;  // same pointers as last step: table is resident
        return DESLOC_OK;
    }
    Slot &s = ctx->res.slots[ctx->next_slot];
    if (s.in_flight) {
        // Re-use of a slot whose table was staged kSlots table changes ago: wait until its copy has
        // left the pinned buffer.  (Later kernels that read the same table need no event: every step of a
        // context updates the same state, so whatever stream this one is on comes behind them, and the copy
        // below with it.)
        cudaError_t e = cudaEventSynchronize(s.done);
        if (e != cudaSuccess) return cuda_fail(ctx, e);
        s.in_flight = false;
    }
    std::memcpy(s.host, grads, bytes);
    cudaError_t e = cudaMemcpyAsync(s.dev, s.host, bytes, cudaMemcpyHostToDevice, stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    std::memcpy(ctx->last_grads.data(), grads, bytes);
    ctx->last_layout = desloc::grad_layout(ctx->cfg, grads, ctx->res.heads.data(), ctx->res.full_round);
    ctx->cur_slot = ctx->next_slot;
    ctx->next_slot = (ctx->next_slot + 1) % kSlots;
    ctx->last_stream = stream;
    *dev_out = s.dev;
    return DESLOC_OK;
}

// The gradients of a small problem as contiguous pieces that a kernel can read where they are, in pinned host memory;
// false where there are too many bytes or pieces, or some of them in memory that only the copy engine reaches.
bool host_runs_of(const desloc_ctx *ctx, const void *const *host_grads, const void *const *grads, desloc::HostRuns &runs) {
    const desloc_config &c = ctx->cfg;
    const int64_t gsz = c.grad_dtype == DESLOC_BF16 ? 2 : 4;
    desloc::HostRange known;
    return ctx->total_elems <= desloc::HOST_KERNEL_BYTES / gsz / c.M &&
           desloc::gather_host_runs(host_grads, grads, ctx->nptr, c.numel, c.num_tensors, static_cast<size_t>(gsz), runs,
                                    [&](const void *p, size_t bytes) { return desloc::device_reads_host(p, bytes, known); });
}

// The pieces of a group, contiguous on both sides, in order: piece(from, to, bytes) until it says no.
template <typename Piece>
bool for_pieces(const desloc_ctx *ctx, const HostGroup &grp, const void *const *host_grads, const void *const *grads, const Piece &piece) {
    const desloc_config &c = ctx->cfg;
    const size_t gsz = c.grad_dtype == DESLOC_BF16 ? 2 : 4;
    const auto upto = [&](int32_t k) { return static_cast<size_t>(k == grp.k1 ? grp.e1 : ctx->numel[k]) * gsz; };
    for (int m = 0; m < c.M; ++m) {
        for (int32_t k = grp.k0; k <= grp.k1;) {
            const int64_t i0 = static_cast<int64_t>(m) * c.num_tensors;
            const size_t from = k == grp.k0 ? static_cast<size_t>(grp.e0) * gsz : 0;
            const char *hp = static_cast<const char *>(host_grads[i0 + k]) + from;
            char *dp = static_cast<char *>(const_cast<void *>(grads[i0 + k])) + from;
            size_t bytes = upto(k) - from;
            for (++k; k <= grp.k1 && static_cast<const char *>(host_grads[i0 + k]) == hp + bytes &&
                      static_cast<const char *>(grads[i0 + k]) == dp + bytes; ++k)
                bytes += upto(k);
            if (!piece(hp, dp, bytes)) return false;
        }
    }
    return true;
}

// Is a group brought by a kernel: many pieces, all of them in memory that the device reads?
bool group_by_kernel(const desloc_ctx *ctx, const HostGroup &grp, const void *const *host_grads, const void *const *grads,
                     desloc::HostRange &known) {
    const int64_t bytes = grp.elems * ctx->cfg.M * (ctx->cfg.grad_dtype == DESLOC_BF16 ? 2 : 4);
    int64_t pieces = 0;
    for_pieces(ctx, grp, host_grads, grads, [&](const char *, char *, size_t) { return ++pieces != 0; });
    return desloc::gather_pays(pieces, bytes) &&
           for_pieces(ctx, grp, host_grads, grads, [&](const char *hp, char *, size_t n) { return desloc::device_reads_host(hp, n, known); });
}

// The table of host addresses on the device, for kernels on the copy stream.
cudaError_t stage_host_table(desloc_ctx *ctx, const void *const *host_grads, const void *const **out) {
    const size_t bytes = static_cast<size_t>(ctx->nptr) * sizeof(void *);
    cudaError_t e = cudaSuccess;
    if (ctx->cur_host < 0 || std::memcmp(ctx->last_host.data(), host_grads, bytes) != 0) {
        const int next = ctx->cur_host == 0 ? 1 : 0;
        Slot &s = ctx->res.host_slots[next];
        if (s.in_flight) e = cudaEventSynchronize(s.done);   // (the copy of two tables ago)
        if (e != cudaSuccess) return e;
        s.in_flight = false;
        ctx->cur_host = -1;
        std::memcpy(s.host, host_grads, bytes);
        e = cudaMemcpyAsync(s.dev, s.host, bytes, cudaMemcpyHostToDevice, ctx->copy_stream);
        if (e == cudaSuccess) e = cudaEventRecord(s.done, ctx->copy_stream);
        if (e != cudaSuccess) return e;
        s.in_flight = true;
        std::memcpy(ctx->last_host.data(), host_grads, bytes);
        ctx->cur_host = next;
    }
    *out = reinterpret_cast<const void *const *>(ctx->res.host_slots[ctx->cur_host].dev);
    return e;
}

// Raises the kernel's shared-memory limit, once per kernel and context (the attribute call costs a microsecond that a
// latency-bound step notices).
cudaError_t prepare_once(desloc_ctx *ctx, const desloc::LaunchPlan &plan) {
    if (std::find(ctx->prepared.begin(), ctx->prepared.end(), plan.fn) != ctx->prepared.end()) return cudaSuccess;
    const cudaError_t e = desloc::prepare_launch(plan);
    if (e == cudaSuccess && ctx->prepared.size() < ctx->prepared.capacity()) ctx->prepared.push_back(plan.fn);
    return e;
}

// max_norm > 0: norm-based clipping first (a reduction launch or two, see launch_grad_norms()), then the step.
// diag: the step kernel also leaves sums of squares of g, x_{t+1} and d_t, per chunk or part of one.
// host_grads != nullptr: the gradients are first brought from host memory into `grads` (device): by a kernel on `stream`
// where host_runs_of() allows it, else tensor group by tensor group on the context's copy stream, each group's
// kernel starting as soon as its copies have landed.
int run_step(desloc_ctx *ctx, uint32_t mask, float lr_t, float clip_bound_t,
             const void *const *grads, cudaStream_t stream, float max_norm = 0.f,
             const void *const *host_grads = nullptr, bool diag = false) {
    const desloc_config &c = ctx->cfg;
    if (std::isnan(max_norm)) return DESLOC_E_RANGE;
    int rc = desloc::validate_step(&c, lr_t, clip_bound_t);
    if (rc != DESLOC_OK) return rc;
    for (int64_t i = 0; i < ctx->nptr; ++i)
        if (!grads[i]) return DESLOC_E_NULL;
    if (wait_ran_out(ctx)) return DESLOC_E_DEVICE_WAIT;

    int dev_before = -1;
    cudaError_t e = cudaGetDevice(&dev_before);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    if (dev_before != ctx->device) {
        e = cudaSetDevice(ctx->device);
        if (e != cudaSuccess) return cuda_fail(ctx, e);
    }
    do {
        // Under stream capture nothing may be staged through the pinned ring (a replay would
        // read whatever the ring holds by then) and no event of the ring may be recorded.
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        e = cudaStreamIsCapturing(stream, &cap);
        if (e != cudaSuccess) {
            rc = cuda_fail(ctx, e);
            break;
        }
        const bool capturing = cap != cudaStreamCaptureStatusNone;
        if (capturing && host_grads) {
            rc = DESLOC_E_INVALID;
            break;
        }
        void **d_g = nullptr;
        bool inline_g = false;
        if (!capturing) {
            rc = stage_grads(ctx, grads, stream, &d_g);
            if (rc != DESLOC_OK) break;
        } else if (ctx->nptr <= desloc::INLINE_PTRS && max_norm <= 0.f) {
            inline_g = true;  // pointers travel in the kernel parameters: nothing to keep alive
        } else if (ctx->cur_slot >= 0 && stream == ctx->last_stream &&
                   std::memcmp(ctx->last_grads.data(), grads,
                               static_cast<size_t>(ctx->nptr) * sizeof(void *)) == 0) {
            d_g = ctx->res.slots[ctx->cur_slot].dev;  // table already resident in this slot
        } else {
            rc = DESLOC_E_INVALID;  // stage these pointers with one un-captured step first
            break;
        }
        const float *d_gscale = nullptr;
        if (max_norm > 0.f) {
            int n = 0;
            e = desloc::launch_grad_norms(ctx->d_rchunks, ctx->nrchunks, ctx->total_elems,
                                          reinterpret_cast<const void *const *>(d_g), c.num_tensors,
                                          c.M, c.grad_dtype == DESLOC_BF16, max_norm,
                                          ctx->res.d_partial, ctx->res.d_norms, ctx->res.d_norms + c.M,
                                          ctx->d_err, ctx->wait_limit, stream, &n);
            if (e != cudaSuccess) {
                rc = cuda_fail(ctx, e);
                break;
            }
            ctx->launches += n;
            d_gscale = ctx->res.d_norms + c.M;
        }

        const desloc::GradLayout layout =
            inline_g ? desloc::grad_layout(c, grads, ctx->res.heads.data(), ctx->res.full_round) : ctx->last_layout;
        const bool lanes_ok = ctx->staging_mode < 0 && ctx->max_blocks == 0;
        const desloc::LaunchPlan plan = desloc::plan_launch(c, mask, ctx->res.set, diag, max_norm > 0.f, layout, lanes_ok);
        if (!plan.fn) {
            rc = DESLOC_E_INVALID;
            break;
        }
        desloc::StepArgs a{};
        a.chunks = ctx->res.d_chunks;
        a.nchunks = ctx->res.nchunks;
        a.x = reinterpret_cast<float *const *>(ctx->res.d_tables);
        a.u = reinterpret_cast<float *const *>(ctx->res.d_tables + ctx->nptr);
        a.v = reinterpret_cast<float *const *>(ctx->res.d_tables + 2 * ctx->nptr);
        a.g = reinterpret_cast<const void *const *>(d_g);
        if (inline_g)
            for (int64_t i = 0; i < ctx->nptr; ++i) a.g_inline[i] = grads[i];
        a.gscale = d_gscale;
        a.diag = diag ? ctx->res.d_diag : nullptr;
        a.diag_stride = ctx->res.nchunks * (plan.kernel == desloc::Kernel::CROWD ? plan.parts : 1);
        a.diag_parts = ctx->res.d_diag_parts;
        desloc::fill_hyper(a, c, lr_t, clip_bound_t);
        a.err = ctx->d_err;
        a.wait_limit = ctx->wait_limit;
        desloc::fill_plan(a, plan);
        const bool forced = ctx->staging_mode == 0 || ctx->staging_mode == 1;
        if (forced && !plan.whole) a.direct = ctx->staging_mode;

        void *params[] = {&a};
        const auto capped = [ctx](const desloc::LaunchPlan &lp) {
            const bool cap = lp.strides && ctx->max_blocks > 0 && lp.grid > ctx->max_blocks;
            return dim3(static_cast<unsigned>(cap ? ctx->max_blocks : lp.grid), lp.grid_y);
        };
        bool on_device = !host_grads;
        if (host_grads) {
            desloc::HostRuns runs;
            if (host_runs_of(ctx, host_grads, grads, runs)) {
                e = desloc::launch_host_copy(runs, stream);
                if (e == cudaSuccess) ctx->launches += 1;
                on_device = true;
            }
        }
        if (on_device) {
            if (e == cudaSuccess) e = prepare_once(ctx, plan);
            if (e == cudaSuccess)
                e = desloc::launch_kernel(plan.fn, capped(plan), dim3(plan.threads, plan.threads_y), plan.smem, stream, params, plan.overlap);
            if (e == cudaSuccess) ctx->launches += 1;
        } else {
            // A group of chunks may run in another kernel than the whole list would.  All are planned and prepared
            // before the first one is launched: a kernel that is refused leaves the state as it was.
            desloc::LaunchPlan plans[kHostGroups];
            for (size_t gi = 0; gi < ctx->res.groups.size() && e == cudaSuccess; ++gi) {
                const HostGroup &grp = ctx->res.groups[gi];
                desloc::ChunkSet set = ctx->res.set;
                set.n = grp.c1 - grp.c0;
                set.total = grp.elems;
                plans[gi] = desloc::plan_launch(c, mask, set, diag, false, layout, lanes_ok);
                e = plans[gi].fn ? prepare_once(ctx, plans[gi]) : cudaErrorInvalidDeviceFunction;
            }
            // The device gradient buffers may still be read by earlier work on `stream`.
            if (e == cudaSuccess) e = cudaEventRecord(ctx->ev_entry, stream);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(ctx->copy_stream, ctx->ev_entry, 0);
            desloc::HostRange known;
            for (size_t gi = 0; gi < ctx->res.groups.size() && e == cudaSuccess; ++gi) {
                const HostGroup &grp = ctx->res.groups[gi];
                if (group_by_kernel(ctx, grp, host_grads, grads, known)) {
                    desloc::HostGather hg{ctx->d_rchunks, grp.r0, grp.r1, nullptr, a.g, c.num_tensors, c.M, grp.k0, grp.k1, grp.e0, grp.e1,
                                          c.grad_dtype == DESLOC_BF16 ? 2 : 4};
                    e = stage_host_table(ctx, host_grads, &hg.src);
                    if (e == cudaSuccess) e = desloc::launch_host_gather(hg, ctx->copy_stream);   // (in the copies' place, and not counted either)
                    if (e == cudaSuccess) ctx->gathers += 1;
                } else {
                    for_pieces(ctx, grp, host_grads, grads, [&](const char *hp, char *dp, size_t bytes) {
                        e = cudaMemcpyAsync(dp, hp, bytes, cudaMemcpyHostToDevice, ctx->copy_stream);
                        return e == cudaSuccess;
                    });
                }
                if (e == cudaSuccess) e = cudaEventRecord(ctx->ev_group[gi], ctx->copy_stream);
                if (e == cudaSuccess) e = cudaStreamWaitEvent(stream, ctx->ev_group[gi], 0);
                if (e != cudaSuccess) break;
                a.chunks = ctx->res.d_chunks + grp.c0;
                a.nchunks = grp.c1 - grp.c0;
                const desloc::LaunchPlan &gp = plans[gi];
                desloc::fill_plan(a, gp);
                if (forced && !gp.whole) a.direct = ctx->staging_mode;
                // (no overlap: this kernel also depends on the other stream's copies)
                e = desloc::launch_kernel(gp.fn, capped(gp), dim3(gp.threads, gp.threads_y), gp.smem, stream, params, false);
                if (e == cudaSuccess) ctx->launches += 1;
            }
        }
        if (e != cudaSuccess) {
            rc = cuda_fail(ctx, e);
            break;
        }
        if (!capturing) {
            // An event behind the first kernel that reads a table; a loop with the same gradient buffers
            // needs no more (0.5 us of host time a step), see stage_grads().
            Slot &s = ctx->res.slots[ctx->cur_slot];
            if (!s.in_flight) {
                e = cudaEventRecord(s.done, stream);
                if (e != cudaSuccess) {
                    rc = cuda_fail(ctx, e);
                    break;
                }
                s.in_flight = true;
            }
        }
        if (diag) ctx->diag_valid = true;
        ctx->counters[0] += 1;
        ctx->counters[1] += (mask & DESLOC_SYNC_X) ? 1 : 0;
        ctx->counters[2] += (mask & DESLOC_SYNC_U) ? 1 : 0;
        ctx->counters[3] += (mask & DESLOC_SYNC_V) ? 1 : 0;
    } while (false);
    if (dev_before != ctx->device) cudaSetDevice(dev_before);
    return rc;
}

}  // namespace

extern "C" {

uint32_t desloc_sync_mask(const desloc_config *cfg, int64_t t) {
    if (!cfg || t < 0) return 0;
    return mask_at(cfg, t);
}

int64_t desloc_chunk_elems(const desloc_config *cfg) {
    if (!cfg || !cfg->numel) return DESLOC_E_NULL;
    if (cfg->M < 1 || cfg->M > DESLOC_MAX_M || cfg->num_tensors < 1) return DESLOC_E_RANGE;
    for (int32_t k = 0; k < cfg->num_tensors; ++k)
        if (cfg->numel[k] < 1) return DESLOC_E_RANGE;
    return desloc::chunk_elems_for(*cfg, cfg->M);
}

int64_t desloc_plan_chunks_at(const int64_t *numel, int32_t num_tensors, int64_t chunk_elems,
                              const void *const *x0, int64_t *out, int64_t cap) {
    if (!numel) return DESLOC_E_NULL;
    if (num_tensors < 1 || chunk_elems < 1 || cap < 0) return DESLOC_E_RANGE;
    if (cap > 0 && !out) return DESLOC_E_NULL;
    for (int32_t k = 0; k < num_tensors; ++k)
        if (numel[k] < 1) return DESLOC_E_RANGE;
    try {
        // the context's own planner, so that this is the table a context works from
        std::vector<int64_t> heads(static_cast<size_t>(num_tensors), 0);
        if (x0)
            for (int32_t k = 0; k < num_tensors; ++k) heads[k] = desloc::head_elems(x0[k], numel[k]);
        const int64_t n = desloc::count_chunks(numel, num_tensors, chunk_elems, heads.data());
        if (cap > 0) {
            std::vector<desloc::Chunk> chunks(static_cast<size_t>(n));
            desloc::fill_chunks(numel, num_tensors, chunk_elems, chunks.data(), heads.data());
            for (int64_t c = 0; c < n && c < cap; ++c) {
                out[3 * c + 0] = chunks[c].tensor;
                out[3 * c + 1] = chunks[c].start;
                out[3 * c + 2] = chunks[c].count;
            }
        }
        return n;
    } catch (const std::bad_alloc &) {
        return DESLOC_E_NOMEM;
    }
}

int64_t desloc_plan_chunks(const int64_t *numel, int32_t num_tensors, int64_t chunk_elems,
                           int64_t *out, int64_t cap) {
    return desloc_plan_chunks_at(numel, num_tensors, chunk_elems, nullptr, out, cap);
}

int desloc_create(desloc_ctx **out, const desloc_config *cfg, float *const *x, float *const *u,
                  float *const *v, int cuda_device) {
    if (!out) return DESLOC_E_NULL;
    *out = nullptr;
    int rc = validate_config(cfg);
    if (rc != DESLOC_OK) return rc;
    if (!cfg->numel || !x || !u) return DESLOC_E_NULL;
    if (cfg->opt != DESLOC_SGDM && !v) return DESLOC_E_NULL;
    if (cuda_device < 0) return DESLOC_E_RANGE;
    const int64_t nptr = static_cast<int64_t>(cfg->M) * cfg->num_tensors;
    int64_t total = 0;
    rc = desloc::validate_numel(cfg, &total);
    if (rc != DESLOC_OK) return rc;
    for (int64_t i = 0; i < nptr; ++i) {
        if (!x[i] || !u[i]) return DESLOC_E_NULL;
        if (cfg->opt != DESLOC_SGDM && !v[i]) return DESLOC_E_NULL;
    }
    // (the reduction kernels' chunks start with the tensors: cutting them at 2 KB boundaries like
    // the step kernels' made no measurable difference, and this way the norms do not depend on
    // where the buffers are)
    const int64_t nrchunks = desloc::count_chunks(cfg->numel, cfg->num_tensors, desloc::REDUCE_CHUNK_ELEMS);
    if (!desloc::grid_fits(*cfg, cfg->M)) return DESLOC_E_RANGE;

    desloc_ctx *ctx = new (std::nothrow) desloc_ctx();
    if (!ctx) return DESLOC_E_NOMEM;
    std::vector<desloc::Chunk> rchunks;
    try {
        ctx->numel.assign(cfg->numel, cfg->numel + cfg->num_tensors);
        ctx->last_grads.assign(static_cast<size_t>(nptr), nullptr);
        ctx->last_host.assign(static_cast<size_t>(nptr), nullptr);
        ctx->prepared.reserve(64);   // steps never allocate: beyond this the attribute is simply set again
        rchunks.resize(static_cast<size_t>(nrchunks));
        desloc::fill_chunks(cfg->numel, cfg->num_tensors, desloc::REDUCE_CHUNK_ELEMS, rchunks.data());
    } catch (const std::bad_alloc &) {
        delete ctx;
        return DESLOC_E_NOMEM;
    }
    ctx->cfg = *cfg;
    ctx->cfg.numel = ctx->numel.data();
    ctx->device = cuda_device;
    ctx->total_elems = total;
    ctx->nptr = nptr;
    ctx->nrchunks = nrchunks;

    int dev_before = -1;
    cudaError_t e = cudaGetDevice(&dev_before);
    if (e == cudaSuccess && dev_before != cuda_device) e = cudaSetDevice(cuda_device);
    if (e == cudaSuccess) e = cudaMalloc(&ctx->d_rchunks, rchunks.size() * sizeof(desloc::Chunk));
    if (e == cudaSuccess)
        e = cudaMemcpy(ctx->d_rchunks, rchunks.data(), rchunks.size() * sizeof(desloc::Chunk),
                       cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaHostAlloc(reinterpret_cast<void **>(&ctx->h_err), sizeof(int), cudaHostAllocMapped);
    if (e == cudaSuccess) {
        *ctx->h_err = 0;
        e = cudaHostGetDevicePointer(reinterpret_cast<void **>(&ctx->d_err), ctx->h_err, 0);
    }
    // (ahead of the step's blocks: a kernel on this stream holds few of them, and the bus waits for it)
    int least = 0, greatest = 0;
    if (e == cudaSuccess) e = cudaDeviceGetStreamPriorityRange(&least, &greatest);
    if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&ctx->copy_stream, cudaStreamNonBlocking, greatest);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->ev_entry, cudaEventDisableTiming);
    for (size_t i = 0; i < kHostGroups && e == cudaSuccess; ++i)
        e = cudaEventCreateWithFlags(&ctx->ev_group[i], cudaEventDisableTiming);
    if (e == cudaSuccess) {
        try {
            e = make_worker_res(ctx->res, ctx->cfg, cfg->M, ctx->numel.data(), cfg->num_tensors, total, nrchunks,
                                cfg->opt != DESLOC_SGDM, x, u, v);
        } catch (const std::bad_alloc &) {
            e = cudaErrorMemoryAllocation;
        }
    }
    if (dev_before >= 0 && dev_before != cuda_device) cudaSetDevice(dev_before);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        free_ctx(ctx);
        return e == cudaErrorMemoryAllocation ? DESLOC_E_NOMEM : DESLOC_E_CUDA;
    }
    *out = ctx;
    return DESLOC_OK;
}

int desloc_step(desloc_ctx *ctx, int64_t t, float lr_t, float clip_bound_t,
                const void *const *grads, void *stream, uint32_t *mask_out) {
    desloc::NvtxRange range("desloc_step");
    if (!ctx || !grads) return DESLOC_E_NULL;
    if (t < 0) return DESLOC_E_RANGE;
    const uint32_t mask = mask_at(&ctx->cfg, t);
    const int rc = run_step(ctx, mask, lr_t, clip_bound_t, grads, static_cast<cudaStream_t>(stream));
    if (rc == DESLOC_OK && mask_out) *mask_out = mask;
    return rc;
}

int desloc_step_diag(desloc_ctx *ctx, int64_t t, float lr_t, float clip_bound_t, float max_norm,
                     const void *const *grads, void *stream, uint32_t *mask_out) {
    desloc::NvtxRange range("desloc_step_diag");
    if (!ctx || !grads) return DESLOC_E_NULL;
    if (t < 0 || !(max_norm >= 0.f) || !std::isfinite(max_norm)) return DESLOC_E_RANGE;
    const uint32_t mask = mask_at(&ctx->cfg, t);
    const int rc = run_step(ctx, mask, lr_t, clip_bound_t, grads, static_cast<cudaStream_t>(stream),
                            max_norm, nullptr, true);
    if (rc == DESLOC_OK && mask_out) *mask_out = mask;
    return rc;
}

int desloc_get_diag_norms(desloc_ctx *ctx, float *per_tensor_out, float *total_out, void *stream) {
    if (!ctx) return DESLOC_E_NULL;
    if (!ctx->diag_valid) return DESLOC_E_INVALID;
    const desloc_config &c = ctx->cfg;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int dev_before = -1;
    cudaError_t e = cudaGetDevice(&dev_before);
    if (e == cudaSuccess && dev_before != ctx->device) e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    const size_t rows = static_cast<size_t>(desloc::DIAG_KINDS) * c.M;
    const size_t per = rows * c.num_tensors;
    float *const out = ctx->res.h_out;
    desloc::expect_results(out, per + rows + 1);
    e = desloc::launch_diag_norms(ctx->res.d_diag, ctx->res.nchunks, ctx->res.d_diag_parts, ctx->res.d_tstart, c.num_tensors, c.M,
                                  ctx->res.d_out, ctx->res.d_out + per, ctx->res.d_out + per + rows, st);
    if (e == cudaSuccess) ctx->launches += 1;
    if (e == cudaSuccess) e = desloc::wait_for_results(out, per + rows + 1, [st] { return cudaStreamSynchronize(st); });
    const bool valid = e == cudaSuccess && !wait_ran_out(ctx);
    if (valid) {
        if (per_tensor_out) std::memcpy(per_tensor_out, out, per * sizeof(float));
        if (total_out) std::memcpy(total_out, out + per, rows * sizeof(float));
    }
    if (dev_before != ctx->device) cudaSetDevice(dev_before);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    return valid ? DESLOC_OK : DESLOC_E_DEVICE_WAIT;
}

int desloc_step_host(desloc_ctx *ctx, int64_t t, float lr_t, float clip_bound_t,
                     const void *const *host_grads, void *const *dev_grads, void *stream,
                     uint32_t *mask_out) {
    desloc::NvtxRange range("desloc_step_host");
    if (!ctx || !host_grads || !dev_grads) return DESLOC_E_NULL;
    if (t < 0) return DESLOC_E_RANGE;
    for (int64_t i = 0; i < ctx->nptr; ++i)
        if (!host_grads[i]) return DESLOC_E_NULL;
    const uint32_t mask = mask_at(&ctx->cfg, t);
    const int rc = run_step(ctx, mask, lr_t, clip_bound_t,
                            reinterpret_cast<const void *const *>(dev_grads),
                            static_cast<cudaStream_t>(stream), 0.f, host_grads);
    if (rc == DESLOC_OK && mask_out) *mask_out = mask;
    return rc;
}

int desloc_step_masked(desloc_ctx *ctx, uint32_t mask, float lr_t, float clip_bound_t,
                       const void *const *grads, void *stream) {
    desloc::NvtxRange range("desloc_step_masked");
    if (!ctx || !grads) return DESLOC_E_NULL;
    if (mask & ~7u) return DESLOC_E_INVALID;
    if (ctx->cfg.opt == DESLOC_SGDM && (mask & DESLOC_SYNC_V)) return DESLOC_E_INVALID;
    return run_step(ctx, mask, lr_t, clip_bound_t, grads, static_cast<cudaStream_t>(stream));
}

int desloc_step_normclip(desloc_ctx *ctx, int64_t t, float lr_t, float clip_bound_t,
                         float max_norm, const void *const *grads, void *stream,
                         uint32_t *mask_out) {
    desloc::NvtxRange range("desloc_step_normclip");
    if (!ctx || !grads) return DESLOC_E_NULL;
    if (t < 0 || !(max_norm > 0.f) || !std::isfinite(max_norm)) return DESLOC_E_RANGE;
    const uint32_t mask = mask_at(&ctx->cfg, t);
    const int rc = run_step(ctx, mask, lr_t, clip_bound_t, grads, static_cast<cudaStream_t>(stream),
                            max_norm);
    if (rc == DESLOC_OK && mask_out) *mask_out = mask;
    return rc;
}

int desloc_get_grad_norms(desloc_ctx *ctx, float *norms_out, float *scales_out, void *stream) {
    if (!ctx) return DESLOC_E_NULL;
    const size_t bytes = static_cast<size_t>(ctx->cfg.M) * sizeof(float);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int dev_before = -1;
    cudaError_t e = cudaGetDevice(&dev_before);
    if (e == cudaSuccess && dev_before != ctx->device) e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    if (norms_out) e = cudaMemcpyAsync(norms_out, ctx->res.d_norms, bytes, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && scales_out)
        e = cudaMemcpyAsync(scales_out, ctx->res.d_norms + ctx->cfg.M, bytes, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (dev_before != ctx->device) cudaSetDevice(dev_before);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    return wait_ran_out(ctx) ? DESLOC_E_DEVICE_WAIT : DESLOC_OK;
}

int desloc_rel_change(desloc_ctx *ctx, int32_t array, const float *const *then, float *out,
                      void *stream) {
    if (!ctx || !then || !out) return DESLOC_E_NULL;
    if (array < 0 || array > 2 || (array == 2 && ctx->cfg.opt == DESLOC_SGDM)) return DESLOC_E_INVALID;
    for (int64_t i = 0; i < ctx->nptr; ++i)
        if (!then[i]) return DESLOC_E_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int dev_before = -1;
    cudaError_t e = cudaGetDevice(&dev_before);
    if (e == cudaSuccess && dev_before != ctx->device) e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    const size_t tbytes = static_cast<size_t>(ctx->nptr) * sizeof(void *);
    // The call ends when the kernels behind this copy have their results, so the pinned table is free again on return.
    std::memcpy(ctx->res.h_snap, then, tbytes);
    e = cudaMemcpyAsync(ctx->res.d_snap, ctx->res.h_snap, tbytes, cudaMemcpyHostToDevice, st);
    const size_t M = static_cast<size_t>(ctx->cfg.M), at = desloc::DIAG_KINDS * M * (ctx->cfg.num_tensors + 1) + 1;
    float *const change = ctx->res.h_out + at;
    desloc::expect_results(change, M + 1);
    if (e == cudaSuccess)
        e = desloc::launch_rel_change(
            ctx->d_rchunks, ctx->nrchunks,
            reinterpret_cast<const float *const *>(ctx->res.d_tables + array * ctx->nptr),
            reinterpret_cast<const float *const *>(ctx->res.d_snap), ctx->cfg.num_tensors, ctx->cfg.M,
            ctx->res.d_partial, ctx->res.d_out + at, ctx->res.d_out + at + M, ctx->d_err, ctx->wait_limit, st);
    if (e == cudaSuccess) ctx->launches += 2;
    if (e == cudaSuccess) e = desloc::wait_for_results(change, M + 1, [st] { return cudaStreamSynchronize(st); });
    const bool valid = e == cudaSuccess && !wait_ran_out(ctx);
    if (valid) std::memcpy(out, change, M * sizeof(float));
    if (dev_before != ctx->device) cudaSetDevice(dev_before);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    return valid ? DESLOC_OK : DESLOC_E_DEVICE_WAIT;
}

int desloc_set_workers(desloc_ctx *ctx, int32_t M_new, int32_t first_new, float *const *x,
                       float *const *u, float *const *v, void *stream) {
    if (!ctx || !x || !u) return DESLOC_E_NULL;
    const bool has_v = ctx->cfg.opt != DESLOC_SGDM;
    if (has_v && !v) return DESLOC_E_NULL;
    if (M_new < 1 || M_new > DESLOC_MAX_M || first_new < 0 || first_new > M_new) return DESLOC_E_RANGE;
    if (!desloc::grid_fits(ctx->cfg, M_new)) return DESLOC_E_RANGE;
    const int nt = ctx->cfg.num_tensors;
    const int64_t nptr_new = static_cast<int64_t>(M_new) * nt;
    for (int64_t i = 0; i < nptr_new; ++i) {
        if (!x[i] || !u[i] || (has_v && !v[i])) return DESLOC_E_NULL;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int dev_before = -1;
    cudaError_t e = cudaGetDevice(&dev_before);
    if (e == cudaSuccess && dev_before != ctx->device) e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    // Earlier steps must have finished with the old tables before they are replaced.
    e = cudaStreamSynchronize(st);
    WorkerRes fresh;
    if (e == cudaSuccess) {
        try {
            e = make_worker_res(fresh, ctx->cfg, M_new, ctx->numel.data(), nt, ctx->total_elems, ctx->nrchunks, has_v, x, u, v);
            for (auto *last : {&ctx->last_grads, &ctx->last_host})
                if (last->capacity() < static_cast<size_t>(nptr_new))
                    last->reserve(static_cast<size_t>(nptr_new));  // may throw; no state changed yet
        } catch (const std::bad_alloc &) {
            e = cudaErrorMemoryAllocation;
        }
    }
    const int n_new = M_new - first_new;
    if (e == cudaSuccess && n_new > 0) {
        // New replicas start from the mean of ALL replicas the context held so far.
        const int n_arr = has_v ? 3 : 2;
        for (int arr = 0; arr < n_arr && e == cudaSuccess; ++arr)
            e = desloc::launch_mean_fill(
                ctx->d_rchunks, ctx->nrchunks,
                reinterpret_cast<const float *const *>(ctx->res.d_tables + arr * ctx->nptr), ctx->cfg.M,
                reinterpret_cast<float *const *>(fresh.d_tables + arr * nptr_new +
                                                 static_cast<int64_t>(first_new) * nt),
                n_new, nt, st);
        if (e == cudaSuccess) ctx->launches += n_arr;
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    int rc = DESLOC_OK;
    if (e == cudaSuccess) {
        free_worker_res(ctx->res);
        ctx->res = std::move(fresh);
        ctx->last_grads.assign(static_cast<size_t>(nptr_new), nullptr);  // capacity reserved above
        ctx->last_host.assign(static_cast<size_t>(nptr_new), nullptr);
        ctx->cur_host = -1;
        ctx->cfg.M = M_new;
        ctx->nptr = nptr_new;
        ctx->next_slot = 0;
        ctx->cur_slot = -1;
        ctx->diag_valid = false;
    } else {
        free_worker_res(fresh);
        rc = (e == cudaErrorMemoryAllocation) ? DESLOC_E_NOMEM : cuda_fail(ctx, e);
        (void)cudaGetLastError();
    }
    if (dev_before != ctx->device) cudaSetDevice(dev_before);
    return rc;
}

int desloc_destroy(desloc_ctx *ctx) {
    if (!ctx) return DESLOC_OK;
    int dev_before = -1;
    if (cudaGetDevice(&dev_before) == cudaSuccess && dev_before != ctx->device)
        cudaSetDevice(ctx->device);
    const int device = ctx->device;
    free_ctx(ctx);
    if (dev_before >= 0 && dev_before != device) cudaSetDevice(dev_before);
    (void)cudaGetLastError();
    return DESLOC_OK;
}

int desloc_get_counters(const desloc_ctx *ctx, int64_t out[4]) {
    if (!ctx || !out) return DESLOC_E_NULL;
    for (int i = 0; i < 4; ++i) out[i] = ctx->counters[i];
    return DESLOC_OK;
}

int64_t desloc_get_launch_count(const desloc_ctx *ctx) { return ctx ? ctx->launches : 0; }

int desloc_testing_set_max_blocks(desloc_ctx *ctx, int64_t max_blocks) {
    if (!ctx) return DESLOC_E_NULL;
    if (max_blocks < 0) return DESLOC_E_RANGE;
    ctx->max_blocks = max_blocks;
    return DESLOC_OK;
}

int desloc_testing_set_staging(desloc_ctx *ctx, int32_t mode) {
    if (!ctx) return DESLOC_E_NULL;
    if (mode < -1 || mode > 2) return DESLOC_E_RANGE;
    ctx->staging_mode = mode;
    return DESLOC_OK;
}

int desloc_testing_set_wait_limit(desloc_ctx *ctx, int32_t polls) {
    if (!ctx) return DESLOC_E_NULL;
    ctx->wait_limit = polls < 0 ? desloc::DEFAULT_WAIT_LIMIT : polls;
    if (polls < 0) *static_cast<volatile int *>(ctx->h_err) = 0;
    return DESLOC_OK;
}

int32_t desloc_testing_kernel_of(const desloc_config *cfg, uint32_t mask, int64_t nchunks, int32_t layout, int32_t diag, int64_t *blocks) {
    if (!cfg || !cfg->numel) return DESLOC_E_NULL;
    if (validate_config(cfg) != DESLOC_OK || (mask & ~7u) || nchunks < 0 || layout < 0 || layout > 2) return DESLOC_E_INVALID;
    desloc::ChunkSet set = desloc::chunk_set(cfg->numel, cfg->num_tensors, desloc::chunk_elems_for(*cfg, cfg->M));
    if (nchunks > 0) set.n = nchunks;
    const desloc::LaunchPlan p = desloc::plan_launch(*cfg, mask, set, diag != 0, false, static_cast<desloc::GradLayout>(layout));
    if (blocks) *blocks = p.grid * p.grid_y;
    return p.fn ? static_cast<int32_t>(p.kernel) : DESLOC_E_INVALID;
}

int64_t desloc_testing_gathers(const desloc_ctx *ctx) { return ctx ? ctx->gathers : 0; }

int desloc_last_cuda_error(const desloc_ctx *ctx) { return ctx ? ctx->last_cuda_error : 0; }

const char *desloc_strerror(int status) {
    switch (status) {
        case DESLOC_OK: return "ok";
        case DESLOC_E_NULL: return "a required pointer is NULL";
        case DESLOC_E_RANGE: return "argument out of range";
        case DESLOC_E_INVALID: return "invalid optimizer, dtype, flag or mask";
        case DESLOC_E_NOMEM: return "out of memory";
        case DESLOC_E_CUDA: return "CUDA call failed";
        case DESLOC_E_TOO_LARGE: return "problem exceeds the fixed scratch of desloc_step_static";
        case DESLOC_E_DEVICE_WAIT: return "a bounded wait on the device ran out in an earlier step";
        default: return "unknown status";
    }
}

}  // extern "C"
