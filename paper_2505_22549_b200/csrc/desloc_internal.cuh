// Host-side pieces shared by the context path (desloc_host.cu) and the allocation-free entry
// point (desloc_static.cu): argument validation, the sync schedule, the chunk-size rule and the
// kernel-argument block, so that both paths validate, plan and launch identically.
#pragma once
#include <cmath>
#include <cstdint>
#include <limits>

#include <nvtx3/nvToolsExt.h>

#include "../../include/desloc.h"
#include "desloc_crowd.cuh"

namespace desloc {

// Polls a block gives its tile's copies before it gives up (each poll itself waits a while in
// hardware): far beyond any healthy latency, still finite.
constexpr int DEFAULT_WAIT_LIMIT = 1 << 22;

// A named range around every step call, visible to tools that record NVTX (no cost otherwise).
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

inline bool finite_in(float v, float lo, bool lo_incl, float hi, bool hi_incl) {
    if (!std::isfinite(v)) return false;
    if (lo_incl ? v < lo : v <= lo) return false;
    if (hi_incl ? v > hi : v >= hi) return false;
    return true;
}

// Everything about a desloc_config that can be checked without looking at numel or the device.
inline int validate_config(const desloc_config *c) {
    if (!c) return DESLOC_E_NULL;
    if (c->opt != DESLOC_ADAM && c->opt != DESLOC_ADOPT && c->opt != DESLOC_SGDM) return DESLOC_E_INVALID;
    if (c->grad_dtype != DESLOC_F32 && c->grad_dtype != DESLOC_BF16) return DESLOC_E_INVALID;
    if (c->flags & ~(DESLOC_FLAG_ADOPT_NORM_CLIP | DESLOC_FLAG_POST_AVERAGE)) return DESLOC_E_INVALID;
    if ((c->flags & DESLOC_FLAG_ADOPT_NORM_CLIP) && c->opt != DESLOC_ADOPT) return DESLOC_E_INVALID;
    if (c->M < 1 || c->M > DESLOC_MAX_M) return DESLOC_E_RANGE;
    if (c->num_tensors < 1) return DESLOC_E_RANGE;
    if (c->Kx < 0 || c->Ku < 0 || c->Kv < 0) return DESLOC_E_RANGE;
    if (!finite_in(c->beta1, 0.f, true, 1.f, false)) return DESLOC_E_RANGE;
    if (c->opt != DESLOC_SGDM && !finite_in(c->beta2, 0.f, true, 1.f, false)) return DESLOC_E_RANGE;
    if (!finite_in(c->eps, 0.f, true, std::numeric_limits<float>::max(), true)) return DESLOC_E_RANGE;
    if (!finite_in(c->weight_decay, 0.f, true, std::numeric_limits<float>::max(), true)) return DESLOC_E_RANGE;
    if (std::isnan(c->clip_rho)) return DESLOC_E_RANGE;
    return DESLOC_OK;
}

// numel[k] >= 1 for every tensor and a total that cannot overflow the byte arithmetic.
inline int validate_numel(const desloc_config *c, int64_t *total_out) {
    if (!c->numel) return DESLOC_E_NULL;
    int64_t total = 0;
    for (int32_t k = 0; k < c->num_tensors; ++k) {
        if (c->numel[k] < 1) return DESLOC_E_RANGE;
        if (c->numel[k] > (INT64_MAX >> 4) - total) return DESLOC_E_RANGE;
        total += c->numel[k];
    }
    if (total_out) *total_out = total;
    return DESLOC_OK;
}

// Per-step scalar arguments.
inline int validate_step(const desloc_config *c, float lr_t, float clip_bound_t) {
    if (!std::isfinite(lr_t)) return DESLOC_E_RANGE;
    if ((c->flags & DESLOC_FLAG_ADOPT_NORM_CLIP) && !(clip_bound_t >= 0.f)) return DESLOC_E_RANGE;
    return DESLOC_OK;
}

// Algorithm 1's three "t mod K = 0" tests, t from 0; K = 0 never syncs; SGDM has no second state.
inline uint32_t mask_at(const desloc_config *c, int64_t t) {
    uint32_t m = 0;
    if (c->Kx > 0 && t % c->Kx == 0) m |= DESLOC_SYNC_X;
    if (c->Ku > 0 && t % c->Ku == 0) m |= DESLOC_SYNC_U;
    if (c->opt != DESLOC_SGDM && c->Kv > 0 && t % c->Kv == 0) m |= DESLOC_SYNC_V;
    return m;
}

constexpr int NUM_SMS = 148;   // of a B200

// Chunk length of a context: a run of tiles of the kernel that serves its worker count -- as
// many as amortise the per-chunk pointer look-up on a large problem (max_tiles_per_chunk), fewer
// on a small one, so that it still spreads over about four blocks per SM of a B200.
// Three to eight workers, whose averaging steps give a chunk to a block: a problem between two and
// 8 * 8 rounds of blocks takes the run that fills its last round -- as few rounds of at most 8 tiles as
// it needs, and the shortest run that does with these.  All-sync steps, Adam, bf16 gradients, against
// the first rule: eight workers, 400 K parameters 16.2 us instead of 22.7, 700 K 27.3 (32.1), 2 M 72.3 (80.2), 5 M 164.8
// (172.2); four workers, 1 M 19.5 (21.1), 2 M 36.2 (39.3).  A tensor costs a block more for its short first chunk
// (head_elems), and how many blocks are in a round depends on optimizer and gradient type: without both, models of 47
// tensors, x averaged, cold in L2, took eight workers x 690 K parameters 35.8 us (now 31.6), x 1 M 46.3 (39.9), with fp32 gradients
// and ADOPT x 690 K 35.3 (28.7), six x 920 K 35.3 (29.6).  The rule knows no addresses: a tensor on a 2 KB boundary has no short
// first chunk, and is counted as if it had.  Averaging steps of 3060 random lists, packed, padded and allocated apart,
// against the first rule: 0.68 to 1.28 of the time, 0.98 on average, 584 faster and 127 slower by more than 3 % (the best
// length of each list: 0.96).
constexpr int64_t ALIGN_PHASE_ELEMS = 512;
inline int64_t chunk_elems_for(int opt, bool bf16, int32_t M, const int64_t *numel, int32_t num_tensors) {
    const int64_t T = M <= MAX_MT ? plan_tile_elems(M) : GENERIC_CHUNK_ELEMS;
    const int64_t most = M <= MAX_MT ? max_tiles_per_chunk(M) : 8;
    int64_t tiles = 0, heads = 0;
    for (int32_t k = 0; k < num_tensors; ++k) {
        tiles += (numel[k] + T - 1) / T;
        heads += numel[k] > ALIGN_PHASE_ELEMS ? 1 : 0;
    }
    int64_t per_chunk = tiles / (4 * NUM_SMS);
    if (M > 2 && M <= MAX_MT) {
        const int64_t slots = static_cast<int64_t>(NUM_SMS) * step_min_blocks(opt, M, bf16);
        // chunks of t tiles, a tensor's last one half full on average
        const auto chunks_with = [&](int64_t t) { return (tiles + num_tensors * (t - 1) / 2 + t - 1) / t + heads; };
        // (at most eight of the kernel's own tiles: ADOPT, eight workers, fp32 gradients, 1.5 M parameters in a round of long
        // chunks 62 us, in two of shorter ones 57)
        const int64_t limit = tile_elems(opt, M, bf16) < T ? most / 2 : most;
        const int64_t rounds = (chunks_with(limit) + slots - 1) / slots;
        if (tiles > 2 * slots && rounds <= 8) {
            per_chunk = 1;
            while (per_chunk < limit && chunks_with(per_chunk) > rounds * slots) ++per_chunk;
        }
    }
    if (per_chunk < 1) per_chunk = 1;
    if (per_chunk > most) per_chunk = most;
    return per_chunk * T;
}
inline int64_t chunk_elems_for(const desloc_config &c, int32_t M) {
    return chunk_elems_for(c.opt, c.grad_dtype == DESLOC_BF16, M, c.numel, c.num_tensors);
}

// Where the copy engine's 2 KB pieces start matters: measured on B200, tiles that begin 256 or
// 512 bytes off a 2 KB boundary of the fp32 arrays run 3 % slower than tiles on the boundary
// (1 KB off: 0.7 %).  So the first chunk of a tensor is cut short by `head` elements, such that
// every later chunk of it starts on a 2 KB boundary of worker 0's x -- and with it of every
// array that shares x's element offsets, the usual layout (one flat buffer per worker and array).
// The same cut turns a tensor that starts at an odd offset of a tightly packed buffer (x not
// 16-byte aligned: every chunk of it would take the scalar path), or at an odd multiple of four
// elements of a buffer padded to 16 bytes (x aligned, a bf16 gradient with the same offsets
// 8 bytes off), into a short head and an aligned rest.  A gradient that does NOT share x's
// offsets can lose its 16-byte alignment by the cut; where it keeps 8 bytes, the chunk is
// updated with 128-bit accesses from global memory (0.66-0.86 of the copy bandwidth), else
// coordinate by coordinate.
inline int64_t head_elems(const void *x0, int64_t numel) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(x0);
    if ((a & 3u) != 0) return 0;
    const int64_t phase = static_cast<int64_t>(a >> 2) & (ALIGN_PHASE_ELEMS - 1);
    const int64_t head = (ALIGN_PHASE_ELEMS - phase) & (ALIGN_PHASE_ELEMS - 1);
    return head < numel ? head : 0;
}

// Chunks of one tensor: an optional short first chunk of `head` elements, then chunk_elems each.
inline int64_t chunks_of(int64_t numel, int64_t chunk_elems, int64_t head) {
    return (head > 0 ? 1 : 0) + (numel - head + chunk_elems - 1) / chunk_elems;
}

// heads: per tensor, elements of the short first chunk (0 = none), or nullptr for none at all.
inline int64_t count_chunks(const int64_t *numel, int32_t num_tensors, int64_t chunk_elems,
                            const int64_t *heads = nullptr) {
    int64_t n = 0;
    for (int32_t k = 0; k < num_tensors; ++k) n += chunks_of(numel[k], chunk_elems, heads ? heads[k] : 0);
    return n;
}

// The chunks of a launch, as its plan sees them.
struct ChunkSet {
    int64_t n = 0;
    int64_t length = 0;     // of a whole chunk,
    int64_t longest = 0;    // and of the longest one that there is: a list of small tensors has none of whole length
    int64_t total = 0;      // of all
};
inline ChunkSet chunk_set(const int64_t *numel, int32_t num_tensors, int64_t chunk_elems, const int64_t *heads = nullptr) {
    ChunkSet s{count_chunks(numel, num_tensors, chunk_elems, heads), chunk_elems, 0, 0};
    for (int32_t k = 0; k < num_tensors; ++k) {
        const int64_t head = heads ? heads[k] : 0, rest = numel[k] - head;
        const int64_t most = rest < chunk_elems ? rest : chunk_elems;
        s.longest = s.longest > most ? s.longest : most;
        s.longest = s.longest > head ? s.longest : head;
        s.total += numel[k];
    }
    return s;
}

// Blocks that share a chunk of all mt replicas (of one, for mt = 1).
inline int64_t parts_for(int64_t chunk_elems, int opt, int mt, bool bf16) {
    const int64_t most = most_part_elems(opt, mt, bf16);
    return (chunk_elems + most - 1) / most;
}

// The same where `items` chunks (times replicas, for mt = 1) make no more than four rounds of blocks: the split that
// takes the fewest tile times, a round costing its tiles and 0.7 of one to fill and drain.  Measured, all-sync: sixteen
// workers, 100 K parameters 11.7 us instead of 15.9, 1.5 M 107 (114); two workers, 200 K 3.5 (5.2), 2 M 18.9 (20.1).
inline int64_t parts_for(int64_t items, int64_t chunk_elems, int opt, int mt, bool bf16) {
    const int64_t least = parts_for(chunk_elems, opt, mt, bf16), tile = tile_elems(opt, mt, bf16);
    const int64_t tiles = (chunk_elems + tile - 1) / tile;
    const int64_t slots = static_cast<int64_t>(NUM_SMS) * step_min_blocks(opt, mt, bf16);
    int64_t best = least, best_cost = INT64_MAX;
    if (items * least > 4 * slots) return least;
    for (int64_t p = least; p <= tiles; ++p) {
        const int64_t cost = (items * p + slots - 1) / slots * (10 * ((tiles + p - 1) / p) + 7);
        if (cost < best_cost) best = p, best_cost = cost;
    }
    return best;
}

// One thread block per part of a chunk and worker on a local step, one per chunk on the others: does
// the largest grid of a context with M workers fit, whatever the first chunks are cut to?
inline bool grid_fits(const desloc_config &c, int32_t M) {
    const int64_t chunk_elems = chunk_elems_for(c, M);
    const int64_t nchunks = count_chunks(c.numel, c.num_tensors, chunk_elems) + c.num_tensors;
    const int64_t per_chunk = M * parts_for(chunk_elems, OPT_ADAM, 1, true);
    return nchunks <= 0x7fffffffLL / per_chunk;
}

// Writes the chunk table for the list (every tensor starts a new chunk); `out` has room for
// count_chunks() entries.
inline void fill_chunks(const int64_t *numel, int32_t num_tensors, int64_t chunk_elems, Chunk *out,
                        const int64_t *heads = nullptr) {
    int64_t c = 0;
    for (int32_t k = 0; k < num_tensors; ++k) {
        const int64_t head = heads ? heads[k] : 0;
        if (head > 0) {
            out[c].tensor = k;
            out[c].count = static_cast<int32_t>(head);
            out[c].start = 0;
            ++c;
        }
        for (int64_t s = head; s < numel[k]; s += chunk_elems) {
            const int64_t left = numel[k] - s;
            out[c].tensor = k;
            out[c].count = static_cast<int32_t>(left < chunk_elems ? left : chunk_elems);
            out[c].start = s;
            ++c;
        }
    }
}

// The hyper-parameter part of the kernel arguments (tables and sizes are the caller's).
inline void fill_hyper(StepArgs &a, const desloc_config &c, float lr_t, float clip_bound_t) {
    a.nt = c.num_tensors;
    a.M = c.M;
    a.b1 = c.beta1;
    a.omb1 = static_cast<float>(1.0 - static_cast<double>(c.beta1));
    a.b2 = c.beta2;
    a.omb2 = static_cast<float>(1.0 - static_cast<double>(c.beta2));
    a.eps2 = static_cast<float>(static_cast<double>(c.eps) * static_cast<double>(c.eps));
    a.lam2 = static_cast<float>(static_cast<double>(c.eps) * static_cast<double>(c.eps));
    a.lr = lr_t;
    a.lrwd = static_cast<float>(static_cast<double>(lr_t) * static_cast<double>(c.weight_decay));
    a.rho = c.clip_rho > 0.f ? c.clip_rho : std::numeric_limits<float>::infinity();
    a.cbound = (c.flags & DESLOC_FLAG_ADOPT_NORM_CLIP) ? clip_bound_t
                                                       : std::numeric_limits<float>::infinity();
    a.wait_limit = DEFAULT_WAIT_LIMIT;
    a.err = nullptr;
    a.direct = 0;
    a.parts = 1;
    a.parts_inv = 0;
    a.part_elems = 0;
}

inline const void *lookup_crowd_kernel(int opt, bool post, bool bf16, int kind, int mask, bool diag) {
    return opt == OPT_ADAM ? lookup_crowd_adam(post, bf16, kind, mask, diag)
           : opt == OPT_ADOPT ? lookup_crowd_adopt(post, bf16, kind, mask, diag) : lookup_crowd_sgdm(post, bf16, kind, mask, diag);
}

inline const void *lookup_lanes_kernel(int opt, bool post, bool bf16, int mt, int mask) {
    return opt == OPT_ADAM ? lookup_lanes_adam(post, bf16, mt, mask)
           : opt == OPT_ADOPT ? lookup_lanes_adopt(post, bf16, mt, mask) : lookup_lanes_sgdm(post, bf16, mt, mask);
}

// Which kernel a step of this configuration runs, and over how many blocks.
enum class Kernel { TILES, RUNTIME_M, LANES, CROWD };
struct LaunchPlan {
    Kernel kernel = Kernel::TILES;
    const void *fn = nullptr;
    long long grid = 0;       // blocks in x
    unsigned grid_y = 1;      // one-replica kernel: workers
    bool strides = true;  // a smaller grid may stride over the work items (not the runtime-M kernel)
    int smem = 0;         // dynamic shared memory of the launch
    int smem_limit = 0;   // of any launch of this kernel
    int threads = BLOCK_THREADS, threads_y = 1;
    int parts = 1, part_elems = 0;   // blocks that share a chunk, and elements of it for each
    bool direct = false;  // too small to gain from staging: update straight from global memory
    bool whole = false;   // a block takes a whole chunk, straight from global memory: no shared memory to stage in
    bool overlap = true;  // may begin while the kernel in front of it still runs (not the runtime-M kernel)
};

// Steps with norm diagnostics (small problems without them, and averaging ones of more than eight workers with them, run in
// desloc_lanes_kernel and desloc_crowd_kernel): launches of at most this many blocks of single-tile chunks (two per SM of a B200: one wave)
// skip the staging.  Measured on 4096 parameters and two workers: 3.08 us per step in a
// CUDA graph of 16 steps against 3.34 us staged.
constexpr long long DIRECT_GRID = 2 * NUM_SMS;
// Blocks of desloc_lanes_kernel that are resident at once.
constexpr long long LANES_WAVE = 10 * NUM_SMS;
// As many that their loads (8 KB a block) find room in the 28 KB of L1 that a kernel with much shared memory leaves behind.
constexpr long long LANES_FEW = 3 * NUM_SMS;
// One-replica kernel: at most seven blocks of one tile per SM go straight to global memory.
constexpr long long LOCAL_WAVE = 7 * NUM_SMS;

// The tile kernels use more than the 48 KB of shared memory a kernel gets by default: raise the
// function's limit to the most that any launch of it asks for (launches of other contexts, with
// more tiles per block, share it).  Not an allocation.
inline cudaError_t prepare_launch(const LaunchPlan &p) {
    if (p.smem_limit <= 32 * 1024) return cudaSuccess;   // with the kernel's static part still under 48 KB
    return cudaFuncSetAttribute(p.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, p.smem_limit);
}

// Launches `fn`.  overlap: the kernel may begin while the one in front of it in the stream still runs
// (see begin_and_let_next_begin); also under capture, where it becomes an edge of the graph.  Measured
// on B200: a graph window of 16 dependent steps on 4096 parameters 28.0 us instead of 43.0, a 5 M-parameter
// step of four workers 82.0 us instead of 85.7, 135 M parameters 2044 us instead of 2050.  The runtime-M
// kernel neither begins early nor lets others: its blocks are few and long, and those of the next step crowded
// onto the SMs this one left free (24 workers x 125 K parameters, 123 blocks: 23.9 us instead of 14.4).
inline cudaError_t launch_kernel(const void *fn, dim3 grid, dim3 threads, size_t smem, cudaStream_t stream,
                                 void **params, bool overlap) {
    cudaLaunchConfig_t lc{};
    lc.gridDim = grid;
    lc.blockDim = threads;
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = &at;
    lc.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelExC(&lc, fn, params);
}

// Nine to sixteen workers, a problem of few single-tile chunks: the runtime-M kernel has three places for a chunk
// per SM where the tiles have two, and needs a round of blocks less for some counts.  It is the faster one there,
// measured over all counts of workers, optimizers and types with 350 to 420 chunks by 1.1 to 1.75 (nine workers, 350
// chunks, u averaged: 11.9 us instead of 19.7), with 600 to 870 by 1.0 to 1.4, beyond, with one array
// averaged, by 0.97 to 1.13; ADOPT with several arrays averaged and more than a round of blocks: 0.87 to 1.3, not taken.
// For as many rounds it is the faster one where one array of three is averaged (with more than a chunk per SM, 1.0
// to 1.47; from 13 workers on not in the second round, 0.87 to 1.05).
inline bool generic_fills_rounds_better(const desloc_config &c, uint32_t mask, long long nchunks, int64_t chunk_elems) {
    if (chunk_elems > GENERIC_CHUNK_ELEMS || nchunks <= NUM_SMS) return false;
    const long long tile_slots = static_cast<long long>(NUM_SMS) * step_min_blocks(c.opt, c.M, c.grad_dtype == DESLOC_BF16);
    const long long slots = static_cast<long long>(NUM_SMS) * GENERIC_MIN_BLOCKS, rounds = (nchunks + slots - 1) / slots;
    const bool fewer = rounds < (nchunks + tile_slots - 1) / tile_slots;
    if ((mask & (mask - 1)) == 0 && (fewer || (c.opt != DESLOC_SGDM && (rounds == 1 || c.M <= 12)))) return true;
    return fewer && (rounds == 1 || (rounds == 2 && c.opt != DESLOC_ADOPT));
}

// How the gradients lie towards the copy engine, which takes 16-byte aligned pieces: FIT, or at least a quarter of
// the parameters have gradients that it cannot take, most of these (bf16) 8-byte aligned -- OFF -- or less -- NARROW.
// fp32 gradients are FIT or OFF.  heads: elements of the short first chunks; grads: [M][num_tensors].
enum class GradLayout { FIT, OFF, NARROW };
// asked: a smaller problem's plan asks, too.
inline GradLayout grad_layout(const desloc_config &c, const void *const *grads, const int64_t *heads, bool asked) {
    const bool bf16 = c.grad_dtype == DESLOC_BF16;
    int64_t total = 0, off = 0, narrow = 0;
    // (no plan for fewer elements than this asks: the look at 1088 pointers takes 6 us)
    for (int32_t k = 0; k < c.num_tensors; ++k) total += c.numel[k];
    if (total * c.M < (1 << 21) && !asked) return GradLayout::FIT;
    for (int32_t k = 0; k < c.num_tensors; ++k) {
        const uintptr_t head = static_cast<uintptr_t>(heads[k]) * (bf16 ? 2 : 4);
        uintptr_t bits = 0;
        for (int32_t m = 0; m < c.M; ++m)
            bits |= reinterpret_cast<uintptr_t>(grads[static_cast<int64_t>(m) * c.num_tensors + k]) + head;
        if ((bits & 15u) != 0) off += c.numel[k];
        if (bf16 && (bits & 7u) != 0) narrow += c.numel[k];
    }
    if (off < total - off - off - off) return GradLayout::FIT;
    return narrow > off - narrow ? GradLayout::NARROW : GradLayout::OFF;
}

// The most coordinates (parameters times workers) of a step with mt replicas that runs with these in the lanes of a warp.
// Measured with the arrays cold in L2, 4260 points of lists of 1 to 200 tensors (Adam, ADOPT, SGDM, both gradient types), against the tile
// kernels: local steps of 2 to 7 million 0.91 to 0.95 of the time on average, of 10 to 15 million 0.97, of a hundred million at the power cap
// 1.02 to 1.03; two workers 3 million 0.95, 4.6 million 1.02; four 5 to 7 million 0.98, 10 million 1.0; eight 3 to 5 million 0.8 to 0.9
// (from 4.2 million on, behind one another from Python, 1.05 to 1.13), 10 million 1.07; three, and five to seven, of which lanes are idle, 1.5 million 0.7 to 0.9, 2.2 million 0.8 to 1.05, 5 million 1.02 to 1.06.
// Counted by chunks times their length, as they were before, lists of many tensors left these kernels at half the size.  Averaging steps that
// moved, 1600 random lists at the lines against the tiles: four workers 0.98 of the time (up to 1.07), five to seven 0.7 (five: see
// full_round_of_three), eight 0.85 (3 in 100 lists above 1.04, up to 1.1: a single round of tile blocks, exactly filled).
inline int64_t lanes_most(int mt) {
    return mt == 1 ? 16000000 : mt == 2 ? 5000000 : mt == 3 ? 1700000 : mt == 4 ? 7000000 : mt == 8 ? 3800000 : 2000000;
}

// One round of tile blocks that each update three tiles, at least nineteen in twenty of them full, five workers, Adam or ADOPT, fp32 gradients that
// fit: where all arrays are averaged, and before the update, the tiles take 0.81 to 1.03 of the lanes' time (once 1.14) from 1.6 million on, 0.9 on
// average (5 x 350 K 10.8 us, 13.1).  (Smaller ones were not compared.  Not taken: one or two arrays 0.85 to 1.18, 1.0 on average; six workers 0.9 to
// 1.26, 1.02; SGDM 1.2, averages behind the update 1.5, gradients off the state's layout 1.7.)
inline bool full_round_of_three(const desloc_config &c, const ChunkSet &chunks) {
    if (c.M != 5 || c.opt == DESLOC_SGDM || c.grad_dtype == DESLOC_BF16 || (c.flags & DESLOC_FLAG_POST_AVERAGE) ||
        chunks.total * c.M <= 1600000 || chunks.total * c.M > lanes_most(c.M)) return false;
    const int64_t tile = tile_elems(c.opt, c.M, false), tiles = (chunks.length + tile - 1) / tile, parts = parts_for(chunks.n, chunks.length, c.opt, c.M, false);
    const int64_t blocks = chunks.n * parts;
    return blocks <= static_cast<int64_t>(NUM_SMS) * step_min_blocks(c.opt, c.M, false) && (tiles + parts - 1) / parts == 3 && 20 * chunks.total >= 57 * blocks * tile;
}

// The same of averaging steps of more than eight workers that run in desloc_crowd_kernel.  Measured, as above: nine and ten workers
// 1.5 million 0.67 to 0.79, 2.2 million 0.9 to 0.97; 12 and 14 2.2 million 0.7 to 0.8, 3.2 million 0.87 to 0.98; 16 3.2 million 0.87, 4.6 million 1.0;
// 20 and 24 3.2 million 0.67, 4.2 million 0.7, 5.6 million 0.9 (up to 1.2); 32 5.6 million 0.78, 10 million 0.9; 64 7 million 0.7, 10 million 0.98; 128 and
// 256 up to ten million 0.03 to 0.82 (15: 0.7 to 1.2).  SGDM, which has the least to load, by itself: nine and ten 1.8 million 0.8, 2.4 million 1.13; 12 and
// 14 2.3 to 2.5 million 0.6 to 0.95 (12 x 196 K 11.2 us, tiles 18.6), three lists of large aligned tensors 1.04; 16 2.4 million 0.73, 3.2 million 1.09; 20 and 24 4.2 million 0.94, 5.6 million 1.03; 32 5.6 million 0.72, 10 million 1.03.
// Steps that moved with the count by coordinates, 900 random lists: nine and ten workers 0.7 of the time, 12 and 14 0.82, 16 0.78; 2 in 100 above 1.04, up to
// 1.19 (all arrays averaged, a single round of tile blocks, exactly filled; half of the lists that fill one so take 0.8, by how the workers' tensors lie).
inline int64_t crowd_most(int opt, int mt) {
    if (opt == OPT_SGDM) return mt < 12 ? 1590000 : mt <= 16 ? 2500000 : mt <= 24 ? 4000000 : mt <= 32 ? 5500000 : mt <= 64 ? 8000000 : 10000000;
    return mt < 12 ? 2100000 : mt < 16 ? 3100000 : mt == 16 ? 4200000 : mt <= 24 ? 4500000 : mt <= 32 ? 8000000 : 10000000;
}

// A part of a chunk per block, as many as the longest chunk has.  (With as many as a chunk of whole length has, lists of small
// tensors launched 2 to 64 times the blocks that had work, a nanosecond each: 200 tensors of 78 elements x 12 workers, averaged,
// 7.6 us where the tiles took 4.8; 38 of 16 elements x 128 workers, local, 11.1 and 6.1.)
inline void plan_parts(LaunchPlan &p, const ChunkSet &chunks, int part_elems) {
    p.part_elems = part_elems;
    p.parts = static_cast<int>((chunks.longest + part_elems - 1) / part_elems);
    p.grid = chunks.n * p.parts;
    p.strides = false;
}

// lanes_ok: (false in tests of the tile kernels)
inline LaunchPlan plan_launch(const desloc_config &c, uint32_t mask, const ChunkSet &chunks,
                              bool diag, bool scaled, GradLayout layout, bool lanes_ok = true) {
    LaunchPlan p;
    const long long nchunks = chunks.n;
    const int64_t chunk_elems = chunks.length;
    // The mean of one replica is the replica: M = 1 always runs the local kernel.
    const uint32_t kmask = (c.M == 1) ? 0u : mask;
    const bool post = (c.flags & DESLOC_FLAG_POST_AVERAGE) != 0;
    const bool bf16 = c.grad_dtype == DESLOC_BF16;
    const bool local = kmask == 0;
    // More than eight workers, beyond crowd_most(): tiles of all replicas up to sixteen, the runtime-M kernel beyond, for the
    // post-average ordering and for the norm diagnostics.  All-sync steps of sixteen workers (Adam, bf16
    // gradients): 6.52 TB/s in tiles, 6.29 in the runtime-M kernel; nine workers 6.2 and 5.89.
    const int mt = local ? 1 : c.M;
    const int64_t replicas = local ? c.M : 1;
    // (a launch may cover some of the chunks)
    const int64_t coords = (chunks.total < nchunks * chunk_elems ? chunks.total : nchunks * chunk_elems) * c.M;
    if (lanes_ok && !diag && mt <= MAX_MT && coords <= lanes_most(mt)) {
        plan_parts(p, chunks, lanes_part_elems(mt));
        // Local steps of long lists whose chunks differ so much in length that most of the blocks' room is empty.  More than four
        // waves of chunks, three quarters of the room empty: 0.96 to 1.25 of the tiles' time, 1.09 on average (fewer chunks 0.54 to
        // 1.15, 0.87; more of the room filled 0.49 to 1.14, 0.82).  SGDM, which has the least to load, two waves and 55 %: 0.95 to
        // 1.75, 1.3 on average (else 0.58 to 1.37, 0.9).  Where a block takes a whole chunk there is one for each, as there
        // would be of tiles: 0.49 to 1.06.
        const bool sgdm = c.opt == OPT_SGDM, sparse = p.parts > 1 && 20 * chunks.total < (sgdm ? 9 : 5) * p.grid * p.part_elems;
        // Blocks for more than twice as many coordinates as the line allows, of lists of thousands of tensors: tiles, too.
        const bool crowded = p.grid * p.part_elems * c.M > 2 * lanes_most(mt);
        const bool tiles_full = kmask == 7 && layout == GradLayout::FIT && full_round_of_three(c, chunks);
        if (!crowded && !tiles_full && !(local && sparse && nchunks * c.M > (sgdm ? 2 : 4) * LANES_WAVE)) {
            p.kernel = Kernel::LANES;
            p.fn = lookup_lanes_kernel(c.opt, post, bf16, mt, static_cast<int>(kmask));
            p.threads = LANES_THREADS;
            if (local) p.grid_y = static_cast<unsigned>(c.M);
            p.direct = p.grid * p.grid_y <= LANES_FEW;
            return p;
        }
        p = LaunchPlan();
    }
    if (lanes_ok && mt > MAX_MT && coords <= crowd_most(c.opt, mt)) {
        const int L = crowd_lanes(c.M), threads = c.M * L;
        plan_parts(p, chunks, 4 * L);
        if (p.grid * p.part_elems * c.M <= 2 * crowd_most(c.opt, mt)) {   // (else crowded, as above)
            const int kind = threads > 512 ? CROWD_1024 : threads > 256 ? CROWD_512
                             : p.grid <= crowd_min_blocks(CROWD_FEW) * NUM_SMS ? CROWD_FEW : CROWD_256;
            p.kernel = Kernel::CROWD;
            p.fn = lookup_crowd_kernel(c.opt, post, bf16, kind, static_cast<int>(kmask), diag);
            p.threads = L;
            p.threads_y = c.M;
            p.smem = crowd_smem_bytes(c.opt, bf16, c.M);
            p.smem_limit = crowd_smem_limit(kind);
            return p;
        }
        p = LaunchPlan();
    }
    // Gradients that the copy engine cannot take, in problems of more than four rounds of blocks (smaller ones are served
    // from L2 and gain nothing).  Measured with 60 M parameters x workers, Adam, gradients 8 bytes off the state's layout:
    // whole chunks per block, nothing staged, for one replica (247 -> 213 us) and two (272 -> 222); the runtime-M
    // kernel, which reads with 128-bit accesses, for nine workers and more (sixteen: 404 -> 258 us; where the
    // accesses are narrow anyway, from thirteen on: 595 -> 470).
    const bool off_many = layout != GradLayout::FIT && mt <= MAX_TILE_MT &&
                          nchunks * replicas * parts_for(chunk_elems, c.opt, mt, bf16) >
                              4LL * NUM_SMS * step_min_blocks(c.opt, mt, bf16);
    const bool off_generic = off_many && ((bf16 && layout == GradLayout::OFF) || mt > 12);
    const bool generic = !local && c.M > MAX_MT &&
                         (c.M > MAX_TILE_MT || post || diag || off_generic ||
                          generic_fills_rounds_better(c, kmask, nchunks, chunk_elems));
    p.kernel = generic ? Kernel::RUNTIME_M : Kernel::TILES;
    p.fn = generic ? lookup_generic_kernel(c.opt, post, bf16, static_cast<int>(kmask), diag)
                   : lookup_step_kernel(c.opt, post, bf16, c.M, static_cast<int>(kmask), diag);
    p.strides = p.overlap = !generic;
    p.grid = nchunks;
    if (!generic) {
        const int64_t tile = tile_elems(c.opt, mt, bf16), tiles = (chunk_elems + tile - 1) / tile;
        // (with a factor on the gradients, behind norm clipping, whole chunks were 3-6 % slower)
        const bool whole = p.whole = off_many && layout == GradLayout::OFF && mt <= 2 && !diag && !scaled;
        // (the diagnostics write one partial sum per chunk: their blocks take whole chunks)
        int64_t parts = diag || whole ? 1 : parts_for(nchunks * replicas, chunk_elems, c.opt, mt, bf16);
        // Gradients that neither the copy engine nor 128-bit accesses take: blocks go coordinate by coordinate, and what
        // counts is that none stands idle.  Five to eight workers, where more than a fifth of the rounds' tiles would be
        // empty: a tile to a block, 0.41 to 1.09 of the time (0.83 on average; 7 x 580 K parameters in 100 tensors, ADOPT, fp32
        // gradients, x averaged: 86.9 us and 44.3).  In fuller rounds up to 1.17, with three and four workers up to 1.21: not taken.
        const int64_t slots = static_cast<int64_t>(NUM_SMS) * step_min_blocks(c.opt, mt, bf16), rounds = (nchunks * parts + slots - 1) / slots;
        if (!diag && mt > 4 && mt <= MAX_MT && layout != GradLayout::FIT && !(bf16 && layout == GradLayout::OFF) && rounds <= 4 &&
            5 * chunks.total < 4 * rounds * slots * ((tiles + parts - 1) / parts) * tile)
            parts = tiles;
        p.parts = static_cast<int>(parts);
        p.part_elems = static_cast<int>((tiles + parts - 1) / parts * tile);
        p.threads = step_threads(c.opt, mt, bf16);
        p.smem = whole ? 0 : step_smem_bytes(c.opt, mt, bf16, p.part_elems);
        p.smem_limit = step_smem_bytes(c.opt, mt, bf16, most_part_elems(c.opt, mt, bf16));
        p.grid = nchunks * parts;
        if (local) p.grid_y = static_cast<unsigned>(c.M);
        p.direct = whole || (p.grid * replicas <= (local ? LOCAL_WAVE : DIRECT_GRID) && p.part_elems <= (local ? tile : plan_tile_elems(mt)));
    }
    return p;
}

// How a launch cuts its chunks, into the kernel arguments.
inline void fill_plan(StepArgs &a, const LaunchPlan &p) {
    a.parts = p.parts;
    a.parts_inv = p.parts > 1 ? static_cast<unsigned>(((1ull << 32) + p.parts - 1) / p.parts) : 0;
    a.part_elems = p.part_elems;
    a.direct = p.direct ? 1 : 0;
}

}  // namespace desloc
