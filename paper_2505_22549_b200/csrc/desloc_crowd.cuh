// Averaging steps of more than eight workers on small and mid-sized problems: a thread per worker and four
// coordinates, as in desloc_lanes.cuh, with the worker means through shared memory.
//
// Bound: latency, then HBM.  The tile kernels of nine to sixteen workers have two blocks per SM and update small
// problems worker by worker from global memory; the runtime-M kernel goes over the workers in batches of one to four,
// one round trip after another: 64 workers took 23 us for 60 K coordinates (parameters times workers).  Here every
// load of a block is in flight at once; a block writes the arrays to be averaged to shared memory, each of its
// threads sums some columns over the workers -- trees of four and a compensated sum over them, as the
// other kernels (post-average: trees of one, two or four, as the runtime-M kernel) -- and all read the means back.  The addresses are looked up
// again for the stores (from L1), which leaves the registers for six blocks of 256 threads instead of four.
//
// Measured on B200, arrays cold in L2, Adam, bf16 gradients, all arrays averaged (before): 16 workers x 4 K parameters 2.4 us
// (6.1), x 62 K 7.2 (14.4), x 100 K 9.9 (11.0); 24 x 100 K 14.5 (24.6); 64 x 1 K 2.9 (26.3), x 55 K 21.7 (54.5);
// 256 x 250 5.3 (79.6), x 27 K 76 (196).  Half as many lanes per worker and twice as many blocks, or
// the reverse, were 2 to 20 % slower at a million coordinates and above.
#pragma once
#include <utility>

#include "desloc_lanes.cuh"

namespace desloc {

// Mean of column[0], column[T], ... column[(M - 1) T]: trees of B values (1, 2 or 4; what is left value by value) in a
// compensated sum.
template <int B>
__device__ __forceinline__ float column_mean(const float *column, int T, int M, float inv_m) {
    float sum = 0.f, err = 0.f;
    const auto add = [&](float x) {
        const float t = sum + x, bp = t - sum;
        err += (sum - (t - bp)) + (x - bp);
        sum = t;
    };
    int m = 0;
#pragma unroll 2
    for (; m + 4 <= M; m += 4) {
        const float s[4] = {column[m * T], column[(m + 1) * T], column[(m + 2) * T], column[(m + 3) * T]};
        if constexpr (B == 4) {
            add(tree_sum<0, 4, 4>(s));
        } else if constexpr (B == 2) {
            add(s[0] + s[1]);
            add(s[2] + s[3]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) add(s[k]);
        }
    }
    if (B == 2 && m + 2 <= M) {
        add(column[m * T] + column[(m + 1) * T]);
        m += 2;
    }
    for (; m < M; ++m) add(column[m * T]);
    const float hi = sum + err, lo = err - (hi - sum);   // hi + lo = sum + err
    return div_by_count(hi, lo, static_cast<float>(M), inv_m);
}

// Lanes of a worker, threads of a block and blocks per SM.  FEW: blocks that all fit at once four to an SM, where
// the registers are better spent than on more blocks (12 x 40 K: 4.2 us against 4.5; 2320 lists of 9 to 64 workers: with
// CROWD_256 0.91 to 1.26 of the time, 1.017 on average).
__host__ __device__ constexpr int crowd_lanes(int M) { return M < 12 ? 16 : M <= 32 ? 8 : 4; }
constexpr int CROWD_FEW = 0, CROWD_256 = 1, CROWD_512 = 2, CROWD_1024 = 3;
__host__ __device__ constexpr int crowd_threads(int kind) { return kind <= CROWD_256 ? 256 : kind == CROWD_512 ? 512 : 1024; }
__host__ __device__ constexpr int crowd_min_blocks(int kind) {
    return kind == CROWD_FEW ? 4 : kind == CROWD_256 ? 6 : kind == CROWD_512 ? 3 : 1;
}
// Shared memory: [array][worker][coordinate], where the loads land and what is averaged is found, and three arrays of means.
__host__ __device__ constexpr int crowd_smem_bytes(int opt, bool bf16, int M) {
    return (((opt == OPT_SGDM ? 2 : 3) + (bf16 ? 0 : 1)) * M + 3) * 4 * crowd_lanes(M) * 4;
}
__host__ __device__ constexpr int crowd_smem_limit(int kind) { return 4 * crowd_threads(kind) * 16 + 3 * 4 * 16 * 4; }

// Blocks of crowd_lanes(M) x M threads; a work item is 4 * crowd_lanes(M) coordinates of a chunk, of all replicas.
// DIAG: also the sums of squares of gradient, new parameters and update, a partial sum per block, worker and kind, reduced by shuffles where they
// arise; two thirds of the blocks, for the registers.  205 random lists of 9 to 64 workers, averaging steps with diagnostics (before: the
// runtime-M kernel, which lets one block go over all workers of a chunk): up to 0.5 million coordinates 3.3 to 7 us (15 to 29), a million 14.5 (27.7),
// two million 21 (38).
template <int OPT, int MASK, typename GT, bool POST, int KIND, bool DIAG = false>
__global__ void __launch_bounds__(crowd_threads(KIND), DIAG && KIND != CROWD_1024 ? crowd_min_blocks(KIND) * 2 / 3 : crowd_min_blocks(KIND))
desloc_crowd_kernel(const __grid_constant__ StepArgs a) {
    extern __shared__ __align__(16) float pool[];
    begin_and_let_next_begin();
    const unsigned c = item_chunk(a, blockIdx.x);
    const int part0 = static_cast<int>(blockIdx.x - c * a.parts) * a.part_elems;
    const Chunk ch = a.chunks[c];
    const int cnt = min(ch.count - part0, a.part_elems);
    const int M = a.M, L = blockDim.x, T = 4 * L, m = threadIdx.y, lx = threadIdx.x;
    const auto put = [&](int kind, float v) {
        a.diag[(static_cast<long long>(kind) * M + m) * a.diag_stride + blockIdx.x] = v;
    };
    if (cnt <= 0) {   // (of the whole block)
        if (DIAG && lx == 0) {
            wait_for_earlier_kernels();
            for (int kind = 0; kind < DIAG_KINDS; ++kind) put(kind, 0.f);
        }
        return;
    }
    const auto norms = [&](int kind, float v) {
        const int first = (m * L + lx) & ~31, there = M * L - first;   // (the last warp may be a part of one)
        const unsigned lanes = there >= 32 ? 0xffffffffu : (1u << there) - 1;
        for (int o = L / 2; o > 0; o /= 2) v += __shfl_down_sync(lanes, v, o, L);
        if (lx == 0) put(kind, v);
    };
    const auto replica = [&] { return Replica<OPT, GT>(a, static_cast<long long>(m) * a.nt + ch.tensor, ch.start + part0); };
    const Replica<OPT, GT> w = replica();
    // (the stores' addresses: kept where there are registers for it -- 478 random lists of 10 K to 0.3 million coordinates 0.96 of the time)
    const auto to = [&] { return KIND == CROWD_FEW ? w : replica(); };
    const bool wide = __syncthreads_and(w.wide_ok() && (cnt & 3) == 0) != 0;
    float *const means = pool + landing_arrays<OPT, GT>() * M * T;
    const Landing land{pool + m * T + 4 * lx, M * T};
    float inv_m = 1.f / static_cast<float>(M);
    asm volatile("" : "+f"(inv_m));   // (the division stays in front of the wait: 0.99 of the time)
    const auto mean_of_arrays = [&](const auto &q, auto &s, auto arrays, bool landed) {
        using Batch = PostBatch<OPT, MASK, GT>;
        constexpr int N = arrays.N, B = !POST ? 4 : arrays.at(0) == 0 ? Batch::X : Batch::STATES;
        if (!landed) {
#pragma unroll
            for (int i = 0; i < N; ++i) q.st(pool + (arrays.at(i) * M + m) * T, s[i]);
        }
        __syncthreads();
        for (int i = m * L + lx; i < N * T; i += M * L) {
            const int k = i / T, e = i - k * T;
            if (e < cnt) means[i] = column_mean<B>(pool + arrays.at(k) * M * T + e, T, M, inv_m);
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < N; ++i) s[i] = q.ld(means + i * T);
    };
    const Quad<true> q4{4 * lx, 1, cnt, true};
    const auto mean4 = [&](auto &s, auto arrays) { mean_of_arrays(q4, s, arrays, !POST); };
    const Quad<false> q1{lx, L, cnt, true};
    const auto mean1 = [&](auto &s, auto arrays) { mean_of_arrays(q1, s, arrays, false); };
    if constexpr (DIAG) {
        wait_for_earlier_kernels();
        if (blockIdx.x == 0 && m == 0 && lx == 0) *a.diag_parts = a.parts;
        const float sc = a.gscale ? a.gscale[m] : 1.f;
        if (wide) update_quad<OPT, MASK, GT, POST, false, true>(a, sc, q4, land, w, to, mean4, norms);
        else update_quad<OPT, MASK, GT, POST, false, false>(a, sc, q1, land, w, to, mean1, norms);
    } else {
        if (wide && plain_step<OPT>(a)) {   // (the common form: nothing but its loads behind the wait)
            wait_for_earlier_kernels();
            update_quad<OPT, MASK, GT, POST, true, true>(a, 1.f, q4, land, w, to, mean4);
            return;
        }
        wait_for_earlier_kernels();
        const float sc = a.gscale ? a.gscale[m] : 1.f;
        if (wide) update_quad<OPT, MASK, GT, POST, false, true>(a, sc, q4, land, w, to, mean4);
        else update_quad<OPT, MASK, GT, POST, false, false>(a, sc, q1, land, w, to, mean1);
    }
}

template <int OPT, typename GT, bool POST, bool DIAG, int NMASK, int... I>
const void *pick_crowd(int kind, int mask, std::integer_sequence<int, I...>) {
    static const void *const tbl[] = {
        reinterpret_cast<const void *>(&desloc_crowd_kernel<OPT, 1 + I % NMASK, GT, POST, I / NMASK, DIAG>)...};
    if (kind < CROWD_FEW || kind > CROWD_1024 || mask < 1 || mask > NMASK) return nullptr;
    return tbl[kind * NMASK + mask - 1];
}

template <int OPT, typename GT>
const void *lookup_crowd(bool post, int kind, int mask, bool diag) {
    constexpr int NMASK = OPT == OPT_SGDM ? 3 : 7;
    using Seq = std::make_integer_sequence<int, 4 * NMASK>;
    if (diag) return post ? pick_crowd<OPT, GT, true, true, NMASK>(kind, mask, Seq{}) : pick_crowd<OPT, GT, false, true, NMASK>(kind, mask, Seq{});
    return post ? pick_crowd<OPT, GT, true, false, NMASK>(kind, mask, Seq{}) : pick_crowd<OPT, GT, false, false, NMASK>(kind, mask, Seq{});
}

// One unit per optimizer.
const void *lookup_crowd_adam(bool post, bool bf16, int kind, int mask, bool diag);
const void *lookup_crowd_adopt(bool post, bool bf16, int kind, int mask, bool diag);
const void *lookup_crowd_sgdm(bool post, bool bf16, int kind, int mask, bool diag);

}  // namespace desloc
