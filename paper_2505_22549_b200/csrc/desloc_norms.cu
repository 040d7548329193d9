// Reductions around the DES-LOC step: per-worker gradient norms for norm-based clipping (the
// clipping the paper's language-model runs used), the relative rate of change of a state,
// ||s_now - s_then||_2 / ||s_then||_2 (Section 5.1, "Metrics"), and the finalisation of the
// per-tensor gradient / parameter / update norms a diagnostics step accumulated.
//
// All are deterministic and, but for the gradient norms of small problems, two-stage: stage 1 writes one fp32 partial per work item -- per-thread
// sums of up to 128 squares, a shuffle tree, then the warp sums in order; stage 2 adds the
// partials of a row in fp64 in a fixed pattern.  No atomics.
#include "desloc_norms.cuh"

#include <type_traits>

namespace desloc {

namespace {

// ---- stage 1: sums of squares over 32 KB of one worker's array(s) ------------------------------
// Bound: HBM reads.  A block requests all it will read -- 32 KB, as bulk copies into shared memory --
// at once, sums it and leaves; six blocks per SM keep 192 KB in flight.  (Before: 64 KB per block and
// three blocks for bf16 gradients, register loads for fp32 gradients and for the rate of change.)
// Measured on 135 M parameters x 4 workers: rate of change (4.3 GB) 620 us instead of 740, the whole call;
// 20 M x 8 workers 200 us instead of 245; the norm-clipped step 2210 us instead of 2259 with bf16 gradients,
// 2494 instead of 2533 with tightly packed fp32 gradients.
constexpr int RED_THREADS = 128;
constexpr int RED_BYTES = 32 * 1024;

// MODE 0, 1: g of fp32, bf16 -- one sum of g^2.  MODE 2: a state and its snapshot -- sums of
// (now - then)^2 and of then^2.
constexpr int RED_F32 = 0, RED_BF16 = 1, RED_CHANGE = 2;
__host__ __device__ constexpr int red_chunks(int mode) {   // reduction chunks (4096 elements) per work item
    return RED_BYTES / (REDUCE_CHUNK_ELEMS * (mode == RED_BF16 ? 2 : mode == RED_F32 ? 4 : 8));
}

template <int MODE>
__device__ __forceinline__ void add_squares(const uint4 &p, const uint4 &q, float (&acc)[2]) {
    const unsigned w[4] = {p.x, p.y, p.z, p.w}, z[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if constexpr (MODE == RED_BF16) {
            const float lo = __uint_as_float(w[k] << 16), hi = __uint_as_float(w[k] & 0xffff0000u);
            acc[0] = fmaf(lo, lo, acc[0]);
            acc[1] = fmaf(hi, hi, acc[1]);
        } else if constexpr (MODE == RED_F32) {
            const float f = __uint_as_float(w[k]);
            acc[k & 1] = fmaf(f, f, acc[k & 1]);
        } else {
            const float b = __uint_as_float(z[k]), d = __uint_as_float(w[k]) - b;
            acc[0] = fmaf(d, d, acc[0]);
            acc[1] = fmaf(b, b, acc[1]);
        }
    }
}

// partial[m * stride + q]: item q of worker m (MODE 2: the squares of `then` at (M + m) * stride + q).
// One work item per block: red_chunks(MODE) consecutive reduction chunks of one worker.
template <int MODE>
__global__ void __launch_bounds__(RED_THREADS, 6)
sumsq_kernel(const Chunk *chunks, long long nchunks, const void *const *now, const void *const *then, int nt, int M,
             float *partial, long long stride, int *err, int wait_limit) {
    using GT = std::conditional_t<MODE == RED_BF16, bf16_t, float>;
    constexpr int NC = red_chunks(MODE), NA = MODE == RED_CHANGE ? 2 : 1;
    constexpr int CHUNK_BYTES = REDUCE_CHUNK_ELEMS * static_cast<int>(sizeof(GT));
    extern __shared__ __align__(128) char stage[];   // [chunk][array][CHUNK_BYTES]
    __shared__ const char *s_base[NC][2];
    __shared__ int s_count[NC], s_head[NC], s_staged[NC];   // elements, how many in front of the staged ones
    __shared__ float warp_sums[2][RED_THREADS / 32];
    __shared__ __align__(8) uint64_t bar;
    const int tid = threadIdx.x;
    begin_and_let_next_begin();
    const unsigned ngroups = static_cast<unsigned>((nchunks + NC - 1) / NC);
    const int m = static_cast<int>(blockIdx.x / ngroups);
    const long long q = blockIdx.x - m * ngroups;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(&bar)), "r"(NC) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // one thread per chunk of the item
    const char *p0 = nullptr, *p1 = nullptr;
    int count = 0;
    if (tid < NC && q * NC + tid < nchunks) {
        const Chunk ch = chunks[q * NC + tid];
        const long long idx = static_cast<long long>(m) * nt + ch.tensor, off = ch.start * static_cast<long long>(sizeof(GT));
        p0 = reinterpret_cast<const char *>(now[idx]) + off;
        if constexpr (MODE == RED_CHANGE) p1 = reinterpret_cast<const char *>(then[idx]) + off;
        count = ch.count;
    }
    __syncthreads();   // the barrier exists
    wait_for_earlier_kernels();
    if (tid < NC) {
        // Staged is what lies behind the first 128-byte boundary, in whole 16-byte pieces; the elements in
        // front of it and the last ones are read directly (all of them where the two arrays lie
        // differently).  Copies that start off a 128-byte line fetch every line twice: 4.2 TB/s instead of 6.9
        // on a tightly packed fp32 buffer.
        constexpr int ESZ = static_cast<int>(sizeof(GT)), PIECE = 16 / ESZ;
        const uintptr_t a0 = reinterpret_cast<uintptr_t>(p0), a1 = MODE == RED_CHANGE ? reinterpret_cast<uintptr_t>(p1) : a0;
        const bool can = a0 % ESZ == 0 && ((a0 ^ a1) & 15u) == 0;
        const int head = can ? min(count, static_cast<int>((0 - a0) & 127u) / ESZ) : 0;
        const int staged = can ? (count - head) & ~(PIECE - 1) : 0;
        const uint32_t bytes = staged * static_cast<uint32_t>(ESZ);
        if (bytes) {
            bulk_load(stage + tid * NA * CHUNK_BYTES, p0 + head * ESZ, bytes, &bar);
            if constexpr (MODE == RED_CHANGE) bulk_load(stage + (tid * NA + 1) * CHUNK_BYTES, p1 + head * ESZ, bytes, &bar);
        }
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                     :: "r"(smem_u32(&bar)), "r"(NA * bytes) : "memory");
        s_base[tid][0] = p0; s_base[tid][1] = p1;
        s_count[tid] = count; s_head[tid] = head; s_staged[tid] = staged;
    }
    __syncthreads();
    float acc[2] = {0.f, 0.f};
    // what is not staged
#pragma unroll 1
    for (int k = 0; k < NC; ++k) {
        for (int r = tid; r < s_count[k] - s_staged[k]; r += RED_THREADS) {
            const int e = r < s_head[k] ? r : r + s_staged[k];
            const float a = ld_grad<1, GT>(s_base[k][0], e).a[0];
            if constexpr (MODE == RED_CHANGE) {
                const float b = ld_f32<1>(s_base[k][1], e).a[0], d = a - b;
                acc[0] = fmaf(d, d, acc[0]);
                acc[1] = fmaf(b, b, acc[1]);
            } else {
                acc[0] = fmaf(a, a, acc[0]);
            }
        }
    }
    const bool landed = bar_wait(&bar, 0, wait_limit);
    if (__syncthreads_or(!landed)) {
        // give up: say so, let the copies land (bounded as well), leave
        if (tid == 0 && err) *reinterpret_cast<volatile int *>(err) = 1;
        bar_wait(&bar, 0, DRAIN_WAIT_LIMIT);
        __syncthreads();
        return;
    }
#pragma unroll 1
    for (int k = 0; k < NC; ++k) {
        const uint4 *a = reinterpret_cast<const uint4 *>(stage + k * NA * CHUNK_BYTES);
        const uint4 *b = a + (NA - 1) * (CHUNK_BYTES / 16);
        const int n = s_staged[k] * static_cast<int>(sizeof(GT)) / 16;
#pragma unroll 4
        for (int v = tid; v < n; v += RED_THREADS) add_squares<MODE>(a[v], b[v], acc);
    }
    if constexpr (MODE != RED_CHANGE) acc[0] += acc[1];
#pragma unroll
    for (int j = 0; j < NA; ++j) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc[j] += __shfl_down_sync(0xffffffffu, acc[j], off);
        if ((tid & 31) == 0) warp_sums[j][tid >> 5] = acc[j];
    }
    __syncthreads();
    if (tid < NA) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < RED_THREADS / 32; ++w) t += warp_sums[tid][w];
        partial[(static_cast<long long>(tid) * M + m) * stride + q] = t;
    }
}

// ---- stage 2 -------------------------------------------------------------------------------------
// Sum of row[0 .. n) in fp64 in a fixed pattern (each thread its groups of four, in order; then a
// shuffle tree and the warps in order), the same in every thread.  All loads of a thread are independent:
// a row of 16 K partials takes 2-3 us instead of 10 with one serial load per thread and 256 entries.
// `row` is 16-byte aligned and n a multiple of four where WIDE.
template <bool WIDE>
__device__ __forceinline__ double row_sum_f64(const float *row, long long n, double *sh) {
    double acc = 0.0;
    const int threads = blockDim.x;
    if constexpr (WIDE) {
        const float4 *r4 = reinterpret_cast<const float4 *>(row);
#pragma unroll 8
        for (long long i = threadIdx.x; i < n / 4; i += threads) {
            const float4 v = r4[i];
            acc += (static_cast<double>(v.x) + v.y) + (static_cast<double>(v.z) + v.w);
        }
    } else {
#pragma unroll 16
        for (long long i = threadIdx.x; i < n; i += threads) acc += static_cast<double>(row[i]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    __syncthreads();   // sh may still be read from the previous use
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    double r = 0.0;
    for (int w = 0; w < threads / 32; ++w) r += sh[w];
    return r;
}

// Rows of partials are padded to a multiple of four entries: block m adds zeros there.
__device__ __forceinline__ void pad_row(float *row, long long n, long long stride) {
    if (threadIdx.x < stride - n) row[n + threadIdx.x] = 0.f;
    __syncthreads();
}

// norm = sqrt(sum of squares), scale = min(1, max_norm / norm) (1 when max_norm <= 0).
__device__ __forceinline__ void finish_norm(double ss, float max_norm, float *norm, float *scale) {
    const double nrm = sqrt(ss);
    *norm = static_cast<float>(nrm);
    *scale = (max_norm > 0.f && nrm > static_cast<double>(max_norm)) ? static_cast<float>(static_cast<double>(max_norm) / nrm) : 1.f;
}

// The last word of a read-out: behind it, all that is complete for this kernel's wait is complete for the host that sees the word -- the flag of
// a bounded wait that ran out, too, which an earlier kernel has stored there.  By a block of its own, the first, while the others add up.
__device__ __forceinline__ void release_results(float *word) {
    if (threadIdx.x != 0) return;
    __threadfence_system();
    *reinterpret_cast<volatile float *>(word) = 1.f;
}

constexpr int FINAL_THREADS = 512;

// norms[m] = ||g^m||_2, scales[m] = min(1, max_norm / norms[m]) (1 when max_norm <= 0).
__global__ void __launch_bounds__(FINAL_THREADS)
norm_finalize_kernel(float *partial, long long n, long long stride, float max_norm, float *norms, float *scales) {
    __shared__ double sh[FINAL_THREADS / 32];
    begin_and_let_next_begin();
    wait_for_earlier_kernels();
    const int m = blockIdx.x;
    float *row = partial + m * stride;
    pad_row(row, n, stride);
    const double ss = row_sum_f64<true>(row, stride, sh);
    if (threadIdx.x == 0) finish_norm(ss, max_norm, norms + m, scales + m);
}

__global__ void __launch_bounds__(FINAL_THREADS)
relchange_finalize_kernel(float *partial, long long n, long long stride, int M, float *out, float *released) {
    __shared__ double sh[FINAL_THREADS / 32];
    begin_and_let_next_begin();
    wait_for_earlier_kernels();
    if (blockIdx.x == 0) return release_results(released);
    const int m = blockIdx.x - 1;
    float *row = partial + m * stride, *row2 = partial + (static_cast<long long>(M) + m) * stride;
    pad_row(row, n, stride);
    pad_row(row2, n, stride);
    const double num = row_sum_f64<true>(row, stride, sh);
    const double den = row_sum_f64<true>(row2, stride, sh);
    if (threadIdx.x == 0) out[m] = static_cast<float>(sqrt(num) / sqrt(den));
}

// ---- small problems: gradient norms in one launch -------------------------------------------------
// Bound: latency, and the launch (2 us of the host's time, as much as the kernel).  A cluster of eight blocks takes all of a worker's gradients: a
// warp reads a piece of 1024 elements straight into registers, all of it at once, adds the lanes' fp32 sums (32 squares of a
// piece) in fp64, and the blocks hand their sums to the first one through its shared memory.  A warp has one piece to read, of
// lists of many tensors half a chunk or one: few wait for a second round trip.
// A norm-clipped step of SGDM in a graph of dependent steps (before: two stages), bf16 gradients: one worker x 2 K parameters 2.7 us (4.3), x 131 K
// 3.3 (4.9); four x 33 K 3.6 (5.2), x 120 K in 120 tensors 4.5 (7.2); from Python 5.4 (7.9), where the launch counts.  Rates of
// change, which the host waits for either way, gained 1 us of 18 at best and lost as much with many tensors: not taken.
constexpr int SMALL_THREADS = 512, SMALL_BLOCKS = 8, SMALL_PIECE = 1024, SMALL_PIECES = REDUCE_CHUNK_ELEMS / SMALL_PIECE;
constexpr int SMALL_WARPS = SMALL_BLOCKS * SMALL_THREADS / 32;
constexpr int64_t SMALL_BYTES = 4 << 20;   // of all workers
// Workers whose clusters are all resident at once (two blocks per SM with fp32 gradients, three with bf16), and the chunks from which on more of them
// come in one launch, too: clusters come in waves then, which cost what the two stages pay for some 40 chunks per worker.  Norm-clipped steps in a
// graph, one launch and two stages: 64 workers in 3 and 8 tensors 8.3 us and 7.3, 11.4 and 7.7; 128 x 2 K parameters 15.0 and 9.6, 256 x 1 K in 4
// 28.2 and 16.2; but 64 x 29 K in 100 tensors 21.9 and 27.9, 128 x 100 in 100 14.5 and 20.1, 256 in 47 and 56 1.0 to 1.16 in favour of one.
constexpr int SMALL_MANY_CHUNKS = 40;
constexpr int small_workers(bool bf16) { return (bf16 ? 3 : 2) * 148 / SMALL_BLOCKS; }

__device__ __forceinline__ uint32_t first_block_addr(const void *shared) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(shared)));
    return r;
}

template <int MODE>
__global__ void __cluster_dims__(SMALL_BLOCKS, 1, 1) __launch_bounds__(SMALL_THREADS)
small_norms_kernel(const Chunk *chunks, int nchunks, const void *const *g, int nt, float max_norm, float *norms, float *scales) {
    using GT = std::conditional_t<MODE == RED_BF16, bf16_t, float>;
    constexpr int ESZ = static_cast<int>(sizeof(GT)), PER = 16 / ESZ, ROUNDS = SMALL_PIECE / PER / 32;
    __shared__ double warp_sums[SMALL_THREADS / 32];
    __shared__ double block_sums[SMALL_BLOCKS];   // (the first block's)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int m = static_cast<int>(blockIdx.x) / SMALL_BLOCKS, rank = static_cast<int>(blockIdx.x) % SMALL_BLOCKS;
    begin_and_let_next_begin();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // (do the blocks exist?  asked below)
    // Half chunks or whole ones where there is not a warp for each piece of them.
    const int at = rank * (SMALL_THREADS / 32) + warp;
    const int share = nchunks <= SMALL_WARPS / 4 ? SMALL_PIECES : nchunks <= SMALL_WARPS / 2 ? 2 : 1;
    const int c = at / share, part = REDUCE_CHUNK_ELEMS / share;
    double total = 0.0;
    int count = 0;
    const char *p = nullptr;
    if (c < nchunks) {
        const Chunk ch = chunks[c];
        const int e0 = (at - c * share) * part;
        count = min(ch.count - e0, part);
        p = reinterpret_cast<const char *>(g[static_cast<long long>(m) * nt + ch.tensor]) + (ch.start + e0) * static_cast<long long>(ESZ);
    }
    wait_for_earlier_kernels();
#pragma unroll 1
    for (int done = 0; done < count; done += SMALL_PIECE, p += SMALL_PIECE * ESZ) {
        // 16-byte loads from the first boundary on; what lies around them element by element
        const int n = min(count - done, SMALL_PIECE);
        const uintptr_t addr = reinterpret_cast<uintptr_t>(p);
        const bool can = addr % ESZ == 0;
        const int head = can ? min(n, static_cast<int>((0 - addr) & 15u) / ESZ) : 0, wide = can ? (n - head) / PER : 0;
        const uint4 *w = reinterpret_cast<const uint4 *>(p + head * ESZ);
        uint4 v[ROUNDS];
#pragma unroll
        for (int r = 0; r < ROUNDS; ++r) v[r] = r * 32 + lane < wide ? w[r * 32 + lane] : make_uint4(0, 0, 0, 0);
        float acc[2] = {0.f, 0.f};
        for (int i = lane; i < n - wide * PER; i += 32) {
            const float f = ld_grad<1, GT>(p, i < head ? i : i + wide * PER).a[0];
            acc[0] = fmaf(f, f, acc[0]);
        }
#pragma unroll
        for (int r = 0; r < ROUNDS; ++r) add_squares<MODE>(v[r], v[r], acc);
        total += static_cast<double>(acc[0]) + acc[1];
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) total += __shfl_down_sync(0xffffffffu, total, off);
    if (lane == 0) warp_sums[warp] = total;
    __syncthreads();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    if (threadIdx.x == 0) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < SMALL_THREADS / 32; ++w) t += warp_sums[w];
        asm volatile("st.shared::cluster.f64 [%0], %1;" :: "r"(first_block_addr(&block_sums[rank])), "d"(t) : "memory");
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (rank == 0 && threadIdx.x == 0) {
        double t = 0.0;
#pragma unroll
        for (int r = 0; r < SMALL_BLOCKS; ++r) t += block_sums[r];
        finish_norm(t, max_norm, norms + m, scales + m);
    }
}

// dst^j[i] = mean over the M_src source replicas of src^m[i] (fp64 sum in the order
// m = 0..M_src-1, rounded once), for every destination replica j.  Work item = chunk.
__global__ void __launch_bounds__(BLOCK_THREADS, 4)
mean_fill_kernel(const Chunk *chunks, long long nchunks, const float *const *src, int m_src,
                 float *const *dst, int m_dst, int nt) {
    begin_and_let_next_begin();
    wait_for_earlier_kernels();
    for (long long c = blockIdx.x; c < nchunks; c += gridDim.x) {
        const Chunk ch = chunks[c];
        for (int e = threadIdx.x; e < ch.count; e += BLOCK_THREADS) {
            double acc = 0.0;
            for (int m = 0; m < m_src; ++m)
                acc += static_cast<double>(src[static_cast<long long>(m) * nt + ch.tensor][ch.start + e]);
            const float mean = static_cast<float>(acc / static_cast<double>(m_src));
            for (int j = 0; j < m_dst; ++j)
                dst[static_cast<long long>(j) * nt + ch.tensor][ch.start + e] = mean;
        }
    }
}

// Norm diagnostics of a DIAG step.  partial[row * nchunks * parts + i], row = kind * M + m, holds the sum of
// squares of part i % parts of chunk i / parts (parts = *parts_of: of the step that ran last); tstart[k] .. tstart[k + 1] are the chunks of tensor k.  A block per (row,
// tensor): fp64 sum of the tensor's chunks, its root as the per-tensor norm.  In front of them `rows` blocks that
// take a whole row each: the norm over the tensor list.  One launch, and all results go
// straight to the host's memory.  (A warp per row and tensor spent 20 us in a row on the 6912 chunks of an
// embedding; three partial sums per chunk, for shorter blocks in the step, made the step no faster.)
constexpr int DIAG_THREADS = 256;

__global__ void __launch_bounds__(DIAG_THREADS)
diag_norms_kernel(const float *partial, long long nchunks, const int *parts_of, const long long *tstart, int nt, int rows, float *norms,
                  float *totals, float *released) {
    __shared__ double sh[DIAG_THREADS / 32];
    begin_and_let_next_begin();
    wait_for_earlier_kernels();
    if (blockIdx.x == 0) return release_results(released);
    const int parts = *parts_of, block = static_cast<int>(blockIdx.x) - 1;
    const long long stride = nchunks * parts;
    const bool whole = block < rows;
    const long long item = static_cast<long long>(block) - rows;
    const long long row = whole ? block : item / nt;
    const int k = static_cast<int>(item - row * nt);
    const long long c0 = whole ? 0 : tstart[k] * parts, c1 = whole ? stride : tstart[k + 1] * parts;
    const double ss = row_sum_f64<false>(partial + row * stride + c0, c1 - c0, sh);
    if (threadIdx.x == 0) (whole ? totals + row : norms + item)[0] = static_cast<float>(sqrt(ss));
}

// All launches of this file may begin while the kernel in front of them still runs.
template <typename... P, typename... A>
cudaError_t launch(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream, A... args) {
    cudaLaunchConfig_t lc{};
    lc.gridDim = grid;
    lc.blockDim = dim3(threads);
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = &at;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, kernel, static_cast<P>(args)...);
}

unsigned grid_for(long long nitems) {
    return static_cast<unsigned>(nitems < 0x7fffffffLL ? (nitems > 0 ? nitems : 1) : 0x7fffffffLL);
}

}  // namespace

template <int MODE>
static cudaError_t launch_sumsq(const Chunk *chunks, long long nchunks, const void *const *now, const void *const *then,
                                int nt, int M, float *partial, long long *items, long long *stride, int *err,
                                int wait_limit, cudaStream_t stream) {
    *items = (nchunks + red_chunks(MODE) - 1) / red_chunks(MODE);
    *stride = reduce_row(*items);
    return launch(sumsq_kernel<MODE>, grid_for(*items * M), RED_THREADS, RED_BYTES, stream, chunks, nchunks, now, then, nt,
                  M, partial, *stride, err, wait_limit);
}

cudaError_t launch_grad_norms(const Chunk *chunks, long long nchunks, int64_t elems, const void *const *g, int nt,
                              int M, bool bf16, float max_norm, float *partial, float *norms,
                              float *scales, int *err, int wait_limit, cudaStream_t stream, int *launches) {
    // A piece, half a chunk or a chunk for each warp of a cluster.  Beyond 4 MB in all the two stages read no slower (16 workers x 129 K parameters,
    // fp32, in 33 and 65 tensors, in a graph: 19.1 and 18.9 us in two stages, 20.0 and 20.2 in one; 2 bytes each 16.8 and 15.3, 15.7 and 14.1).
    if ((M <= small_workers(bf16) || nchunks >= SMALL_MANY_CHUNKS) && elems <= SMALL_WARPS * SMALL_PIECE && nchunks <= SMALL_WARPS &&
        elems * M * (bf16 ? 2 : 4) <= SMALL_BYTES) {
        *launches = 1;
        return launch(bf16 ? small_norms_kernel<RED_BF16> : small_norms_kernel<RED_F32>, M * SMALL_BLOCKS, SMALL_THREADS, 0, stream, chunks,
                      nchunks, g, nt, max_norm, norms, scales);
    }
    *launches = 2;
    long long items, stride;
    const cudaError_t e =
        bf16 ? launch_sumsq<RED_BF16>(chunks, nchunks, g, nullptr, nt, M, partial, &items, &stride, err, wait_limit, stream)
             : launch_sumsq<RED_F32>(chunks, nchunks, g, nullptr, nt, M, partial, &items, &stride, err, wait_limit, stream);
    if (e != cudaSuccess) return e;
    return launch(norm_finalize_kernel, M, FINAL_THREADS, 0, stream, partial, items, stride, max_norm, norms, scales);
}

cudaError_t launch_rel_change(const Chunk *chunks, long long nchunks, const float *const *now,
                              const float *const *then, int nt, int M, float *partial, float *out, float *released,
                              int *err, int wait_limit, cudaStream_t stream) {
    long long items, stride;
    const cudaError_t e = launch_sumsq<RED_CHANGE>(
        chunks, nchunks, reinterpret_cast<const void *const *>(now), reinterpret_cast<const void *const *>(then), nt, M,
        partial, &items, &stride, err, wait_limit, stream);
    if (e != cudaSuccess) return e;
    return launch(relchange_finalize_kernel, M + 1, FINAL_THREADS, 0, stream, partial, items, stride, M, out, released);
}

cudaError_t launch_diag_norms(const float *partial, long long nchunks, const int *parts, const long long *tstart,
                              int nt, int M, float *per_tensor, float *totals, float *released,
                              cudaStream_t stream) {
    const int rows = DIAG_KINDS * M;
    const long long blocks = 1 + rows + static_cast<long long>(rows) * nt;
    return launch(diag_norms_kernel, grid_for(blocks), DIAG_THREADS, 0, stream, partial, nchunks, parts, tstart, nt, rows,
                  per_tensor, totals, released);
}

cudaError_t launch_mean_fill(const Chunk *chunks, long long nchunks, const float *const *src,
                             int m_src, float *const *dst, int m_dst, int nt, cudaStream_t stream) {
    return launch(mean_fill_kernel, grid_for(nchunks), BLOCK_THREADS, 0, stream, chunks, nchunks, src, m_src, dst, m_dst, nt);
}

}  // namespace desloc
