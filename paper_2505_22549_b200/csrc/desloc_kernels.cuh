// DES-LOC fused step kernel for sm_100a: one streaming pass over g, x, u, v of all M
// worker replicas (Algorithm 1 with the Adam, ADOPT and SGDM rules of Algorithms 2-3).
//
// Work decomposition.  The tensor list is cut into chunks of one tensor (table built once on the
// host); a chunk is a run of up to 8 or 16 tiles.  A thread block takes a chunk (or a part of one) of
// ALL M replicas -- on local steps, and for M = 1, of one replica -- and streams its tiles
// through two shared-memory buffers (one replica: as many as it has tiles):
//   1. the first 4*M threads look up the chunk's pointers once; each owns one (array, worker)
//      and issues ONE 1-D bulk asynchronous copy per tile (cp.async.bulk, the TMA engine; no
//      multicast, this GPU's own memory) of its 1-2 KB slice into the tile's buffer, all
//      signalling the buffer's mbarrier;
//   2. the block waits for the mbarrier (bounded; see bar_wait), then every thread updates its
//      coordinates in place in shared memory: the arrays whose period divides t are averaged
//      over the workers in a fixed tree order, then each worker takes its optimizer step -- a
//      sync step moves the same bytes as a local step, through the same code shape;
//   3. the owners of x, u, v each issue one bulk copy of the updated slice back, and, once
//      that copy has read the buffer, request the tile after next into it.
// While tile k is updated, tile k + 1 is landing and tile k - 1 is on its way back.  Two to
// seven blocks are resident per SM (one replica: ten).  A chunk whose pointers are not 16-byte aligned, and a
// ragged last tile whose byte counts are not multiples of 16, take the same arithmetic straight
// from and to global memory: four coordinates per thread with 128-bit accesses where the fp32
// arrays are 16-byte and the gradients at least 8-byte aligned, else one coordinate per thread.
//
// Measured on B200 (Adam, 4 workers, bf16 gradients, 1.7 G parameters; one local step):
//   registers only, 128-bit loads (4096-element chunks, 3 blocks/SM)   26.74 ms  1.015 of copy
//   registers only, 256-bit loads (ld.global.v8.f32)                   26.39 ms  1.029
//   bulk copies, 1024-element tiles, 2-stage pipeline, 2 blocks/SM     26.08 ms  1.041
//   bulk copies, persistent grid (2 blocks/SM striding)                30.2  ms  0.90
//   bulk copies, 512-element tiles, no pipeline, 6-8 blocks/SM         25.76 ms  1.055
// ("copy" = the device-to-device copy bandwidth of the same GPU; these are single-tensor
// experiments with the pointers in the kernel parameters).  In the library, with the tensor
// list's pointer look-up on every block's path, tiles of all replicas need the pipelined form: a run
// of 8 tiles per block through two buffers gives 26.1 ms (1.04) on the 218-tensor list.  Local
// steps take one replica per block, three tiles in buffers of their own: 25.5 ms (1.06).
//
// DIAG instantiations also accumulate, from values already in registers, the squared L2 norms
// of the gradient as read, of the update d_t and of the new parameters per (worker, chunk):
// no extra pass over memory, 12 bytes written per worker and chunk.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace desloc {

constexpr int OPT_ADAM = 0, OPT_ADOPT = 1, OPT_SGDM = 2;
constexpr int SYNC_X = 1, SYNC_U = 2, SYNC_V = 4;
constexpr int BLOCK_THREADS = 256; // of every kernel but the one-replica step kernel
constexpr int MAX_MT = 8;          // largest worker count with a kernel instantiated for every step
constexpr int MAX_TILE_MT = 16;    // ... for the pre-average sync steps without norm diagnostics
constexpr int DIAG_G = 0, DIAG_X = 1, DIAG_D = 2, DIAG_KINDS = 3;
constexpr int REDUCE_CHUNK_ELEMS = BLOCK_THREADS * 16;  // chunks of the reduction kernels (4096)
constexpr int GENERIC_CHUNK_ELEMS = 1024;               // chunks of contexts with M > MAX_MT
constexpr int GENERIC_MIN_BLOCKS = 3;                   // blocks per SM of the runtime-M kernel (80 registers)
constexpr int DRAIN_WAIT_LIMIT = 1 << 22;               // bound on the wait for copies in flight

// Elements per tile and worker for a kernel that holds mt replicas per tile: bulk copies of 2 KB per
// state array, 7-57 KB of shared memory per buffer (with bf16 gradients copies of 1 KB and 512 B,
// with 256-element tiles, were 5 % slower on eight workers).  Eight replicas with fp32 gradients and
// two states would need 64 KB per buffer, which leaves room for one block per SM: 256-element
// tiles and three blocks move 6.64 TB/s there instead of 5.5 (all-sync steps of 14 GB).
//
// Nine to sixteen replicas: as many elements, in units of a warp, as two buffers and two blocks per
// SM leave room for -- these kernels are bound by the bytes they keep in flight (twelve replicas, all-sync, with
// 256 elements 4.95 TB/s, with 320 6.2).
__host__ __device__ constexpr int tile_bytes_per_elem(int opt, int mt, bool bf16) {
    return mt * ((bf16 ? 2 : 4) + 4 * (opt == OPT_SGDM ? 2 : 3));
}
__host__ __device__ constexpr int tile_elems(int opt, int mt, bool bf16) {
    if (mt > MAX_MT) {
        const int t = 56 * 1024 / tile_bytes_per_elem(opt, mt, bf16) / 32 * 32;
        return t < 512 ? t : 512;
    }
    return mt == 8 && !bf16 && opt != OPT_SGDM ? 256 : 512;
}
// The unit in which a context's chunk table is cut (chunks are whole multiples of it).
__host__ __device__ constexpr int plan_tile_elems(int m) { return m <= 2 ? 1024 : 512; }
// Tiles per chunk on large problems (one pointer look-up and one pipeline fill serve them all):
// 8 measured best (4: sync steps 2 % slower; 16: 0.5-1 % slower; 32: 2 % slower).
__host__ __device__ constexpr int max_tiles_per_chunk(int) { return 8; }

// Elements of a chunk that one block takes.  One replica (local steps, a single worker): three
// tiles, one for each of its buffers.  Blocks that request everything they will ever need at once
// and leave keep the memory system busiest, the more of them the better: measured on B200 (Adam,
// bf16 gradients, 14 GB per step, a third of a second into the board's power cap) 6.92 TB/s with three
// tiles and ten blocks per SM, 6.86 with four and seven, 6.84-6.91 with two and ten to fifteen,
// 6.24-6.49 with tiles twice or four times as long, 6.79 for tiles of all replicas.  Two replicas: four tiles
// through two buffers, 6.85 against 6.78 with eight tiles of 1024 elements.  More: whole chunks
// (four tiles instead of eight cost eight workers 2 %, four workers nothing).
__host__ __device__ constexpr int most_part_elems(int opt, int mt, bool bf16) {
    return mt == 1 ? 3 * 512 : mt == 2 ? 4 * 512 : mt <= MAX_MT ? 8 * 512 : 8 * tile_elems(opt, mt, bf16);
}

struct __align__(16) Chunk {
    int32_t tensor;  // index into the tensor list
    int32_t count;   // elements in this chunk (<= the context's chunk length)
    int64_t start;   // first element within the tensor
};

// Programmatic dependent launch.  Every kernel here is launched so that it may begin while the kernel in
// front of it in the stream is still running: each block tells the next kernel at once that it may come
// (its blocks move in as the last ones of this kernel leave), does what depends on no earlier kernel --
// barriers, look-ups in tables that only copies write -- and then waits until everything in front
// of it is complete and visible.  No state, gradient, scale factor or partial sum is touched
// before that.  The wait is the launch's own dependency, resolved by the hardware, not a poll.
__device__ __forceinline__ void begin_and_let_next_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_earlier_kernels() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

constexpr int INLINE_PTRS = 32;  // gradient pointers that fit in the kernel parameters

struct StepArgs {
    const Chunk *chunks;
    long long nchunks;
    float *const *x;  // device tables [M * nt], entry m * nt + k
    float *const *u;
    float *const *v;
    const void *const *g;                // device table, or nullptr: use g_inline
    const void *g_inline[INLINE_PTRS];   // small problems under stream capture (no table upload)
    const float *gscale;  // per-worker factor applied to g before the clip, or nullptr (= 1)
    float *diag;          // DIAG kernels: [DIAG_KINDS][M][diag_stride] partial sums of squares
    long long diag_stride;  // chunks of the whole context, times the sums that a chunk gets
    int *diag_parts;        // that number: written by the step itself, which may be a captured one that runs at any time
    int *err;             // set to 1 when a bounded wait ran out (may be nullptr)
    int wait_limit;       // iterations a block polls for its tile before it gives up
    int direct;           // non-zero: no staging, every chunk straight from global memory (tiny launches)
    int parts;            // a chunk is this many work items (per replica, for the one-replica kernel) ...
    unsigned parts_inv;   // ceil(2^32 / parts) for more than one part (see item_chunk)
    int part_elems;       // ... of this many elements (a multiple of the tile; the last ones may be empty)
    int nt;
    int M;
    float b1, omb1;   // beta1, 1 - beta1
    float b2, omb2;   // beta2, 1 - beta2
    float eps2;       // ADOPT epsilon, squared
    float lam2;       // Adam lambda^2
    float lr;         // eta_t
    float lrwd;       // eta_t * weight_decay
    float rho;        // coordinate clip radius, +inf when off
    float cbound;     // ADOPT normalised-gradient bound, +inf when off
};

// No factor on the gradient, coordinate clip off (rho = +inf), epsilon^2 (not SGDM's) a normal number.
template <int OPT>
__device__ __forceinline__ bool plain_step(const StepArgs &a) {
    return a.gscale == nullptr && a.rho > 3.4028235e38f && (OPT == OPT_SGDM || a.lam2 >= 1.17549435e-38f);
}

// item / parts by a multiplication (the division is twenty instructions of every thread): exact for
// item < 2^32 / parts, far beyond what fits into memory.
__device__ __forceinline__ unsigned item_chunk(const StepArgs &a, unsigned item) {
    return a.parts == 1 ? item : __umulhi(item, a.parts_inv);
}

__device__ __forceinline__ const void *grad_ptr(const StepArgs &a, long long idx) {
    return a.g ? a.g[idx] : a.g_inline[idx];
}

struct bf16_t {
    uint16_t bits;
};

template <int VEC>
struct FV {
    float a[VEC];
};

// ---- global memory access: 128-bit or scalar (runtime-M kernel, reductions) ---------------
template <int VEC>
__device__ __forceinline__ FV<VEC> ld_f32(const char *base, long long elem) {
    FV<VEC> r;
    if constexpr (VEC == 4) {
        const float4 t = *(reinterpret_cast<const float4 *>(base) + (elem >> 2));
        r.a[0] = t.x; r.a[1] = t.y; r.a[2] = t.z; r.a[3] = t.w;
    } else if constexpr (VEC == 2) {
        const float2 t = *(reinterpret_cast<const float2 *>(base) + (elem >> 1));
        r.a[0] = t.x; r.a[1] = t.y;
    } else {
        r.a[0] = *(reinterpret_cast<const float *>(base) + elem);
    }
    return r;
}

template <int VEC>
__device__ __forceinline__ void st_f32(char *base, long long elem, const FV<VEC> &r) {
    if constexpr (VEC == 4) {
        *(reinterpret_cast<float4 *>(base) + (elem >> 2)) = make_float4(r.a[0], r.a[1], r.a[2], r.a[3]);
    } else if constexpr (VEC == 2) {
        *(reinterpret_cast<float2 *>(base) + (elem >> 1)) = make_float2(r.a[0], r.a[1]);
    } else {
        *(reinterpret_cast<float *>(base) + elem) = r.a[0];
    }
}

template <int VEC, typename GT>
__device__ __forceinline__ FV<VEC> ld_grad(const char *base, long long elem) {
    FV<VEC> r;
    if constexpr (sizeof(GT) == 4) {
        r = ld_f32<VEC>(base, elem);
    } else if constexpr (VEC == 4) {
        // four bf16 in 8 bytes; bf16 -> fp32 is a 16-bit shift (exact)
        const uint2 t = *(reinterpret_cast<const uint2 *>(base) + (elem >> 2));
        r.a[0] = __uint_as_float(t.x << 16);
        r.a[1] = __uint_as_float(t.x & 0xffff0000u);
        r.a[2] = __uint_as_float(t.y << 16);
        r.a[3] = __uint_as_float(t.y & 0xffff0000u);
    } else if constexpr (VEC == 2) {
        const unsigned t = *(reinterpret_cast<const unsigned *>(base) + (elem >> 1));
        r.a[0] = __uint_as_float(t << 16);
        r.a[1] = __uint_as_float(t & 0xffff0000u);
    } else {
        const unsigned short t = *(reinterpret_cast<const unsigned short *>(base) + elem);
        r.a[0] = __uint_as_float(static_cast<unsigned>(t) << 16);
    }
    return r;
}

template <int VEC>
__device__ __forceinline__ float sum_sq(const FV<VEC> &r) {
    float s = r.a[0] * r.a[0];
#pragma unroll
    for (int c = 1; c < VEC; ++c) s = fmaf(r.a[c], r.a[c], s);
    return s;
}

// ---- two coordinates at a time ------------------------------------------------------------------
// sm_100 has two-wide fp32 add, multiply and fused multiply-add, each half rounded as the scalar
// instruction rounds it: the same bits for half the instructions.  At the board's power cap that is speed: all-sync
// steps of sixteen workers 0.977 -> 1.003 of copy, local steps 1.053 -> 1.056.  An odd count takes the scalar
// forms, and so do (PACK = false) SGDM, whose averaging steps lost 0.3 % to the pairing, and the runtime-M
// kernel, which has no registers for pairs of constants (up to 6 % slower with them).
template <int VEC, bool PACK = true>
__device__ __forceinline__ FV<VEC> vfma(const FV<VEC> &x, const FV<VEC> &y, const FV<VEC> &z) {
    FV<VEC> r;
    if constexpr (PACK && VEC % 2 == 0) {
#pragma unroll
        for (int c = 0; c < VEC; c += 2) {
            const float2 t = __ffma2_rn(make_float2(x.a[c], x.a[c + 1]), make_float2(y.a[c], y.a[c + 1]),
                                        make_float2(z.a[c], z.a[c + 1]));
            r.a[c] = t.x; r.a[c + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int c = 0; c < VEC; ++c) r.a[c] = __fmaf_rn(x.a[c], y.a[c], z.a[c]);
    }
    return r;
}
template <int VEC, bool PACK = true>
__device__ __forceinline__ FV<VEC> vmul(const FV<VEC> &x, const FV<VEC> &y) {
    FV<VEC> r;
    if constexpr (PACK && VEC % 2 == 0) {
#pragma unroll
        for (int c = 0; c < VEC; c += 2) {
            const float2 t = __fmul2_rn(make_float2(x.a[c], x.a[c + 1]), make_float2(y.a[c], y.a[c + 1]));
            r.a[c] = t.x; r.a[c + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int c = 0; c < VEC; ++c) r.a[c] = __fmul_rn(x.a[c], y.a[c]);
    }
    return r;
}
template <int VEC, bool PACK = true>
__device__ __forceinline__ FV<VEC> vadd(const FV<VEC> &x, const FV<VEC> &y) {
    FV<VEC> r;
    if constexpr (PACK && VEC % 2 == 0) {
#pragma unroll
        for (int c = 0; c < VEC; c += 2) {
            const float2 t = __fadd2_rn(make_float2(x.a[c], x.a[c + 1]), make_float2(y.a[c], y.a[c + 1]));
            r.a[c] = t.x; r.a[c + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int c = 0; c < VEC; ++c) r.a[c] = __fadd_rn(x.a[c], y.a[c]);
    }
    return r;
}
template <int VEC>
__device__ __forceinline__ FV<VEC> splat(float v) {
    FV<VEC> r;
#pragma unroll
    for (int c = 0; c < VEC; ++c) r.a[c] = v;
    return r;
}
template <int VEC>
__device__ __forceinline__ FV<VEC> clamp(const FV<VEC> &x, float bound) {
    FV<VEC> r;
#pragma unroll
    for (int c = 0; c < VEC; ++c) r.a[c] = fminf(fmaxf(x.a[c], -bound), bound);
    return r;
}

// ---- the arithmetic of a thread's coordinates ------------------------------------------------------
// Worker sum as a fixed binary tree: the first 2^k workers (2^k the largest power of two
// below the count) against the rest, recursively -- ((s0+s1)+(s2+s3))+((s4+s5)+(s6+s7)) for
// eight.  Deterministic, and exact when all M values are equal and M is a power of two.
template <int LO, int N, int MT>
__device__ __forceinline__ float tree_sum(const float (&s)[MT]) {
    if constexpr (N == 1) {
        return s[LO];
    } else {
        constexpr int H = (N > 4) ? 4 : (N > 2 ? 2 : 1);
        static_assert(N <= 8, "tree_sum covers up to eight values");
        return tree_sum<LO, H, MT>(s) + tree_sum<LO + H, N - H, MT>(s);
    }
}

// (hi + lo) / n for a small whole number n: the product with the rounded reciprocal, corrected once by the residual
// hi + lo - q n, which a fused multiply-add gives exactly (the quotient correction of P. Markstein, "Computation of
// elementary functions on the IBM RISC System/6000 processor", 1990).  Straight-line code, so that the
// workers can be interleaved: all-sync steps of six, seven workers 6.49, 6.54 TB/s against 6.14, 6.22 with `/`.
__device__ __forceinline__ float div_by_count(float hi, float lo, float n, float inv_n) {
    const float q = hi * inv_n;
    const float r = fmaf(fmaf(-q, n, hi) + lo, inv_n, q);
    return fabsf(q) <= 3.0e38f ? r : q;   // (infinities and NaN stay what they are)
}

// More than eight workers: trees of four, then a compensated sum ("two-sum") over them in order -- the
// running sum and the exact rounding error of every addition, about 48 bits -- like the runtime-M kernel's.
template <int MT>
__device__ __forceinline__ float compensated_mean(const float (&s)[MT]) {
    float sum = tree_sum<0, 4, MT>(s), err = 0.f;
    const auto add = [&](float x) {
        const float t = sum + x, bp = t - sum;
        err += (sum - (t - bp)) + (x - bp);
        sum = t;
    };
    add(tree_sum<4, 4, MT>(s));
    if constexpr (MT >= 12) add(tree_sum<8, 4, MT>(s));
    if constexpr (MT >= 16) add(tree_sum<12, 4, MT>(s));
#pragma unroll
    for (int m = MT / 4 * 4; m < MT; ++m) add(s[m]);
    const float hi = sum + err, lo = err - (hi - sum);   // hi + lo = sum + err
    return div_by_count(hi, lo, static_cast<float>(MT), 1.f / MT);
}

// The sum of up to eight values as their mean.
template <int MT>
__device__ __forceinline__ float div_sum(float t) {
    if constexpr ((MT & (MT - 1)) == 0) return t * (1.f / MT);   // exact
    else return div_by_count(t, 0.f, static_cast<float>(MT), 1.f / MT);
}

template <int MT>
__device__ __forceinline__ float mean_of(const float (&s)[MT]) {
    if constexpr (MT > MAX_MT) {
        static_assert(MT <= MAX_TILE_MT, "three or four trees of four, and up to three more");
        return compensated_mean<MT>(s);
    } else {
        return div_sum<MT>(tree_sum<0, MT, MT>(s));
    }
}

// 1 / sqrt(a) to within an ulp: the hardware approximation (2 ulp) with one Newton step.  This
// replaces IEEE sqrt followed by IEEE division (two roundings, about 20 instructions): with the
// tiles staged by the copy engine the arithmetic sits on each block's critical path, and the
// exact pair cost 1 % on Adam with four workers and 5-11 % on ADOPT with eight.  The error is
// that of the exact pair (about one ulp of the quotient), not its bits.
__device__ __forceinline__ float rsqrt_1ulp(float a) {
    const float y = rsqrtf(a);
    const float r = y * fmaf(a * y, -0.5f * y, 1.5f);   // (halving y, not a: half of a denormal number may round)
    return a > 0.f && a < 3.0e38f ? r : y;   // keep the limits (1/0 = inf, 1/inf = 0) free of NaN
}

// The same of VEC values.  PLAIN: they are known to be normal numbers or above (the smallest is
// epsilon squared), so the approximation needs no scaling around it.
template <bool PLAIN, int VEC, bool P>
__device__ __forceinline__ FV<VEC> rsqrt_1ulp(const FV<VEC> &a) {
    FV<VEC> r;
    if constexpr (PLAIN) {
        FV<VEC> y;
#pragma unroll
        for (int c = 0; c < VEC; ++c) asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.a[c]) : "f"(a.a[c]));
        r = vmul<VEC, P>(y, vfma<VEC, P>(vmul<VEC, P>(vmul<VEC, P>(a, splat<VEC>(-0.5f)), y), y, splat<VEC>(1.5f)));
#pragma unroll
        for (int c = 0; c < VEC; ++c) r.a[c] = a.a[c] < 3.0e38f ? r.a[c] : y.a[c];
    } else {
#pragma unroll
        for (int c = 0; c < VEC; ++c) r.a[c] = rsqrt_1ulp(a.a[c]);
    }
    return r;
}

// One worker's state update from its gradient: `up`, `vp` are the previous states the update
// starts from (the worker's own or the worker mean); `vown` is always the worker's own previous v, which
// ADOPT's normaliser uses (Algorithm 3).  PLAIN: no factor `sc` on the gradient, no coordinate
// clip, and an epsilon whose square is a normal number.
template <int OPT, bool PLAIN, int VEC, bool P = OPT != OPT_SGDM>
__device__ __forceinline__ void state_update(const StepArgs &a, const FV<VEC> &g, float sc, const FV<VEC> &up,
                                             const FV<VEC> &vp, const FV<VEC> &vown, FV<VEC> &un, FV<VEC> &vn) {
    // coordinate-wise clip: sgn(g) min(|g|, rho)  (Section 3.1); rho = +inf when off
    FV<VEC> gh = g;
    if constexpr (!PLAIN) gh = clamp<VEC>(vmul<VEC, P>(g, splat<VEC>(sc)), a.rho);
    FV<VEC> r = gh;
    if constexpr (OPT == OPT_ADOPT) {
        FV<VEC> low;
#pragma unroll
        for (int c = 0; c < VEC; ++c) low.a[c] = fmaxf(vown.a[c], a.eps2);
        r = clamp<VEC>(vmul<VEC, P>(gh, rsqrt_1ulp<PLAIN, VEC, P>(low)), a.cbound);   // g / max(sqrt(v), eps)
    }
    un = vfma<VEC, P>(splat<VEC>(a.b1), up, vmul<VEC, P>(splat<VEC>(a.omb1), r));
    if constexpr (OPT == OPT_SGDM) vn = splat<VEC>(0.f);
    else vn = vfma<VEC, P>(splat<VEC>(a.b2), vp, vmul<VEC, P>(vmul<VEC, P>(splat<VEC>(a.omb2), gh), gh));
}

// -d_t: the update of Algorithms 2-3 from the new states, its sign turned.
template <int OPT, bool PLAIN, int VEC, bool P = OPT != OPT_SGDM>
__device__ __forceinline__ FV<VEC> minus_direction(const StepArgs &a, const FV<VEC> &un, const FV<VEC> &vn) {
    const FV<VEC> t = vmul<VEC, P>(splat<VEC>(-a.lr), un);
    if constexpr (OPT == OPT_ADAM) return vmul<VEC, P>(t, rsqrt_1ulp<PLAIN, VEC, P>(vadd<VEC, P>(vn, splat<VEC>(a.lam2))));
    else return t;
}

// x* (1 - eta wd) - d, written as x* - (eta wd x* + d): one rounding at x's scale
template <int VEC, bool P = true>
__device__ __forceinline__ FV<VEC> apply_step(const StepArgs &a, const FV<VEC> &xp, const FV<VEC> &minus_d) {
    return vadd<VEC, P>(xp, vfma<VEC, P>(splat<VEC>(-a.lrwd), xp, minus_d));
}

// ---- helpers of the runtime-M kernel ---------------------------------------------------------
// Registers a worker costs while its batch is in flight (FV<4> = 4 registers; bf16 g = 2).
template <int OPT, typename GT>
__host__ __device__ constexpr int worker_regs(bool ld_x, bool ld_u, bool ld_v) {
    return (sizeof(GT) == 2 ? 2 : 4) + 4 * ((ld_x ? 1 : 0) + (ld_u ? 1 : 0) + (ld_v ? 1 : 0));
}
// Post-average ordering: which per-worker values a parameter step needs after the means are known.
template <int OPT, int MASK>
struct PostPlan {
    static constexpr bool SX = MASK & SYNC_X, SU = MASK & SYNC_U;
    static constexpr bool SV = (MASK & SYNC_V) && OPT != OPT_SGDM;
    // does d_t depend on a state that is averaged?
    static constexpr bool D_NEEDS_MEAN = SU || (OPT == OPT_ADAM && SV);
    static constexpr bool KEEP_U = D_NEEDS_MEAN && !SU;                      // Adam, v synced only
    static constexpr bool KEEP_V = D_NEEDS_MEAN && OPT == OPT_ADAM && !SV;   // Adam, u synced only
};

// Workers per batch of the runtime-M kernel's update loops: what fits in `budget` registers -- 1, 2 or 4 (a power
// of two, so that a full batch can be summed as a tree).  Measured on B200 (134.5 M parameters x 16 workers, fraction of
// the copy bandwidth on all-sync steps): three blocks per SM with small batches 0.96; two blocks with batches twice as large
// 0.85; fp64 worker sums 0.87 and IEEE sqrt / division instead of the hardware reciprocal
// square root 0.87 (this kernel is bound by instruction issue: ~75 instructions per
// worker-coordinate with those, ~45 without).
constexpr int GEN_BUDGET = 24;      // registers a batch of workers may hold in flight
__host__ __device__ constexpr int gen_batch(int per_worker, int budget = GEN_BUDGET) {
    const int b = budget / per_worker;
    return b < 2 ? 1 : (b < 4 ? 2 : 4);
}
// Post-average ordering, more than eight workers: how many values enter the sums of the states, and of x, as one tree.
template <int OPT, int MASK, typename GT>
struct PostBatch {
    using P = PostPlan<OPT, MASK>;
    static constexpr int STATES = gen_batch(worker_regs<OPT, GT>(!P::D_NEEDS_MEAN, true, OPT != OPT_SGDM));
    static constexpr int PARAMS = gen_batch(4 + ((P::KEEP_U || P::KEEP_V) ? 4 : 0));   // where d_t needs a mean
    static constexpr int X = P::D_NEEDS_MEAN ? PARAMS : STATES;
};


// ---- where a tile lives -----------------------------------------------------------------------
// Position q of a thread covers VEC consecutive elements.  Both accessors expose the same four
// operations, so that one routine serves the staged tile and the straight-from-global fallback.
template <int OPT, int MT, typename GT, int T>
struct TileLayout {
    static constexpr int NS = OPT == OPT_SGDM ? 2 : 3;   // state arrays: x, u (, v)
    static constexpr int GB = T * static_cast<int>(sizeof(GT)), FB = T * 4;
    static constexpr int BYTES = MT * (GB + NS * FB);    // [g of every worker][x ...][u ...][v ...]
    __device__ static __forceinline__ int g_off(int m) { return m * GB; }
    __device__ static __forceinline__ int f_off(int arr, int m) { return MT * GB + (arr * MT + m) * FB; }
};

template <int OPT, int MT, typename GT, int T, int VEC_>
struct SmemAcc {
    static constexpr int VEC = VEC_;
    using L = TileLayout<OPT, MT, GT, T>;
    char *tile;
    __device__ __forceinline__ FV<VEC> ld(int arr, int m, int q) const {
        const char *p = tile + L::f_off(arr, m);
        FV<VEC> r;
        if constexpr (VEC == 4) {
            const float4 t = reinterpret_cast<const float4 *>(p)[q];
            r.a[0] = t.x; r.a[1] = t.y; r.a[2] = t.z; r.a[3] = t.w;
        } else if constexpr (VEC == 2) {
            const float2 t = reinterpret_cast<const float2 *>(p)[q];
            r.a[0] = t.x; r.a[1] = t.y;
        } else {
            r.a[0] = reinterpret_cast<const float *>(p)[q];
        }
        return r;
    }
    __device__ __forceinline__ void st(int arr, int m, int q, const FV<VEC> &r) const {
        char *p = tile + L::f_off(arr, m);
        if constexpr (VEC == 4)
            reinterpret_cast<float4 *>(p)[q] = make_float4(r.a[0], r.a[1], r.a[2], r.a[3]);
        else if constexpr (VEC == 2)
            reinterpret_cast<float2 *>(p)[q] = make_float2(r.a[0], r.a[1]);
        else
            reinterpret_cast<float *>(p)[q] = r.a[0];
    }
    __device__ __forceinline__ FV<VEC> ldg(int m, int q) const {
        const char *p = tile + L::g_off(m);
        FV<VEC> r;
        if constexpr (sizeof(GT) == 4) {
            if constexpr (VEC == 4) {
                const float4 t = reinterpret_cast<const float4 *>(p)[q];
                r.a[0] = t.x; r.a[1] = t.y; r.a[2] = t.z; r.a[3] = t.w;
            } else if constexpr (VEC == 2) {
                const float2 t = reinterpret_cast<const float2 *>(p)[q];
                r.a[0] = t.x; r.a[1] = t.y;
            } else {
                r.a[0] = reinterpret_cast<const float *>(p)[q];
            }
        } else if constexpr (VEC == 4) {   // bf16 -> fp32 is a 16-bit shift (exact)
            const uint2 t = reinterpret_cast<const uint2 *>(p)[q];
            r.a[0] = __uint_as_float(t.x << 16);
            r.a[1] = __uint_as_float(t.x & 0xffff0000u);
            r.a[2] = __uint_as_float(t.y << 16);
            r.a[3] = __uint_as_float(t.y & 0xffff0000u);
        } else if constexpr (VEC == 2) {
            const unsigned t = reinterpret_cast<const unsigned *>(p)[q];
            r.a[0] = __uint_as_float(t << 16);
            r.a[1] = __uint_as_float(t & 0xffff0000u);
        } else {
            r.a[0] = __uint_as_float(static_cast<unsigned>(reinterpret_cast<const unsigned short *>(p)[q]) << 16);
        }
        return r;
    }
};

// Straight from / to global memory, V coordinates per position with accesses that wide (bf16
// gradients: half): one (unaligned or ragged tiles), four -- chunks whose fp32 arrays are 16-byte aligned while
// the bf16 gradients are only 8-byte aligned, as in a flat layout padded to 16 bytes where the gradient of a
// tensor at an odd multiple of four elements sits 8 bytes off, and the aligned part of a ragged
// last tile -- or two, for the same chunks of more than eight workers (registers).
template <int MT, typename GT, int V>
struct GlobalAcc {
    static constexpr int VEC = V;
    char *const (*sp)[MT];   // chunk-relative base pointers: 0 x, 1 u, 2 v, 3 g
    __device__ __forceinline__ FV<V> ld(int arr, int m, int q) const { return ld_f32<V>(sp[arr][m], static_cast<long long>(V) * q); }
    __device__ __forceinline__ void st(int arr, int m, int q, const FV<V> &r) const { st_f32<V>(sp[arr][m], static_cast<long long>(V) * q, r); }
    __device__ __forceinline__ FV<V> ldg(int m, int q) const { return ld_grad<V, GT>(sp[3][m], static_cast<long long>(V) * q); }
};

// ---- diagnostics ------------------------------------------------------------------------------
// Each thread keeps its own running sums of squares, one per (kind, worker), in registers over
// all tiles of a chunk.  At the end of the chunk a warp reduces each of them (shuffle tree) into
// its slot of shared memory and the block total is the eight warp slots added in order:
// deterministic, and a few dozen shuffles per thread and chunk.
template <bool DIAG, int MT, int THREADS = BLOCK_THREADS>
struct ThreadNorms {
    float acc[DIAG ? DIAG_KINDS * MT : 1];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int j = 0; j < (DIAG ? DIAG_KINDS * MT : 1); ++j) acc[j] = 0.f;
    }
    __device__ __forceinline__ void add(int kind, int m, float v) {
        if constexpr (DIAG) acc[kind * MT + m] += v;
    }
    // all threads of the block call; slots: [DIAG_KINDS * MT][THREADS / 32]
    __device__ __forceinline__ void reduce_into(float *slots) const {
        if constexpr (DIAG) {
#pragma unroll
            for (int j = 0; j < DIAG_KINDS * MT; ++j) {
                float v = acc[j];
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
                if ((threadIdx.x & 31) == 0) slots[j * (THREADS / 32) + (threadIdx.x >> 5)] = v;
            }
        }
    }
};

template <int LO, int N, int VEC, int MT, bool P>
__device__ __forceinline__ FV<VEC> tree_sum_v(const FV<VEC> (&s)[MT]) {
    if constexpr (N == 1) {
        return s[LO];
    } else {
        constexpr int H = (N > 4) ? 4 : (N > 2 ? 2 : 1);   // as tree_sum
        return vadd<VEC, P>(tree_sum_v<LO, H, VEC, MT, P>(s), tree_sum_v<LO + H, N - H, VEC, MT, P>(s));
    }
}

template <int VEC, int MT, bool P, typename Acc>
__device__ __forceinline__ FV<VEC> mean_over_workers(const Acc &acc, int arr, int q) {
    FV<VEC> S[MT];
#pragma unroll
    for (int m = 0; m < MT; ++m) S[m] = acc.ld(arr, m, q);
    if constexpr (MT <= MAX_MT && (MT & (MT - 1)) == 0) {
        return vmul<VEC, P>(tree_sum_v<0, MT, VEC, MT, P>(S), splat<VEC>(1.f / MT));
    } else {
        FV<VEC> r;
#pragma unroll
        for (int c = 0; c < VEC; ++c) {
            float s[MT];
#pragma unroll
            for (int m = 0; m < MT; ++m) s[m] = S[m].a[c];
            r.a[c] = mean_of<MT>(s);
        }
        return r;
    }
}

// ---- one position (VEC coordinates) of all MT workers, in place --------------------------------
// Pre-average (Algorithms 1-3): the arrays to be averaged are first reduced to their worker
// means, then every worker updates from the mean or from its own previous value.
// Post-average (Algorithms 4-5): every worker updates its states, the ones to be averaged are
// replaced by their means, the parameter step uses those, and a synced x is averaged last.
// A thread re-reads values it stored itself (never another thread's), so no barrier is needed.
template <int OPT, int MASK, int MT, bool POST, bool DIAG, bool PLAIN = false, typename Acc, typename Norms>
__device__ __forceinline__ void update_position(const StepArgs &a, const Acc &acc, const float *sscale,
                                                int q, Norms &wn) {
    constexpr int VEC = Acc::VEC;
    constexpr bool SX = MASK & SYNC_X, SU = MASK & SYNC_U;
    constexpr bool SV = (MASK & SYNC_V) && OPT != OPT_SGDM;
    constexpr bool HAS_V = OPT != OPT_SGDM;
    if constexpr (!POST) {
        FV<VEC> xb{}, ub{}, vb{};
        if constexpr (SX) xb = mean_over_workers<VEC, MT, OPT != OPT_SGDM>(acc, 0, q);
        if constexpr (SU) ub = mean_over_workers<VEC, MT, OPT != OPT_SGDM>(acc, 1, q);
        if constexpr (SV) vb = mean_over_workers<VEC, MT, OPT != OPT_SGDM>(acc, 2, q);
        constexpr bool NEED_V = HAS_V && (!SV || OPT == OPT_ADOPT);   // ADOPT: its own old v
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            const FV<VEC> G = acc.ldg(m, q);
            FV<VEC> X{}, U{}, V{}, un, vn;
            if constexpr (!SX) X = acc.ld(0, m, q);
            if constexpr (!SU) U = acc.ld(1, m, q);
            if constexpr (NEED_V) V = acc.ld(2, m, q);
            state_update<OPT, PLAIN, VEC>(a, G, PLAIN ? 1.f : sscale[m], SU ? ub : U, SV ? vb : V, V, un, vn);
            const FV<VEC> D = minus_direction<OPT, PLAIN, VEC>(a, un, vn);
            X = apply_step<VEC, OPT != OPT_SGDM>(a, SX ? xb : X, D);
            acc.st(0, m, q, X);
            acc.st(1, m, q, un);
            if constexpr (HAS_V) acc.st(2, m, q, vn);
            if constexpr (DIAG) {
                wn.add(DIAG_G, m, sum_sq<VEC>(G));
                wn.add(DIAG_D, m, sum_sq<VEC>(D));
                wn.add(DIAG_X, m, sum_sq<VEC>(X));
            }
        }
    } else {
        // states
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            const FV<VEC> G = acc.ldg(m, q);
            FV<VEC> U = acc.ld(1, m, q), V{}, un, vn;
            if constexpr (HAS_V) V = acc.ld(2, m, q);
            state_update<OPT, PLAIN, VEC>(a, G, PLAIN ? 1.f : sscale[m], U, V, V, un, vn);
            acc.st(1, m, q, un);
            if constexpr (HAS_V) acc.st(2, m, q, vn);
            if constexpr (DIAG) wn.add(DIAG_G, m, sum_sq<VEC>(G));
        }
        FV<VEC> mu{}, mv{};
        if constexpr (SU) mu = mean_over_workers<VEC, MT, OPT != OPT_SGDM>(acc, 1, q);
        if constexpr (SV) mv = mean_over_workers<VEC, MT, OPT != OPT_SGDM>(acc, 2, q);
        // parameters
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            FV<VEC> X = acc.ld(0, m, q), U = mu, V = mv;
            if constexpr (!SU) U = acc.ld(1, m, q);
            if constexpr (OPT == OPT_ADAM && !SV) V = acc.ld(2, m, q);
            const FV<VEC> D = minus_direction<OPT, PLAIN, VEC>(a, U, V);
            X = apply_step<VEC, OPT != OPT_SGDM>(a, X, D);
            acc.st(0, m, q, X);
            if constexpr (SU) acc.st(1, m, q, mu);
            if constexpr (SV) acc.st(2, m, q, mv);
            if constexpr (DIAG) wn.add(DIAG_D, m, sum_sq<VEC>(D));
            if constexpr (DIAG && !SX) wn.add(DIAG_X, m, sum_sq<VEC>(X));
        }
        if constexpr (SX) {
            const FV<VEC> mx = mean_over_workers<VEC, MT, OPT != OPT_SGDM>(acc, 0, q);
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                acc.st(0, m, q, mx);
                if constexpr (DIAG) wn.add(DIAG_X, m, sum_sq<VEC>(mx));
            }
        }
    }
}

// ---- bulk asynchronous copies and their barrier ----------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// global -> shared, completion counted in bytes on `bar`.  Both addresses 16-byte aligned and
// `bytes` a multiple of 16 (checked by the caller: anything else takes the fallback path).
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
// shared -> global, tracked by the issuing thread's bulk group
__device__ __forceinline__ void bulk_store(void *dst, const void *src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                 :: "l"(dst), "r"(smem_u32(src)), "r"(bytes) : "memory");
}
// Waits for the phase with the given parity, polling at most `limit` times; false when the limit
// ran out.  No wait in this library is unbounded.
__device__ __forceinline__ bool bar_wait(uint64_t *bar, uint32_t parity, int limit) {
    for (int i = 0; i < limit; ++i) {
        uint32_t ok;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}

// Threads, tile buffers and resident blocks per SM.  Three and more replicas of a tile: two buffers
// of 21-57 KB and 256 threads (one per element beyond eight replicas), as many blocks as the buffers leave room for,
// four at most (three buffers at two blocks per SM: 0.84 of the copy bandwidth).  One
// replica: up to three buffers of 7 KB (bf16 gradients; 5 KB without v) and 128 threads, one float4 of
// each array per thread and tile, ten blocks.
__host__ __device__ constexpr int step_threads(int opt, int mt, bool bf16) {
    return mt <= 2 ? 128 : mt <= MAX_MT ? BLOCK_THREADS : tile_elems(opt, mt, bf16);
}
__host__ __device__ constexpr int step_stages(int mt) { return mt == 1 ? 3 : 2; }
__host__ __device__ constexpr int step_min_blocks(int opt, int mt, bool bf16) {
    if (mt <= 2) return mt == 1 ? 10 : 7;
    const int room = 225 * 1024 / (2 * tile_elems(opt, mt, bf16) * tile_bytes_per_elem(opt, mt, bf16) + 1024);
    return room < 2 ? 2 : room > 4 ? 4 : room;
}

// A chunk is a run of consecutive tiles of one tensor.  The block looks its pointers up
// once, then streams the tiles through a ring of S buffers: while tile k is updated in
// place, tiles k + 1 .. k + S - 1 are already landing; when tile k's copy back has left its
// buffer, tile k + S is requested into it.
template <int OPT, int MASK, int MT, typename GT, bool POST, bool DIAG>
__global__ void __launch_bounds__(step_threads(OPT, MT, sizeof(GT) == 2), step_min_blocks(OPT, MT, sizeof(GT) == 2))
desloc_step_kernel(const __grid_constant__ StepArgs a) {
    constexpr int THREADS = step_threads(OPT, MT, sizeof(GT) == 2);
    constexpr int T = tile_elems(OPT, MT, sizeof(GT) == 2), VEC = T / THREADS, S = step_stages(MT);
    constexpr int ALIGN_ELEMS = 16 / static_cast<int>(sizeof(GT));   // bulk copies move multiples of 16 bytes
    constexpr bool HAS_V = OPT != OPT_SGDM;
    using L = TileLayout<OPT, MT, GT, T>;
    static_assert(4 * MT <= THREADS && T % THREADS == 0, "a thread per (array, worker); whole tiles");
    extern __shared__ __align__(128) char tile_mem[];   // S buffers of L::BYTES
    __shared__ char *sp[4][MT];
    __shared__ float sscale[MT];
    __shared__ unsigned misfit;
    __shared__ __align__(8) uint64_t bar[S];
    ThreadNorms<DIAG, MT, THREADS> wn;
    const int tid = threadIdx.x;
    begin_and_let_next_begin();
    if (tid < S) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&bar[tid])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // this thread's role in the look-up, the loads and the stores: one (array, worker)
    const int arr = tid / MT, m = tid - arr * MT;
    const bool owner = tid < 4 * MT && (HAS_V || arr != 2);
    const int esize = arr == 3 ? static_cast<int>(sizeof(GT)) : 4;
    const int slot = arr == 3 ? L::g_off(m) : L::f_off(arr, m);
    uint32_t phases = 0;  // bit s: parity of the phase barrier s completes next
    // No factor on the gradient, no coordinate clip and an epsilon whose square is a normal number -- the
    // common case -- take a copy of the inner loop without the instructions for these.  The fallback paths
    // keep the one form.
    const bool plain = plain_step<OPT>(a);
    // Work items: parts of a chunk, of all MT replicas or (MT = 1: a single worker, local steps) of
    // replica blockIdx.y.  One item per block as launched (fewer than 2^31); a smaller grid
    // strides over the rest.
    const int m0 = MT == 1 ? static_cast<int>(blockIdx.y) : 0;
    const long long nitems = a.nchunks * a.parts;
    for (long long item = blockIdx.x; item < nitems; item += gridDim.x) {
        const unsigned c = item_chunk(a, static_cast<unsigned>(item));
        const int part0 = static_cast<int>(static_cast<unsigned>(item) - c * a.parts) * a.part_elems;
        const Chunk ch = a.chunks[c];   // the same 16 bytes for every thread
        const int count = min(ch.count - part0, a.part_elems);
        const long long start = ch.start + part0;
        if (count <= 0) continue;   // a short chunk has fewer parts
        // the previous item is done with the shared state
        if (item != blockIdx.x) __syncthreads();
        char *p = nullptr;
        if (owner) {
            const long long idx = static_cast<long long>(m0 + m) * a.nt + ch.tensor;
            if (arr == 0) p = reinterpret_cast<char *>(a.x[idx]) + start * 4;
            if (arr == 1) p = reinterpret_cast<char *>(a.u[idx]) + start * 4;
            if (arr == 2) p = reinterpret_cast<char *>(a.v[idx]) + start * 4;
            if (arr == 3)
                p = const_cast<char *>(reinterpret_cast<const char *>(grad_ptr(a, idx))) +
                    start * static_cast<long long>(sizeof(GT));
            sp[arr][m] = p;
        }
        wn.clear();
        // Bulk copies need 16-byte aligned addresses (bit 0); 128-bit accesses from global memory less: 8
        // bytes for bf16 gradients (bit 1).
        const uintptr_t need = (arr == 3 && sizeof(GT) == 2) ? 7u : 15u;
        unsigned off = ((reinterpret_cast<uintptr_t>(p) & 15u) != 0 ? 1u : 0u) |
                       ((reinterpret_cast<uintptr_t>(p) & need) != 0 ? 2u : 0u);
        if constexpr (4 * MT <= 32) {
            // all owners are lanes of the first warp: one reduction there, one barrier for the block
            if (tid < 32) {
                off = __reduce_or_sync(0xffffffffu, off);
                if (tid == 0) misfit = off;
            }
            __syncthreads();   // (the barriers exist, too)
            off = misfit;
        } else {
            const int any1 = __syncthreads_or(off & 1u), any2 = __syncthreads_or(off & 2u);
            off = (any1 ? 1u : 0u) | (any2 ? 2u : 0u);
        }
        // (a tile needs a byte count that is a multiple of 16, too: only a chunk's last tile can miss that, and
        // is then updated straight from global memory, like every tile of a chunk whose pointers are unaligned)
        const bool unaligned = (off & 1u) != 0, wide_ok = (off & 2u) == 0;
        const int ntiles = (count + T - 1) / T;
        // (a launch of a single wave of single-tile chunks has nothing to overlap: staging would
        // only add the copy engine's round trip to every step of a latency-bound problem)
        const int staged = (unaligned || a.direct) ? 0 : ((count % T) % ALIGN_ELEMS == 0 ? ntiles : ntiles - 1);   // tiles 0 .. staged-1
        // request tile k (< staged) into its buffer: every owner its own slice, one arrival
        auto request = [&](int k) {
            const int cnt = min(T, count - k * T);
            if (owner)
                bulk_load(tile_mem + (k % S) * L::BYTES + slot, p + static_cast<long long>(k) * T * esize,
                          static_cast<uint32_t>(cnt * esize), &bar[k % S]);
            if (tid == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                             :: "r"(smem_u32(&bar[k % S])),
                                "r"(static_cast<uint32_t>(MT * cnt * (static_cast<int>(sizeof(GT)) + 4 * L::NS)))
                             : "memory");
        };
        wait_for_earlier_kernels();
#pragma unroll
        for (int k = 0; k < S; ++k)
            if (k < staged) request(k);
        // (behind the requests: its latency hides in theirs)
        if (tid < MT) sscale[tid] = a.gscale ? a.gscale[m0 + tid] : 1.f;
        if (!plain || staged < ntiles) __syncthreads();
#pragma unroll 1
        for (int k = 0; k < staged; ++k) {
            const int st = k % S;
            const int cnt = min(T, count - k * T);
            // Every thread waits for the tile itself and touches its own coordinates only, so one barrier
            // per tile is enough: behind the updates, in front of the copies back.
            const bool landed = bar_wait(&bar[st], (phases >> st) & 1u, a.wait_limit);
            const SmemAcc<OPT, MT, GT, T, VEC> acc{tile_mem + st * L::BYTES};
            if (landed && tid * VEC < cnt) {
                if (plain) update_position<OPT, MASK, MT, POST, DIAG, true>(a, acc, sscale, tid, wn);
                else update_position<OPT, MASK, MT, POST, DIAG, false>(a, acc, sscale, tid, wn);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // our writes, then the copy engine's reads
            if (__syncthreads_or(!landed)) {
                // Give up on this step: say so, let the copies already requested land (bounded as
                // well), store nothing more, leave.  The host reports the flag on its next call.
                if (tid == 0 && a.err) *reinterpret_cast<volatile int *>(a.err) = 1;
                for (int kk = k; kk < staged && kk < k + S; ++kk)
                    bar_wait(&bar[kk % S], (phases >> (kk % S)) & 1u, DRAIN_WAIT_LIMIT);
                asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
                __syncthreads();
                return;
            }
            phases ^= 1u << st;
            if (owner && arr != 3) {
                bulk_store(p + static_cast<long long>(k) * T * 4, tile_mem + st * L::BYTES + slot,
                           static_cast<uint32_t>(cnt * 4));
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
            if ((MT != 1 || DIAG) && k + S < staged) {   // (one replica: a buffer for every tile)
                // the buffer is free once this thread's own copy back has read it
                if (owner && arr != 3) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                request(k + S);
            }
        }
        if (staged * T < count) {
            // what could not be staged: the whole chunk, or its ragged last tile
            int e0 = staged * T;
            if (wide_ok) {
                constexpr int V = MT <= MAX_MT ? 4 : 2;
                const GlobalAcc<MT, GT, V> wide{sp};
                const int p1 = count / V;
                for (int q = e0 / V + tid; q < p1; q += THREADS)
                    update_position<OPT, MASK, MT, POST, DIAG>(a, wide, sscale, q, wn);
                e0 = p1 * V;
            }
            const GlobalAcc<MT, GT, 1> acc{sp};
            for (int e = e0 + tid; e < count; e += THREADS)
                update_position<OPT, MASK, MT, POST, DIAG>(a, acc, sscale, e, wn);
        }
        // the copies back must have left shared memory before the buffers are reused or freed
        if (owner && arr != 3) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        if constexpr (DIAG) {
            // the tile buffers are idle now: their first bytes serve as the warps' slots
            float *slots = reinterpret_cast<float *>(tile_mem);
            __syncthreads();
            wn.reduce_into(slots);
            __syncthreads();
            if (tid < DIAG_KINDS * MT) {
                float total = 0.f;
#pragma unroll
                for (int w = 0; w < THREADS / 32; ++w) total += slots[tid * (THREADS / 32) + w];
                const int kind = tid / MT, mm = tid - kind * MT;
                a.diag[(static_cast<long long>(kind) * a.M + m0 + mm) * a.diag_stride + c] = total;
                if (tid == 0 && m0 == 0 && c == 0) *a.diag_parts = 1;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before the copy engine writes there again
        }
    }
}

// Dynamic shared memory a launch of desloc_step_kernel<opt, ., mt, grad type, ., .> needs whose
// blocks take up to part_elems elements: a buffer per tile, at most step_stages(mt) of them.
__host__ __device__ constexpr int step_smem_bytes(int opt, int mt, bool bf16, int part_elems) {
    const int t = tile_elems(opt, mt, bf16), tiles = (part_elems + t - 1) / t;
    return (tiles < step_stages(mt) ? tiles : step_stages(mt)) * mt * t * ((bf16 ? 2 : 4) + 4 * (opt == OPT_SGDM ? 2 : 3));
}

// Lookup of an instantiation: opt, post-average?, bf16 gradients?, MT in 1..MAX_MT (pre-average and
// without norms: 1..MAX_TILE_MT), mask,
// with or without the norm diagnostics (MT = 1 exists for mask 0 only, and mask 0 for MT = 1).
// Returns nullptr for combinations that do not exist.
const void *lookup_step_kernel(int opt, bool post, bool bf16, int mt, int mask, bool diag);

// Runtime-M kernel for the sync steps of M > MAX_MT that have no tile kernel.
const void *lookup_generic_kernel(int opt, bool post, bool bf16, int mask, bool diag);

}  // namespace desloc
