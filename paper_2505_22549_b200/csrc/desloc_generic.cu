// DES-LOC step for the worker counts and variants that have no tile kernel (M > 16; from nine workers on also
// the post-average ordering and the norm diagnostics) on steps that average something in problems too large for desloc_crowd_kernel.  Same update
// as desloc_step_kernel, runtime M, compile-time mask.  Worker sums run in the order m = 0..M-1 as
// compensated fp32 sums (see WorkerSum): exact for equal replicas, and within an ulp of a
// sequential fp64 reference.
//
// A block takes one chunk and first puts the chunk-relative pointers of all M workers into
// shared memory, so that the per-position loops read them as broadcasts instead of chasing the
// pointer tables in global memory.  Per position (4 elements per thread):
//   pre-average   the arrays to be averaged are summed in one pass, two or four workers' loads in
//                 flight; then the workers are updated in batches sized to the
//                 register budget, loading only what was not averaged (ADOPT also its own v).
//                 Each array is read once and written once.
//   post-average  phase A updates the states batch by batch, sums the ones to be averaged and
//                 stores the others; the parameter step runs in phase A when d_t uses only the
//                 worker's own states, otherwise in phase B once the means are known.  Only
//                 when Adam averages exactly one of u, v does phase B re-read the other one
//                 (just written, so it is served from cache).
#include "desloc_kernels.cuh"

namespace desloc {

namespace {

constexpr int GEN_MAX_M = 256;    // worker pointers staged per chunk (= the context's limit)
template <int N>
struct Count {
    static constexpr int value = N;
};

// Calls batch(Count<N>, m0, n) for all M workers in order: n <= N workers from m0 on.  WHOLE: every n is its
// batch's N (the last workers by halves), known to the compiler, else only the last n is less.  The kernels with
// norms are faster the first way (their shuffles keep the loads of a batch together), the others the second.
template <int B, bool WHOLE, typename F>
__device__ __forceinline__ void for_batches(int M, const F &batch) {
    if constexpr (WHOLE) {
        int m0 = 0;
#pragma unroll 1
        for (; m0 + B <= M; m0 += B) batch(Count<B>{}, m0, B);
        if constexpr (B > 2) {
            if (m0 + 2 <= M) {
                batch(Count<2>{}, m0, 2);
                m0 += 2;
            }
        }
        if constexpr (B > 1) {
            if (m0 < M) batch(Count<1>{}, m0, 1);
        }
    } else {
#pragma unroll 1
        for (int m0 = 0; m0 < M; m0 += B) batch(Count<B>{}, m0, M - m0);
    }
}

// Sum of N workers' values as a binary tree.
template <int VEC, int N>
__device__ __forceinline__ FV<VEC> sum_of(const FV<VEC> (&v)[N]) {
    FV<VEC> t;
#pragma unroll
    for (int c = 0; c < VEC; ++c) {
        float q[N];
#pragma unroll
        for (int j = 0; j < N; ++j) q[j] = v[j].a[c];
        t.a[c] = tree_sum<0, N, N>(q);
    }
    return t;
}

// Sum over the workers of one coordinate group, in the order m = 0..M-1, as a compensated fp32
// sum ("two-sum"): the running sum and the exact rounding error of every addition are both
// kept, so the pair carries about 48 bits -- the accuracy of an fp64 sum without the fp64 pipe,
// which made an all-sync step 10 % slower here.  The mean divides the pair by M with one
// correction step, and is exact (the value itself) when all M replicas are equal.
template <int VEC>
struct WorkerSum {
    float s[VEC], err[VEC];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int c = 0; c < VEC; ++c) s[c] = err[c] = 0.f;
    }
    __device__ __forceinline__ void add(const FV<VEC> &v) {
#pragma unroll
        for (int c = 0; c < VEC; ++c) {
            const float x = v.a[c];
            const float t = s[c] + x;
            const float bp = t - s[c];
            err[c] += (s[c] - (t - bp)) + (x - bp);  // exact error of t = s + x
            s[c] = t;
        }
    }
    __device__ __forceinline__ FV<VEC> mean(int M) const {
        const float mf = static_cast<float>(M), inv = 1.f / mf;
        FV<VEC> r;
#pragma unroll
        for (int c = 0; c < VEC; ++c) {
            const float hi = s[c] + err[c];
            const float lo = err[c] - (hi - s[c]);          // hi + lo = s + err
            r.a[c] = div_by_count(hi, lo, mf, inv);
        }
        return r;
    }
    // The first n of N consecutive workers, in batches of B (a power of two).  A full batch is summed as a binary tree
    // first (exact when its values are equal) and enters the running sum as one value; a shorter one enters
    // value by value.
    template <int B, int N>
    __device__ __forceinline__ void add_batch(const FV<VEC> (&v)[N], int n) {
        static_assert((B & (B - 1)) == 0 && N <= B, "batches are powers of two");
        if (N == B && n >= B) {
            add(sum_of<VEC, N>(v));
        } else {
#pragma unroll
            for (int j = 0; j < N; ++j)
                if (j < n) add(v[j]);
        }
    }
};

// Worker means of the arrays selected by SX, SU, SV in one pass over the workers: trees of four
// workers enter the compensated sums in order, the last one to three workers value by value (the order
// of compensated_mean(), so that a step with norm diagnostics gives the bits of one without).  The
// loads of four workers are issued together for one array, of two for two or three.
template <int VEC, bool SX, bool SU, bool SV>
__device__ __forceinline__ void means_of_workers(char *const (*sp)[GEN_MAX_M], int M, long long e,
                                                 bool active, FV<VEC> &xb, FV<VEC> &ub, FV<VEC> &vb) {
    if constexpr ((SX ? 1 : 0) + (SU ? 1 : 0) + (SV ? 1 : 0) == 1) {
        // One array: the last batch in the same loop as the full ones.  (A loop of full batches and one of
        // single workers behind it was up to 15 % slower at 100 M parameters x workers, all counts and types.)
        constexpr int ARR = SX ? 0 : SU ? 1 : 2;
        WorkerSum<VEC> sum;
        sum.clear();
#pragma unroll 1
        for (int m0 = 0; m0 < M; m0 += 4) {
            FV<VEC> v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (active && m0 + j < M) v[j] = ld_f32<VEC>(sp[ARR][m0 + j], e);
            if (active) sum.template add_batch<4, 4>(v, M - m0);
        }
        (SX ? xb : SU ? ub : vb) = sum.mean(M);
    } else {
        WorkerSum<VEC> ax, au, av;
        ax.clear(); au.clear(); av.clear();
        int m0 = 0;
#pragma unroll 1
        for (; m0 + 4 <= M; m0 += 4) {
            FV<VEC> px[2], pu[2], pv[2];   // sums of two workers
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                FV<VEC> bx[2], bu[2], bv[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    if (active) {
                        if constexpr (SX) bx[j] = ld_f32<VEC>(sp[0][m0 + h * 2 + j], e);
                        if constexpr (SU) bu[j] = ld_f32<VEC>(sp[1][m0 + h * 2 + j], e);
                        if constexpr (SV) bv[j] = ld_f32<VEC>(sp[2][m0 + h * 2 + j], e);
                    }
                }
                if (active) {
                    if constexpr (SX) px[h] = sum_of<VEC, 2>(bx);
                    if constexpr (SU) pu[h] = sum_of<VEC, 2>(bu);
                    if constexpr (SV) pv[h] = sum_of<VEC, 2>(bv);
                }
            }
            if (active) {
                if constexpr (SX) ax.add(sum_of<VEC, 2>(px));
                if constexpr (SU) au.add(sum_of<VEC, 2>(pu));
                if constexpr (SV) av.add(sum_of<VEC, 2>(pv));
            }
        }
#pragma unroll 1
        for (; m0 < M; ++m0) {
            if (active) {
                FV<VEC> bx, bu, bv;
                if constexpr (SX) bx = ld_f32<VEC>(sp[0][m0], e);
                if constexpr (SU) bu = ld_f32<VEC>(sp[1][m0], e);
                if constexpr (SV) bv = ld_f32<VEC>(sp[2][m0], e);
                if constexpr (SX) ax.add(bx);
                if constexpr (SU) au.add(bu);
                if constexpr (SV) av.add(bv);
            }
        }
        if constexpr (SX) xb = ax.mean(M);
        if constexpr (SU) ub = au.mean(M);
        if constexpr (SV) vb = av.mean(M);
    }
}

// Diagnostics with a runtime worker count: a warp reduces each (kind, worker) value at once
// and lane 0 adds it to the warp's own row of shared memory, in position order.
template <bool DIAG>
struct WarpDiag {
    float *rows;  // [BLOCK_THREADS / 32][DIAG_KINDS][GEN_MAX_M]
    __device__ __forceinline__ void add(int kind, int m, float v) const {
        if constexpr (DIAG) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
            if ((threadIdx.x & 31) == 0)
                rows[((threadIdx.x >> 5) * DIAG_KINDS + kind) * GEN_MAX_M + m] += v;
        }
    }
    // the same value for every worker (a synced x): one reduction, M additions by lane 0
    __device__ __forceinline__ void add_all(int kind, int M, float v) const {
        if constexpr (DIAG) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
            if ((threadIdx.x & 31) == 0) {
                float *row = rows + ((threadIdx.x >> 5) * DIAG_KINDS + kind) * GEN_MAX_M;
                for (int m = 0; m < M; ++m) row[m] += v;
            }
        }
    }
};

// One position (VEC elements) of all M workers.  `active` is false for the lanes a DIAG warp
// carries past the end of the chunk: they touch no memory and contribute zeros to the sums.
template <int OPT, typename GT, bool POST, int MASK, int VEC, bool DIAG, bool PLAIN = false>
__device__ __forceinline__ void generic_position(const StepArgs &a, char *const (*sp)[GEN_MAX_M],
                                                 const float *sscale, long long e, bool active,
                                                 const WarpDiag<DIAG> &wd) {
    const int M = a.M;
    constexpr bool SX = MASK & SYNC_X, SU = MASK & SYNC_U;
    constexpr bool SV = (OPT != OPT_SGDM) && (MASK & SYNC_V);
    if constexpr (!POST) {
        FV<VEC> xb{}, ub{}, vb{};
        means_of_workers<VEC, SX, SU, SV>(sp, M, e, active, xb, ub, vb);
        constexpr bool NEED_V = OPT != OPT_SGDM && (!SV || OPT == OPT_ADOPT);
        constexpr int B0 = gen_batch(worker_regs<OPT, GT>(!SX, !SU, NEED_V));
        constexpr int B = (OPT == OPT_ADOPT && B0 > 2) ? 2 : B0;  // ADOPT's normaliser needs more registers
        for_batches<B, DIAG>(M, [&](auto count, int m0, int n) {
            constexpr int N = decltype(count)::value;
            FV<VEC> G[N], X[N], U[N], V[N];
#pragma unroll
            for (int b = 0; b < N; ++b) {
                if (active && b < n) {
                    G[b] = ld_grad<VEC, GT>(sp[3][m0 + b], e);
                    if constexpr (!SX) X[b] = ld_f32<VEC>(sp[0][m0 + b], e);
                    if constexpr (!SU) U[b] = ld_f32<VEC>(sp[1][m0 + b], e);
                    if constexpr (NEED_V) V[b] = ld_f32<VEC>(sp[2][m0 + b], e);
                }
            }
#pragma unroll
            for (int b = 0; b < N; ++b) {
                if (b < n) {
                    float gg = 0.f, dd = 0.f, xx = 0.f;
                    if (active) {
                        gg = sum_sq<VEC>(G[b]);
                        FV<VEC> vown{}, un, vn;
                        if constexpr (NEED_V) vown = V[b];
                        state_update<OPT, PLAIN, VEC, false>(a, G[b], PLAIN ? 1.f : sscale[m0 + b], SU ? ub : U[b],
                                                      SV ? vb : vown, vown, un, vn);
                        const FV<VEC> D = minus_direction<OPT, PLAIN, VEC, false>(a, un, vn);
                        X[b] = apply_step<VEC, false>(a, SX ? xb : X[b], D);
                        U[b] = un;
                        V[b] = vn;
                        dd = sum_sq<VEC>(D);
                        xx = sum_sq<VEC>(X[b]);
                        st_f32<VEC>(sp[0][m0 + b], e, X[b]);
                        st_f32<VEC>(sp[1][m0 + b], e, U[b]);
                        if constexpr (OPT != OPT_SGDM) st_f32<VEC>(sp[2][m0 + b], e, V[b]);
                    }
                    wd.add(DIAG_G, m0 + b, gg);
                    wd.add(DIAG_D, m0 + b, dd);
                    wd.add(DIAG_X, m0 + b, xx);
                }
            }
        });
    } else {
        using P = PostPlan<OPT, MASK>;
        WorkerSum<VEC> au, av, ax;
        au.clear(); av.clear(); ax.clear();
        constexpr int BA = PostBatch<OPT, MASK, GT>::STATES;
        // phase A: states (and x where d_t needs no mean)
        for_batches<BA, DIAG>(M, [&](auto count, int m0, int n) {
            constexpr int N = decltype(count)::value;
            FV<VEC> G[N], U[N], V[N], X[N];
#pragma unroll
            for (int b = 0; b < N; ++b) {
                if (active && b < n) {
                    G[b] = ld_grad<VEC, GT>(sp[3][m0 + b], e);
                    U[b] = ld_f32<VEC>(sp[1][m0 + b], e);
                    if constexpr (OPT != OPT_SGDM) V[b] = ld_f32<VEC>(sp[2][m0 + b], e);
                    if constexpr (!P::D_NEEDS_MEAN) X[b] = ld_f32<VEC>(sp[0][m0 + b], e);
                }
            }
#pragma unroll
            for (int b = 0; b < N; ++b) {
                if (b < n) {
                    float gg = 0.f, dd = 0.f, xx = 0.f;
                    if (active) {
                        gg = sum_sq<VEC>(G[b]);
                        FV<VEC> vown{}, un, vn, D;
                        if constexpr (OPT != OPT_SGDM) vown = V[b];
                        state_update<OPT, PLAIN, VEC, false>(a, G[b], PLAIN ? 1.f : sscale[m0 + b], U[b], vown, vown, un, vn);
                        U[b] = un;
                        V[b] = vn;
                        if constexpr (!P::D_NEEDS_MEAN) {
                            D = minus_direction<OPT, PLAIN, VEC, false>(a, un, vn);
                            X[b] = apply_step<VEC, false>(a, X[b], D);
                        }
                        // a state that is not averaged has its final value now (phase B re-reads
                        // it where Adam needs it per worker)
                        if constexpr (!P::SU) st_f32<VEC>(sp[1][m0 + b], e, U[b]);
                        if constexpr (OPT != OPT_SGDM && !P::SV) st_f32<VEC>(sp[2][m0 + b], e, V[b]);
                        if constexpr (!P::D_NEEDS_MEAN) {
                            dd = sum_sq<VEC>(D);
                            if constexpr (!P::SX) {
                                xx = sum_sq<VEC>(X[b]);
                                st_f32<VEC>(sp[0][m0 + b], e, X[b]);
                            }
                        }
                    }
                    wd.add(DIAG_G, m0 + b, gg);
                    if constexpr (!P::D_NEEDS_MEAN) {
                        wd.add(DIAG_D, m0 + b, dd);
                        if constexpr (!P::SX) wd.add(DIAG_X, m0 + b, xx);
                    }
                }
            }
            if (active) {
                if constexpr (P::SU) au.template add_batch<BA, N>(U, n);
                if constexpr (P::SV) av.template add_batch<BA, N>(V, n);
                if constexpr (P::SX && !P::D_NEEDS_MEAN) ax.template add_batch<BA, N>(X, n);
            }
        });
        const FV<VEC> mu = au.mean(M), mv = av.mean(M);
        if constexpr (P::D_NEEDS_MEAN) {
            // phase B: parameter step with the averaged states
            constexpr int BB = PostBatch<OPT, MASK, GT>::PARAMS;
            for_batches<BB, DIAG>(M, [&](auto count, int m0, int n) {
                constexpr int N = decltype(count)::value;
                FV<VEC> X[N], K[N];
#pragma unroll
                for (int b = 0; b < N; ++b) {
                    if (active && b < n) {
                        X[b] = ld_f32<VEC>(sp[0][m0 + b], e);
                        if constexpr (P::KEEP_U) K[b] = ld_f32<VEC>(sp[1][m0 + b], e);
                        if constexpr (P::KEEP_V) K[b] = ld_f32<VEC>(sp[2][m0 + b], e);
                    }
                }
#pragma unroll
                for (int b = 0; b < N; ++b) {
                    if (b < n) {
                        float dd = 0.f, xx = 0.f;
                        if (active) {
                            FV<VEC> vn{};
                            if constexpr (P::SV) vn = mv;
                            else if constexpr (P::KEEP_V) vn = K[b];
                            const FV<VEC> D = minus_direction<OPT, PLAIN, VEC, false>(a, P::SU ? mu : K[b], vn);
                            X[b] = apply_step<VEC, false>(a, X[b], D);
                            dd = sum_sq<VEC>(D);
                            if constexpr (!P::SX) {
                                xx = sum_sq<VEC>(X[b]);
                                st_f32<VEC>(sp[0][m0 + b], e, X[b]);
                            }
                            if constexpr (P::SU) st_f32<VEC>(sp[1][m0 + b], e, mu);
                            if constexpr (P::SV) st_f32<VEC>(sp[2][m0 + b], e, mv);
                        }
                        wd.add(DIAG_D, m0 + b, dd);
                        if constexpr (!P::SX) wd.add(DIAG_X, m0 + b, xx);
                    }
                }
                if constexpr (P::SX) {
                    if (active) ax.template add_batch<BB, N>(X, n);
                }
            });
        }
        if constexpr (P::SX || (!P::D_NEEDS_MEAN && P::SV)) {
            const FV<VEC> mx = ax.mean(M);
            const float xx = (P::SX && active) ? sum_sq<VEC>(mx) : 0.f;
            if (active) {
#pragma unroll 1
                for (int m = 0; m < M; ++m) {
                    if constexpr (P::SX) st_f32<VEC>(sp[0][m], e, mx);
                    if constexpr (!P::D_NEEDS_MEAN && P::SV) st_f32<VEC>(sp[2][m], e, mv);
                }
            }
            if constexpr (P::SX) wd.add_all(DIAG_X, M, xx);
        }
    }
}

template <int OPT, typename GT, bool POST, int MASK, bool DIAG>
__global__ void __launch_bounds__(BLOCK_THREADS, GENERIC_MIN_BLOCKS)
desloc_step_generic_kernel(const __grid_constant__ StepArgs a) {
    __shared__ char *sp[4][GEN_MAX_M];
    __shared__ float sscale[GEN_MAX_M];
    __shared__ float srows[DIAG ? (BLOCK_THREADS / 32) * DIAG_KINDS * GEN_MAX_M : 1];
    const WarpDiag<DIAG> wd{srows};
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    // exactly one chunk per block (this kernel does not stride: with a chunk loop around the
    // same body the compiler needs spill slots)
    const long long c = blockIdx.x;
    if (c < a.nchunks) {
        const Chunk ch = a.chunks[c];
        int mis = 0;
        for (int m = tid; m < a.M; m += BLOCK_THREADS) {
            const long long idx = static_cast<long long>(m) * a.nt + ch.tensor;
            char *px = reinterpret_cast<char *>(a.x[idx]) + ch.start * 4;
            char *pu = reinterpret_cast<char *>(a.u[idx]) + ch.start * 4;
            char *pv = (OPT != OPT_SGDM) ? reinterpret_cast<char *>(a.v[idx]) + ch.start * 4 : nullptr;
            char *pg = const_cast<char *>(reinterpret_cast<const char *>(grad_ptr(a, idx))) +
                       ch.start * static_cast<long long>(sizeof(GT));
            sp[0][m] = px; sp[1][m] = pu; sp[2][m] = pv; sp[3][m] = pg;
            sscale[m] = a.gscale ? a.gscale[m] : 1.f;
            mis |= (reinterpret_cast<uintptr_t>(px) | reinterpret_cast<uintptr_t>(pu) |
                    reinterpret_cast<uintptr_t>(pv)) & 15u;
            mis |= reinterpret_cast<uintptr_t>(pg) & (sizeof(GT) == 2 ? 7u : 15u);
        }
        if constexpr (DIAG) {
            for (int j = tid; j < (BLOCK_THREADS / 32) * DIAG_KINDS * GEN_MAX_M; j += BLOCK_THREADS)
                srows[j] = 0.f;
        }
        const bool scalar_path = __syncthreads_or(mis) != 0;
        // DIAG warps run whole: lanes past the end take part in the shuffles with zeros
        if (!scalar_path) {
            const int n4 = ch.count >> 2;
            // (no gradient factor and no coordinate clip, the common case: a copy of the loop
            // without them -- this kernel is bound by instruction issue)
            if (plain_step<OPT>(a)) {
                for (int p = tid; DIAG ? (p - lane < n4) : (p < n4); p += BLOCK_THREADS)
                    generic_position<OPT, GT, POST, MASK, 4, DIAG, true>(a, sp, sscale, static_cast<long long>(p) * 4,
                                                                        p < n4, wd);
            } else {
                for (int p = tid; DIAG ? (p - lane < n4) : (p < n4); p += BLOCK_THREADS)
                    generic_position<OPT, GT, POST, MASK, 4, DIAG>(a, sp, sscale, static_cast<long long>(p) * 4,
                                                                  p < n4, wd);
            }
            const int rem = ch.count & 3;
            if (DIAG ? (tid < 32 && rem > 0) : (tid < rem))
                generic_position<OPT, GT, POST, MASK, 1, DIAG>(a, sp, sscale, (n4 << 2) + tid, tid < rem, wd);
        } else {
            for (int e = tid; DIAG ? (e - lane < ch.count) : (e < ch.count); e += BLOCK_THREADS)
                generic_position<OPT, GT, POST, MASK, 1, DIAG>(a, sp, sscale, e, e < ch.count, wd);
        }
        if constexpr (DIAG) {
            __syncthreads();
            for (int j = tid; j < DIAG_KINDS * a.M; j += BLOCK_THREADS) {
                const int kind = j / a.M, m = j - kind * a.M;
                float total = 0.f;
#pragma unroll
                for (int w = 0; w < BLOCK_THREADS / 32; ++w)
                    total += srows[(w * DIAG_KINDS + kind) * GEN_MAX_M + m];
                a.diag[(static_cast<long long>(kind) * a.M + m) * a.diag_stride + c] = total;
            }
            if (c == 0 && tid == 0) *a.diag_parts = 1;
        }
    }
}

template <int OPT, typename GT, bool POST, bool DIAG, int MASK>
const void *generic_ptr() {
    return reinterpret_cast<const void *>(&desloc_step_generic_kernel<OPT, GT, POST, MASK, DIAG>);
}

template <int OPT, typename GT, bool POST, bool DIAG>
const void *pick_mask(int mask) {
    switch (mask) {
        case 1: return generic_ptr<OPT, GT, POST, DIAG, 1>();
        case 2: return generic_ptr<OPT, GT, POST, DIAG, 2>();
        case 3: return generic_ptr<OPT, GT, POST, DIAG, 3>();
        default: break;
    }
    if constexpr (OPT != OPT_SGDM) {
        switch (mask) {
            case 4: return generic_ptr<OPT, GT, POST, DIAG, 4>();
            case 5: return generic_ptr<OPT, GT, POST, DIAG, 5>();
            case 6: return generic_ptr<OPT, GT, POST, DIAG, 6>();
            case 7: return generic_ptr<OPT, GT, POST, DIAG, 7>();
            default: break;
        }
    }
    return nullptr;
}

template <int OPT, typename GT>
const void *pick_generic(bool post, int mask, bool diag) {
    if (post) return diag ? pick_mask<OPT, GT, true, true>(mask) : pick_mask<OPT, GT, true, false>(mask);
    return diag ? pick_mask<OPT, GT, false, true>(mask) : pick_mask<OPT, GT, false, false>(mask);
}

}  // namespace

const void *lookup_generic_kernel(int opt, bool post, bool bf16, int mask, bool diag) {
    if (opt == OPT_ADAM)
        return bf16 ? pick_generic<OPT_ADAM, bf16_t>(post, mask, diag) : pick_generic<OPT_ADAM, float>(post, mask, diag);
    if (opt == OPT_ADOPT)
        return bf16 ? pick_generic<OPT_ADOPT, bf16_t>(post, mask, diag) : pick_generic<OPT_ADOPT, float>(post, mask, diag);
    if (opt == OPT_SGDM)
        return bf16 ? pick_generic<OPT_SGDM, bf16_t>(post, mask, diag) : pick_generic<OPT_SGDM, float>(post, mask, diag);
    return nullptr;
}

}  // namespace desloc
