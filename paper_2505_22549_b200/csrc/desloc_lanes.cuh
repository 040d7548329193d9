// The step of small and mid-sized problems: a thread per worker and four coordinates, the replicas of a
// coordinate in the lanes of one warp.
//
// Bound: latency up to about a million coordinates (parameters times workers), then HBM.  What a tile
// kernel spends on such a problem is a chain: the copy engine's round trip, or, straight from global memory, one
// round trip per worker (a worker's stores stand in front of the next one's loads), and rounds of few large
// blocks.  Here a thread requests all it needs at once -- x, u, v and g of its four coordinates, 128 bits at a
// time -- and the worker means are shuffles: no barrier, ten blocks of four warps per SM.
// Sums have the order of the tile kernels (tree_sum): same bits.
//
// Measured on B200, Adam, bf16 gradients, per step of a graph of dependent steps, the arrays cold in L2 from 0.25 million
// coordinates on, without the short way behind the wait at the kernel's end (before: the tile kernels).  One array averaged: eight workers x 7.5 K parameters 1.8 us (4.8), x 125 K 6.5
// (9.8), x 300 K 12.6 (17.4); four x 15 K 1.7 (2.8); two x 250 K 3.7 (5.4).  Four x 250 K, all averaged, 6.5 (9.1).
// Local steps: four x 2.5 K 1.5 us (1.7), x 250 K 5.8 (6.6), x 400 K 8.0 (9.5), x 1.25 M 21.9 (22.7).
#pragma once
#include <type_traits>
#include <utility>

#include "desloc_kernels.cuh"

namespace desloc {

// Four coordinates of one worker within a piece of `cnt`: side by side (WIDE, 128-bit accesses), or `step` apart.
template <bool WIDE>
struct Quad {
    int e, step, cnt;
    bool live;   // (lanes of no worker read and write nothing)
    __device__ __forceinline__ bool has(int j) const { return live && (WIDE ? e : e + j * step) < cnt; }
    __device__ __forceinline__ FV<4> ld(const float *p) const {
        FV<4> r = splat<4>(0.f);
        if constexpr (WIDE) {
            if (has(0)) r = ld_f32<4>(reinterpret_cast<const char *>(p), e);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (has(j)) r.a[j] = p[e + j * step];
        }
        return r;
    }
    template <typename GT>
    __device__ __forceinline__ FV<4> ldg(const char *p) const {
        FV<4> r = splat<4>(0.f);
        if constexpr (WIDE) {
            if (has(0)) r = ld_grad<4, GT>(p, e);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (has(j)) r.a[j] = ld_grad<1, GT>(p, e + j * step).a[0];
        }
        return r;
    }
    __device__ __forceinline__ float sum_of_squares(const FV<4> &v) const {
        if constexpr (WIDE) return has(0) ? sum_sq<4>(v) : 0.f;
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (has(j)) s = fmaf(v.a[j], v.a[j], s);
        return s;
    }
    __device__ __forceinline__ void st(float *p, const FV<4> &v) const {
        if constexpr (WIDE) {
            if (has(0)) st_f32<4>(reinterpret_cast<char *>(p), e, v);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (has(j)) p[e + j * step] = v.a[j];
        }
    }
};

// One worker's arrays from the first coordinate of a piece on.
template <int OPT, typename GT>
struct Replica {
    float *x, *u, *v;
    const char *g;
    __device__ __forceinline__ Replica(const StepArgs &a, long long idx, long long start)
        : x(a.x[idx] + start), u(a.u[idx] + start), v(OPT != OPT_SGDM ? a.v[idx] + start : nullptr),
          g(static_cast<const char *>(grad_ptr(a, idx)) + start * static_cast<long long>(sizeof(GT))) {}
    // 16-byte aligned states, and gradients as wide as four of them
    __device__ __forceinline__ bool wide_ok() const {
        return ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(u) | reinterpret_cast<uintptr_t>(v) |
                 (reinterpret_cast<uintptr_t>(g) << (sizeof(GT) == 2 ? 1 : 0))) & 15u) == 0;
    }
};

// Where the loads of a thread land: array k (x, u, v, and fp32 gradients as the fourth) at `p + k * stride`.  128-bit loads
// go there past L1 (cp.async): in registers' place, the bytes in flight need room in L1, and behind a kernel
// that left most of the SM to shared memory, as the tile kernels do, there are 28 KB of it -- local steps of four workers x 1.25 M
// parameters took 26.0 us then instead of 21.9, with loads that allocate no lines 24.9, this way 22.1 behind either.
struct Landing {
    float *p;
    int stride;
    __device__ __forceinline__ void load(int k, const float *src) const {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                     :: "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p + k * stride))), "l"(src) : "memory");
    }
    __device__ __forceinline__ FV<4> get(int k) const { return ld_f32<4>(reinterpret_cast<const char *>(p + k * stride), 0); }
};
template <int OPT, typename GT>
__host__ __device__ constexpr int landing_arrays() { return (OPT == OPT_SGDM ? 2 : 3) + (sizeof(GT) == 4 ? 1 : 0); }

// A thread's four coordinates through the step, out of the arrays `from` and back to the same ones, which to() gives.
// mean(values, arrays) replaces values[i], of array arrays::at(i) (0 x, 1 u, 2 v), by their worker means; all threads that
// share a mean call it together.
template <int... A>
struct Arrays {
    static constexpr int N = sizeof...(A);
    static __device__ constexpr int at(int i) {
        constexpr int a[] = {A...};
        return a[i];
    }
};
// norms(kind, sum) in a step with diagnostics: a thread's sums of squares of the gradient as read, the update and the new parameters.
struct NoNorms {};
// REGS: loads into registers -- a shared-memory round trip less (0.07 us of a step), where a few blocks per SM leave L1 room enough.
template <int OPT, int MASK, typename GT, bool POST, bool PLAIN, bool WIDE, bool REGS = false, typename Mean, typename Where, typename Norms = NoNorms>
__device__ __forceinline__ void update_quad(const StepArgs &a, float sc, const Quad<WIDE> &q, const Landing &land,
                                            const Replica<OPT, GT> &from, const Where &to, const Mean &mean, const Norms &norms = {}) {
    constexpr bool DIAG = !std::is_same_v<Norms, NoNorms>;
    constexpr bool SX = MASK & SYNC_X, SU = MASK & SYNC_U, HAS_V = OPT != OPT_SGDM, P = OPT != OPT_SGDM;
    constexpr bool SV = (MASK & SYNC_V) && HAS_V;
    FV<4> X{}, U{}, V{}, G{}, un, vn;
    if constexpr (WIDE && REGS) {
        if (q.has(0)) {
            X = ld_f32<4>(reinterpret_cast<const char *>(from.x), q.e);
            U = ld_f32<4>(reinterpret_cast<const char *>(from.u), q.e);
            if constexpr (HAS_V) V = ld_f32<4>(reinterpret_cast<const char *>(from.v), q.e);
            G = ld_grad<4, GT>(from.g, q.e);
        }
    } else if constexpr (WIDE) {
        if (q.has(0)) {
            land.load(0, from.x + q.e);
            land.load(1, from.u + q.e);
            if constexpr (HAS_V) land.load(2, from.v + q.e);
            if constexpr (sizeof(GT) == 4) land.load(HAS_V ? 3 : 2, reinterpret_cast<const float *>(from.g) + q.e);
            else G = ld_grad<4, GT>(from.g, q.e);
            asm volatile("cp.async.wait_all;" ::: "memory");
            X = land.get(0);
            U = land.get(1);
            if constexpr (HAS_V) V = land.get(2);
            if constexpr (sizeof(GT) == 4) G = land.get(HAS_V ? 3 : 2);
        }
    } else {
        X = q.ld(from.x);
        U = q.ld(from.u);
        if constexpr (HAS_V) V = q.ld(from.v);
        G = q.template ldg<GT>(from.g);
    }
    if constexpr (DIAG) norms(DIAG_G, q.sum_of_squares(G));
    const auto step = [&] {
        const FV<4> D = minus_direction<OPT, PLAIN, 4>(a, un, vn);
        if constexpr (DIAG) norms(DIAG_D, q.sum_of_squares(D));
        X = apply_step<4, P>(a, X, D);
    };
    if constexpr (!POST) {
        const FV<4> vown = V;
        // (one case per subset of the three arrays)
        if constexpr (SX && SU && SV) {
            FV<4> s[3] = {X, U, V};
            mean(s, Arrays<0, 1, 2>{});
            X = s[0]; U = s[1]; V = s[2];
        } else if constexpr (SX && SU) {
            FV<4> s[2] = {X, U};
            mean(s, Arrays<0, 1>{});
            X = s[0]; U = s[1];
        } else if constexpr (SX && SV) {
            FV<4> s[2] = {X, V};
            mean(s, Arrays<0, 2>{});
            X = s[0]; V = s[1];
        } else if constexpr (SU && SV) {
            FV<4> s[2] = {U, V};
            mean(s, Arrays<1, 2>{});
            U = s[0]; V = s[1];
        } else if constexpr (SX || SU || SV) {
            FV<4> s[1] = {SX ? X : SU ? U : V};
            mean(s, Arrays<SX ? 0 : SU ? 1 : 2>{});
            (SX ? X : SU ? U : V) = s[0];
        }
        state_update<OPT, PLAIN, 4>(a, G, sc, U, V, vown, un, vn);
        step();
    } else {
        state_update<OPT, PLAIN, 4>(a, G, sc, U, V, V, un, vn);
        if constexpr (SU && SV) {
            FV<4> s[2] = {un, vn};
            mean(s, Arrays<1, 2>{});
            un = s[0]; vn = s[1];
        } else if constexpr (SU || SV) {
            FV<4> s[1] = {SU ? un : vn};
            mean(s, Arrays<SU ? 1 : 2>{});
            (SU ? un : vn) = s[0];
        }
        step();
        if constexpr (SX) {
            FV<4> s[1] = {X};
            mean(s, Arrays<0>{});
            X = s[0];
        }
    }
    if constexpr (DIAG) norms(DIAG_X, q.sum_of_squares(X));
    const Replica<OPT, GT> w = to();
    q.st(w.x, X);
    q.st(w.u, un);
    if constexpr (HAS_V) q.st(w.v, vn);
}

// Work item: a run of a chunk, of all MT replicas (of replica blockIdx.y for MT = 1, the local step of any worker
// count).  A worker has 32 / lanes_groups(MT) lanes of every warp.  Five to seven workers take eight groups, of which some
// idle: a sum over eight is three shuffles, a sum over six, of the values one by one, six -- all-sync steps of six
// workers x 270 K parameters 10.7 us against 12.0 with 30 busy lanes.  Three workers have three groups: x 530 K 10.0
// against 10.5 with four.
constexpr int LANES_THREADS = 128;
__host__ __device__ constexpr int lanes_groups(int mt) { return mt <= 4 ? mt : 8; }
__host__ __device__ constexpr int lanes_part_elems(int mt) { return LANES_THREADS / 32 * 4 * (32 / lanes_groups(mt)); }

// Blocks per SM that the compiler has to leave room for, where it would take a step of registers more without a need (34 to 44 instead of 32 or
// 40, nothing spilled without them): a kernel of many blocks lives on those in flight.  Four workers, SGDM, x and u averaged, bf16 gradients,
// 1 to 5 million coordinates: 16 blocks 0.84 to 0.95 of the time with 12, one of three arrays 0.94; Adam, five to eight workers, and ADOPT behind the
// average, 0.5 to 1.5 million: 12 blocks 0.81 to 0.97 of 10.  (The others are faster with the registers: SGDM of two workers behind the
// average 1.1 of the time with 16 blocks, Adam of five to seven that averages all arrays up to 1.16 with 12.)
__host__ __device__ constexpr int lanes_min_blocks(int opt, int mask, int mt, bool post) {
    if (opt == OPT_SGDM) return post ? (mt == 2 ? 10 : 16) : mt == 2 || mt == 3 ? 12 : 16;
    if (opt == OPT_ADOPT) return post && mt >= 5 && mt < 8 ? 12 : 10;
    return !post && mt >= 5 && (mt == 8 ? mask == 5 : mask == 1 || mask == 3) ? 12 : 10;
}

template <int OPT, int MASK, int MT, typename GT, bool POST>
__global__ void __launch_bounds__(LANES_THREADS, lanes_min_blocks(OPT, MASK, MT, POST)) desloc_lanes_kernel(const __grid_constant__ StepArgs a) {
    constexpr int G = lanes_groups(MT), LW = 32 / G;   // lanes of a worker
    begin_and_let_next_begin();
    const unsigned c = item_chunk(a, blockIdx.x);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int part0 = static_cast<int>(blockIdx.x - c * a.parts) * a.part_elems + warp * (4 * LW);
    const Chunk ch = a.chunks[c];
    const int cnt = min(ch.count - part0, 4 * LW);
    const int own = lane / LW, lx = lane - own * LW;
    const int m = MT == 1 ? static_cast<int>(blockIdx.y) : min(own, MT - 1);
    if (cnt <= 0) return;   // (of the whole warp)
    const Replica<OPT, GT> w(a, static_cast<long long>(m) * a.nt + ch.tensor, ch.start + part0);
    __shared__ float4 landing[landing_arrays<OPT, GT>()][LANES_THREADS];
    const Landing land{reinterpret_cast<float *>(&landing[0][threadIdx.x]), 4 * LANES_THREADS};
    const bool live = own < MT, wide = __all_sync(0xffffffffu, w.wide_ok() && (cnt & 3) == 0);
    const auto mean = [&](auto &arrays, auto) {
        if constexpr (MT > 1) {
#pragma unroll
            for (auto &v : arrays) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if constexpr ((G & (G - 1)) == 0) {
                        // a butterfly adds in tree_sum's order (a sum's two sides may change places, and adding -0
                        // for a worker that is not there changes nothing)
                        float t = live ? v.a[j] : -0.f;
#pragma unroll
                        for (int o = LW; o < 32; o *= 2) t += __shfl_xor_sync(0xffffffffu, t, o);
                        v.a[j] = div_sum<MT>(t);
                    } else {
                        float s[MT];
#pragma unroll
                        for (int k = 0; k < MT; ++k) s[k] = __shfl_sync(0xffffffffu, v.a[j], k * LW + lx);
                        v.a[j] = mean_of<MT>(s);
                    }
                }
            }
        }
    };
    // What follows the wait is a latency-bound step's whole time: the common forms have it to themselves, every branch in front.  A step
    // of a graph of dependent ones, 4096 parameters x 2 workers, fp32 gradients: 1.06 us instead of 1.35 (loads through shared memory, branches
    // behind the wait); with the branches in front alone 1.21, with the registers alone 1.28; 1.02 us a kernel that loads and stores x.
    const auto stay = [&] { return w; };
    if (wide && plain_step<OPT>(a)) {
        const Quad<true> q{4 * lx, 1, cnt, live};
        if (a.direct) {
            wait_for_earlier_kernels();
            update_quad<OPT, MASK, GT, POST, true, true, true>(a, 1.f, q, land, w, stay, mean);
        } else {
            wait_for_earlier_kernels();
            update_quad<OPT, MASK, GT, POST, true, true>(a, 1.f, q, land, w, stay, mean);
        }
        return;
    }
    wait_for_earlier_kernels();
    const float sc = a.gscale ? a.gscale[m] : 1.f;
    if (wide) {
        const Quad<true> q{4 * lx, 1, cnt, live};
        update_quad<OPT, MASK, GT, POST, false, true>(a, sc, q, land, w, stay, mean);
    } else {
        const Quad<false> q{lx, LW, cnt, live};
        update_quad<OPT, MASK, GT, POST, false, false>(a, sc, q, land, w, stay, mean);
    }
}

template <int OPT, typename GT, bool POST, int NMASK, int... I>
const void *pick_lanes(int mt, int mask, std::integer_sequence<int, I...>) {
    static const void *const tbl[] = {
        reinterpret_cast<const void *>(&desloc_lanes_kernel<OPT, 1 + I % NMASK, 2 + I / NMASK, GT, POST>)...};
    if (mt < 2 || mt > MAX_MT || mask < 1 || mask > NMASK) return nullptr;
    return tbl[(mt - 2) * NMASK + mask - 1];
}

template <int OPT, typename GT>
const void *lookup_lanes(bool post, int mt, int mask) {
    constexpr int NMASK = OPT == OPT_SGDM ? 3 : 7;
    using Seq = std::make_integer_sequence<int, (MAX_MT - 1) * NMASK>;
    if (mask == 0) return reinterpret_cast<const void *>(&desloc_lanes_kernel<OPT, 0, 1, GT, false>);
    return post ? pick_lanes<OPT, GT, true, NMASK>(mt, mask, Seq{}) : pick_lanes<OPT, GT, false, NMASK>(mt, mask, Seq{});
}

// One unit per optimizer.  Mask 0 is the one-replica kernel, whatever mt; else mt in 2..MAX_MT.
const void *lookup_lanes_adam(bool post, bool bf16, int mt, int mask);
const void *lookup_lanes_adopt(bool post, bool bf16, int mt, int mask);
const void *lookup_lanes_sgdm(bool post, bool bf16, int mt, int mask);

}  // namespace desloc
