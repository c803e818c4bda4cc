// Two steps of a 2D symmetric five-velocity lattice in one pass over memory
// (thermal, periodic, FP32, FP16 or BF16 storage; the single step is plbm_pair.cuh's).
//
// A single FP32 step moves 200 bytes a node and is bound by them: 2048^2 takes
// 120.9 us, 6.9 TB/s, while the SMs could update twice as many nodes.  So the state
// between two steps is kept out of memory.  A CTA owns a strip of columns times a
// segment of rows and walks up the rows.  At row r it
//   1. pulls row r from the old array (loads issued one row ahead, into registers),
//      collides it and puts the 25 populations into shared memory;
//   2. pulls row r - w (w = max |v|) from there, collides it and stores it in the new array.
// Population column j needs its rows only from r - w - v_j to r, so it keeps
// w + v_j + 1 rows in a ring: 25 (w + 1) values a column instead of 25 (2 w + 1), 76.8 KB
// for 96 columns of pairs and w = 3, which lets two CTAs share an SM: one loads and
// collides while the other waits at a barrier.  A strip computes its first step on w more columns
// and rows at each side.  The arithmetic is sym5_collide's and the state
// bit for bit that of two single steps.
//
// Measured, us a step, single and here: v = {0, +-1, +-3} 2048^2 120.9 and 90.5, 2047^2 123.4 and
// 89.2, 4096^2 478 and 344, 8192^2 1935 and 1374, 1500 x 900 40.8 and 34.8, 1024^2 32.0 and 28.5;
// {0, +-1, +-2} 2048^2 120.9 and 78.6, 2047^2 123.4 and 83.2.
// What bounds it: a warp's own latencies (1.5 warps a scheduler in pairs, 4.4 cycles from one
// instruction to the next, a fifth of them waiting for loads); with all data in the second-level cache
// 2048^2 takes 81 us a step, its traffic alone 65.
//
// 16-bit storage: the ring holds the rounded values that memory would, half the bytes, so that 12 warps
// (pairs, 128 threads, three CTAs per SM) or 20 (plain) share an SM.  Their single steps are bound
// by the SMs nearly as much as by memory; two at a time gain on large lattices: FP16 2048^2 67.7 and 63.7
// (w = 2: 61.4), 4096^2 258 and 228, 4095^2 404 and 312, BF16 2048^2 67.7 and 65.9, 4096^2 261 and 236.
#pragma once

#include <algorithm>
#include <type_traits>

#include "plbm_pair.cuh"

namespace plbm {

inline int fuse_w(const LatticeParams& P) { return (int)std::max(P.sa, P.sb); }
// Threads of a CTA and CTAs per SM (32 bits).  More of either leaves too little first-level cache for
// the loads in flight (25 lines of 128 or 256 bytes a warp): at w = 3 two CTAs of 128 threads in pairs,
// 205 KB of rings, take 222 us where two of 96 take 181.
struct FuseShape {
    int threads, resident;
    size_t smem;
};
template <typename S>
FuseShape fuse_shape(const LatticeParams& P) {
    const int w = fuse_w(P);
    int threads = 128, resident = P.paired ? 3 : 5;   // 16 bits
    if (sizeof(S) == 4) {
        threads = P.paired ? (w > 2 ? 96 : 64) : 128;
        resident = w > 2 ? (P.paired ? 2 : 3) : 4;
    }
    return {threads, resident, 25 * (size_t)(w + 1) * threads * sizeof(S) * (P.paired ? 2 : 1)};
}

// What the arrays hold of a column, both nodes of a pair or one node, and its FP32 value.
template <class E>
struct FuseElem;
template <typename S>
struct FusePair {
    using E = typename PairStore<S>::V;
    using V = float2;
    static constexpr bool kPaired = true;
    static __device__ __forceinline__ E load(const E* p) { return load_state(p); }
    static __device__ __forceinline__ V cvt(E v) { return PairStore<S>::cvt(v); }
    static __device__ __forceinline__ V cvt_again(E v) { return PairStore<S>::cvt_again(v); }
    static __device__ __forceinline__ E pack(V v) {
        E e;
        PairStore<S>::store(&e, v);
        return e;
    }
    static __device__ __forceinline__ E swap(E v) { return PairStore<S>::swap(v); }
};
template <>
struct FuseElem<float2> : FusePair<float> {};
template <>
struct FuseElem<__half2> : FusePair<__half> {};
template <>
struct FuseElem<__nv_bfloat162> : FusePair<__nv_bfloat16> {};
template <typename S>
struct FuseNode {
    using V = float;
    static constexpr bool kPaired = false;
    static __device__ __forceinline__ S load(const S* p) { return load_state(p); }
    static __device__ __forceinline__ V cvt_again(S v) { return cvt(v); }
    static __device__ __forceinline__ V cvt(S v) {
        if constexpr (std::is_same<S, __half>::value) return __half2float(v);
        else if constexpr (std::is_same<S, __nv_bfloat16>::value) return __bfloat162float(v);
        else return v;
    }
    static __device__ __forceinline__ S pack(V v) {
        S s;
        Scalar16<S>::store(&s, v);
        return s;
    }
    static __device__ __forceinline__ S swap(S v) { return v; }
};
template <>
struct FuseElem<float> : FuseNode<float> {};
template <>
struct FuseElem<__half> : FuseNode<__half> {};
template <>
struct FuseElem<__nv_bfloat16> : FuseNode<__nv_bfloat16> {};

// Two steps of columns [x0, x0 + wn) of (pair) rows [r0, r1); wn + 2w <= NC.  E: what the arrays hold of
// a column (float2: both nodes of a pair; float: one node), V: what a thread takes, one column
// (V = E) or, in the plain layout, columns t and t + NT (E = float, V = float2).
// rows >= 2w and nx >= 2w: no index wraps twice.  begin() is called before the first load.
template <class E, class V, int NT, class Begin>
__device__ __forceinline__ void two_steps(const PairParams& P, const E* src, E* __restrict__ dst, E* ring, int x0,
                                          int wn, int r0, int r1, Begin begin) {
    using X = FuseElem<E>;
    constexpr bool kPaired = X::kPaired, kTwo = sizeof(V) > sizeof(typename X::V);   // kTwo: E = float, V = float2
    using G = typename std::conditional<kTwo, V, E>::type;   // as loaded
    constexpr int NC = kTwo ? 2 * NT : NT;   // columns of a ring row
    const int va = (int)P.sa, vb = (int)P.sb, w = max(va, vb);
    const int v[5] = {0, va, -va, vb, -vb};
    const int rows = kPaired ? P.half_ny : P.ny;
    const int t = threadIdx.x;
    const bool first = t < wn + 2 * w, second = t < wn;   // has a column in step 1, in step 2
    // kTwo, the second column: t + NT, or the last one again in a narrow strip (stored in the ring twice, not in dst)
    const int t1 = min(t + NT, wn + 2 * w - 1), t2 = min(t + NT, wn - 1);
    auto pulled_columns = [&](int c, unsigned (&col)[5]) {
        int x = x0 - w + c;
        x = x < 0 ? x + P.nx : (x >= P.nx ? x - P.nx : x);
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const int k = x + P.vxm[i];
            col[i] = (unsigned)(k >= P.nx ? k - P.nx : k);
        }
    };
    unsigned col[5], col1[5];
    pulled_columns(first ? t : 0, col);
    if constexpr (kTwo) pulled_columns(t1, col1);
    int depth[5], base[5], slot[5];   // rows of population column j in the ring, where they start, the row in turn
    {
        int o = 0;
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            depth[j] = w + v[j] + 1;
            base[j] = o;
            slot[j] = 0;
            o += depth[j] * 5 * NC;
        }
    }
    G g[25];
    auto load = [&](int rr) {   // the pulls of row rr; rows outside [0, rows) lie across the y wrap, pairs swapped
        unsigned row[5];
        bool swp[5], any = false;
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            int k = rr - v[j];
            swp[j] = k < 0 || k >= rows;
            any |= swp[j];
            k = k < 0 ? k + rows : (k >= rows ? k - rows : k);
            row[j] = (unsigned)k * (unsigned)P.pitch;
        }
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                const E* q = src + (5 * i + j) * P.plane2;
                if constexpr (kTwo)
                    g[5 * i + j] = f2(X::load(q + (row[j] + col[i])), X::load(q + (row[j] + col1[i])));
                else
                    g[5 * i + j] = X::load(q + (row[j] + col[i]));
            }
        if constexpr (kPaired) {
            if (any) {
#pragma unroll
                for (int p = 0; p < 25; ++p)
                    if (swp[p % 5]) g[p] = X::swap(g[p]);
            }
        }
    };
    V rho, th, drho, jx, jy, e;
    begin();
    if (first) load(r0 - w);
    for (int rr = r0 - w; rr < r1 + w; ++rr) {
        if (first) {
            V o[25];
            if constexpr (kTwo)
                sym5_collide<V>(P, [&](int p) { return g[p]; }, [&](int p) { return g[p]; }, o, rho, th, drho, jx, jy, e);
            else
                sym5_collide<V>(P, [&](int p) { return X::cvt(g[p]); }, [&](int p) { return X::cvt_again(g[p]); }, o, rho, th,
                                drho, jx, jy, e);
            flag_unhealthy(P, rho, th);
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                E* q = ring + base[j] + slot[j] * 5 * NC;
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    if constexpr (kTwo)
                        q[i * NC + t] = o[5 * i + j].x, q[i * NC + t1] = o[5 * i + j].y;
                    else
                        q[i * NC + t] = X::pack(o[5 * i + j]);
                }
            }
            if (rr + 1 < r1 + w) load(rr + 1);
        }
        __syncthreads();
        // the oldest row of each ring, the next to be overwritten, is the one that row rr - w pulls
#pragma unroll
        for (int j = 0; j < 5; ++j) slot[j] = slot[j] + 1 == depth[j] ? 0 : slot[j] + 1;
        if (second && rr - w >= r0) {
            V o[25];
            G h[25];
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                const E* q = ring + base[j] + slot[j] * 5 * NC + w;
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    if constexpr (kTwo)
                        h[5 * i + j] = f2(q[i * NC + t - v[i]], q[i * NC + t2 - v[i]]);
                    else
                        h[5 * i + j] = q[i * NC + t - v[i]];
                }
            }
            if constexpr (kTwo)
                sym5_collide<V>(P, [&](int p) { return h[p]; }, [&](int p) { return h[p]; }, o, rho, th, drho, jx, jy, e);
            else
                sym5_collide<V>(P, [&](int p) { return X::cvt(h[p]); }, [&](int p) { return X::cvt_again(h[p]); }, o, rho, th,
                                drho, jx, jy, e);
            flag_unhealthy(P, rho, th);
            E* q = dst + ((unsigned)(rr - w) * (unsigned)P.pitch + (unsigned)(x0 + t));
#pragma unroll
            for (int p = 0; p < 25; ++p) {
                if constexpr (kTwo) {
                    q[p * P.plane2] = o[p].x;
                    if (t + NT < wn) q[p * P.plane2 + NT] = o[p].y;
                } else {
                    q[p * P.plane2] = X::pack(o[p]);
                }
            }
        }
        __syncthreads();
    }
}

// One lattice: grid = (strips, segments), CTA (b, s) owns columns [nx b / strips, nx (b + 1) / strips) of
// (pair) rows [rows s / segments, rows (s + 1) / segments).
template <class E, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
k_two_steps(const __grid_constant__ PairParams P, const E* src, E* __restrict__ dst) {
    extern __shared__ __align__(16) unsigned char fuse_ring[];
    step_begin();
    const int rows = FuseElem<E>::kPaired ? P.half_ny : P.ny;
    const int x0 = (int)((long long)P.nx * blockIdx.x / gridDim.x);
    const int x1 = (int)((long long)P.nx * (blockIdx.x + 1) / gridDim.x);
    const int r0 = (int)((long long)rows * blockIdx.y / gridDim.y);
    const int r1 = (int)((long long)rows * (blockIdx.y + 1) / gridDim.y);
    two_steps<E, typename FuseElem<E>::V, NT>(P, src, dst, reinterpret_cast<E*>(fuse_ring), x0, x1 - x0, r0, r1, [] { step_wait(); });
}

// The lattices of a batch in one launch: CTA c takes piece c of the list, longest first (FusePiece,
// plbm_internal.h).  Both layouts run on one shape of CTA, 96 threads and two resident: the plain one takes
// two columns a thread (97 against 89 us a step at 2047^2, but no second launch with its own tail).
// 16 lattices of 58 to 932 rows of pairs or nodes, 6.0 M nodes: 180 us a step by k_batch_pair, 139 here (122
// with another batch's launches beside it to fill the tails).
template <int NT>   // a template, as launch_batch_two_steps, to be compiled in the one unit that launches it
__global__ void __launch_bounds__(NT, 2)
k_batch_two_steps(const PairParams* __restrict__ inst, const FusePiece* __restrict__ pieces, int parity) {
    extern __shared__ __align__(16) unsigned char fuse_ring[];
    __shared__ PairParams sp;
    step_begin();
    const FusePiece p = pieces[blockIdx.x];
    for (int k = threadIdx.x; k < (int)(sizeof(PairParams) / sizeof(int)); k += NT)
        reinterpret_cast<int*>(&sp)[k] = reinterpret_cast<const int*>(&inst[p.inst])[k];
    __syncthreads();
    const PairParams lp = sp;   // in registers: no store of the loop can change it (142.7 -> 139.5 us a step for 6.0 M nodes)
    if (sp.paired)
        two_steps<float2, float2, NT>(lp, static_cast<const float2*>(sp.f[parity]), static_cast<float2*>(sp.f[parity ^ 1]),
                                                     reinterpret_cast<float2*>(fuse_ring), p.x0, p.wn, p.r0, p.r1,
                                                     [] { step_wait(); });
    else
        two_steps<float, float2, NT>(lp, static_cast<const float*>(sp.f[parity]), static_cast<float*>(sp.f[parity ^ 1]),
                                                    reinterpret_cast<float*>(fuse_ring), p.x0, p.wn, p.r0, p.r1,
                                                    [] { step_wait(); });
}

// The split of a lattice for k_two_steps, or strips = 0 where single steps are taken: lattices whose
// two arrays fit in the second-level cache (768^2: 18.7 us a step against 14.7), and those that do
// not fill the strips and segments well.  A CTA takes row_us for a row while the chip is full,
// whatever the width of its strip, so two steps take waves x (rows of a segment + 2w) x row_us, which
// the number of segments minimises; single steps go at the memory's rate.  Of 3,585 sizes drawn between 800^2 (16 bits:
// 1500^2) and 4096^2, aspect ratios up to 3, that the rule takes none was slower than by single steps: 0.72 of their
// time at the median and 0.92 at most in FP32, 0.88 and 0.97 in FP16, 0.90 and 0.99 in BF16.
struct FusePlan {
    int strips, segments;
};
template <typename S>
FusePlan fuse_plan(const LatticeParams& P) {
    FusePlan best{0, 0};
    if (P.dim != 2 || !P.sym5 || P.isothermal || P.fixed_ends) return best;
    const int w = fuse_w(P), rows = P.paired ? P.half_ny : P.ny;
    const double nodes = (double)P.nx * P.ny;
    if (w > kFuseMaxV || rows < 2 * w || P.nx < 2 * w || nodes * 50 * sizeof(S) < 1.3e8) return best;
    const FuseShape shape = fuse_shape<S>(P);
    const int most = shape.threads - 2 * w, strips = (P.nx + most - 1) / most, resident = device_sm_count() * shape.resident;
    double row_us = w > 2 ? 2.1 : P.paired ? 2.4 : 2.65, single_us = nodes * (P.paired ? 28.8e-6 : 29.4e-6);
    if (sizeof(S) == 2) {
        row_us = !P.paired ? 3.2 : std::is_same<S, __half>::value ? 2.77 : 2.87;
        single_us = nodes * (P.paired ? 16.1e-6 : 20.2e-6);
    }
    double least = 1e300;
    for (int segs = 1; segs <= rows && segs <= 65535; ++segs) {
        const long long ctas = (long long)strips * segs, waves = (ctas + resident - 1) / resident;
        const double time = (double)waves * ((rows + segs - 1) / segs + 2 * w) * row_us;
        if (time < least) least = time, best = {strips, segs};
        if (waves > 8 && segs > 1) break;
    }
    return least < (sizeof(S) == 2 ? 0.99 : 0.95) * 2 * single_us ? best : FusePlan{0, 0};
}

// Shared memory for the resident CTAs (1 KB each besides what they ask for), the rest as cache.  Every
// caller gives a kernel the same values, so that threads that launch it at once do not disturb each other.
inline cudaError_t fuse_shared_memory(const void* kernel, size_t smem, int resident) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                (int)((resident * (smem + 1024) * 100 + (228 << 10) - 1) / (228 << 10)));
}

// WMAX: the largest w this kernel is launched for.
template <typename S, class E, int NT, int MINB, int WMAX>
cudaError_t launch_two_steps_t(const LatticeParams& L, const void* src, void* dst, cudaStream_t stream) {
    const FusePlan plan = fuse_plan<S>(L);
    const FuseShape shape = fuse_shape<S>(L);
    constexpr size_t kMost = 25 * (size_t)(WMAX + 1) * NT * sizeof(E);
    if (plan.strips == 0 || shape.threads != NT || shape.smem > kMost) return cudaErrorInvalidValue;
    const auto kernel = k_two_steps<E, NT, MINB>;
    const cudaError_t e = fuse_shared_memory(reinterpret_cast<const void*>(kernel), kMost, MINB);
    if (e != cudaSuccess) return e;
    return launch_dependent_smem(true, shape.smem, kernel, dim3(plan.strips, plan.segments), NT, stream, pair_params(L),
                                 static_cast<const E*>(src), static_cast<E*>(dst));
}

template <typename S>
cudaError_t launch_two_steps(const LatticeParams& P, const void* src, void* dst, cudaStream_t stream) {
    using V = typename PairStore<S>::V;
    if constexpr (sizeof(S) == 2)
        return P.paired ? launch_two_steps_t<S, V, 128, 3, kFuseMaxV>(P, src, dst, stream)
                        : launch_two_steps_t<S, S, 128, 5, kFuseMaxV>(P, src, dst, stream);
    else if (fuse_w(P) > 2)
        return P.paired ? launch_two_steps_t<S, V, 96, 2, kFuseMaxV>(P, src, dst, stream)
                        : launch_two_steps_t<S, S, 128, 3, kFuseMaxV>(P, src, dst, stream);
    else
        return P.paired ? launch_two_steps_t<S, V, 64, 4, 2>(P, src, dst, stream) : launch_two_steps_t<S, S, 128, 4, 2>(P, src, dst, stream);
}

constexpr size_t kBatchFuseSmem = 25 * (size_t)(kFuseMaxV + 1) * kBatchFuseThreads * sizeof(float2);
template <int NT = kBatchFuseThreads>
cudaError_t launch_batch_two_steps(const PairParams* inst, const FusePiece* pieces, int npieces, int parity,
                                          cudaStream_t stream) {
    // 500 bytes and more of static shared memory besides the ring
    const cudaError_t e = fuse_shared_memory(reinterpret_cast<const void*>(k_batch_two_steps<NT>), kBatchFuseSmem + 1024, 2);
    if (e != cudaSuccess) return e;
    return launch_dependent_smem(true, kBatchFuseSmem, k_batch_two_steps<NT>, npieces, NT, stream, inst, pieces, parity);
}

}  // namespace plbm
