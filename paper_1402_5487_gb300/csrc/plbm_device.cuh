// Device code of the PLBM stream-and-collide step (sm_103a).
//
// One thread updates one node.  Populations are SoA planes f[p][y][pitch].
// A step pulls f_p(x - v_p) for every population (Eq. eq:srt read as
// pull + collide on post-collision states), takes the moments, evaluates the
// Maxwell-Boltzmann moments mu_n(u, theta) by their recurrence, forms
// r_i = sum_j c_ij mu_{j-1} per axis (Eq. eq:rdr), the tensor-product
// equilibrium f^eq = rho r^x r^y (Sec. 2.1) and relaxes with omega.
//
// Two arithmetic cores:
//  * Direct (FP64 storage): moments of f, f^eq = rho r^x r^y,
//    f' = f + omega (f^eq - f).
//  * Deviation (FP32, FP16, BF16 storage, FP32 arithmetic): every population is
//    stored and handled as g = f - w0 with w0 = f^eq(1, 0, theta0) the rest
//    equilibrium.
//    Because the rule reproduces mu_0..mu_{q1-1} exactly (Eq. eq:rdr),
//    sum w0 = 1, sum v w0 = 0 and sum |v|^2 w0 = d theta0, so
//        rho - 1 = sum g,  rho u = sum v g,  d rho theta = d theta0 + sum |v|^2 g - rho |u|^2
//    and the equilibrium deviation is built from
//        dmu_n = mu_n(u, theta) - mu_n(0, theta0)   (recurrence below),
//        dr = C dmu,  f^eq - w0 = (rho - 1) w0 + rho (dr^x r^y + w^x dr^y)
//    which never subtracts two O(1) numbers.  Storing g instead of f also makes
//    the storage rounding proportional to |f - w0| rather than to |f|.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <map>
#include <mutex>
#include <type_traits>
#include <utility>

#include "plbm_internal.h"

namespace plbm {

// ---------------------------------------------------------------------------
// Step kernels follow one another on a stream, each reading what the one before
// wrote.  Launched plainly, a step waits for the last block of the step before, then
// for its own launch: 2-5 us in which the SMs drain and refill.  They are
// launched as programmatic dependents instead: a block says at its start that the
// next grid may be set up (step_begin), whose blocks then take the SM slots that
// fall free and compute their addresses, and every thread that touches memory
// waits for the grid before to be complete and flushed (step_wait) first.  A
// kernel launched without the attribute passes both at once.  Per step: 2048^2 FP32
// 123.2 -> 120.6 us, FP16 69.7 -> 67.3 us, 512^2 FP32 (graph) 6.56 -> 6.29 us.
// The same trigger does harm where the chip holds the whole grid: the slots it leaves free
// then fill with waiting blocks of the next grids, which crowd it and leave their own
// work unevenly spread over the SMs.  Measured against plain launches over 700 drawn 16/32-bit and 500 drawn
// FP64 lattices (time as a dependent over time launched plainly, median and range; "waves": blocks over resident blocks):
//   16/32-bit 2D   below 0.1 waves 0.86-0.91; 0.1-0.83 1.2 (0.84-1.51); above 0.87 (0.69-1.05)
//     the trigger after the arithmetic (LATE, plbm_pair.cuh): below 0.4 0.93 (0.89-1.03), 0.4-1.5 1.02 (0.94-1.12)
//   16/32-bit 3D   0.83 (0.63-1.03), whatever the waves
//   FP64 2D        0.1-0.8 waves 1.45 (0.97-2.25), 0.8-3 1.00 (0.94-1.27), above 0.99 (0.95-1.01); after the arithmetic
//     with blocks of 32 threads and up to five velocities 0.98 (0.95-0.99), otherwise 1.00 (0.95-1.28)
//   FP64 3D        0.15-3 waves 1.24 (0.85-2.76), above 0.99 (0.97-1.00)
// Hence: the trigger at the start from 5/6 of a wave on (FP64: three waves), after the arithmetic where that gains
// always, plainly otherwise; 3D 16/32-bit grids from kDependentThreads threads on.  Of 530 lattices drawn between 2.5e4
// and 9e5 nodes 5 are then more than 2 % slower than plainly, 1.12 at worst and 0.93 on average (with the trigger at
// the start from 65,536 threads on: 87, 1.46, 0.96).  The persistent batch
// kernels, which leave no slot free, are launched plainly (174 us a step either way).
// ---------------------------------------------------------------------------
constexpr long long kDependentThreads = 1 << 16;
__device__ __forceinline__ void step_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void step_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Every load of what the grid before wrote, in the step kernels and in k_finalize.  Such a kernel's grid
// is already running while its source is being written, which is what the read-only path (ld.global.nc:
// __ldg, or a const __restrict__ pointer) is not defined for, and a compiler may move a load that it takes for
// invariant, or that is no volatile statement, across step_wait.  A volatile ld.global stays behind it. (Against the
// read-only path: 512^2 FP32 6.07 -> 5.74 us a step, 64^3 FP64 409 -> 393, the others within 1 %.)
template <class T>
__device__ __forceinline__ T load_state(const T* p) {
    static_assert(sizeof(T) == 2 || sizeof(T) == 4 || sizeof(T) == 8 || sizeof(T) == 16, "size of a load");
    const size_t at = __cvta_generic_to_global(p);
    T v;
    if constexpr (sizeof(T) == 2) {
        unsigned short r;
        asm volatile("ld.global.b16 %0, [%1];" : "=h"(r) : "l"(at));
        memcpy(&v, &r, 2);
    } else if constexpr (sizeof(T) == 4) {
        unsigned r;
        asm volatile("ld.global.b32 %0, [%1];" : "=r"(r) : "l"(at));
        memcpy(&v, &r, 4);
    } else if constexpr (sizeof(T) == 8) {
        unsigned long long r;
        asm volatile("ld.global.b64 %0, [%1];" : "=l"(r) : "l"(at));
        memcpy(&v, &r, 8);
    } else {
        unsigned long long r[2];
        asm volatile("ld.global.v2.b64 {%0, %1}, [%2];" : "=l"(r[0]), "=l"(r[1]) : "l"(at));
        memcpy(&v, r, 16);
    }
    return v;
}
// FP64 kernels of 1D lattices and of blocks of 32 threads: the trigger after the arithmetic.
template <int DIM>
__device__ __forceinline__ bool step_late() {
    return DIM == 1 ? (long long)gridDim.x * blockDim.x < 1 << 18 : blockDim.x == 32;
}

inline int device_sm_count() {
    static int n = 0;
    if (!n) {
        int d = 0;
        cudaGetDevice(&d);
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, d) != cudaSuccess || n < 1) n = 1;
    }
    return n;
}

// Whether `threads` threads with work fill the resident blocks of `kernel` num / den times at least (the occupancy is
// asked for once per kernel and block size).  Idle threads of a row's last block do not count: 38 x 2152 BF16
// (1.01 waves of blocks, 0.3 of threads) takes 4.3 us a step as a dependent and 3.7 plainly.  (FP64 grids, whose rule asks
// for three waves, count them.)
inline bool grid_waves(const void* kernel, long long threads, int block, int num, int den) {
    static std::mutex lock;
    static std::map<std::pair<const void*, int>, int> known;   // resident blocks per SM
    int per_sm;
    {
        std::lock_guard<std::mutex> g(lock);
        auto it = known.find({kernel, block});
        if (it == known.end()) {
            int n = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, block, 0) != cudaSuccess || n < 1) n = 1;
            it = known.emplace(std::make_pair(kernel, block), n).first;
        }
        per_sm = it->second;
    }
    return threads * den >= (long long)per_sm * block * device_sm_count() * num;
}

template <class... P, class... A>
cudaError_t launch_dependent_smem(bool dependent, size_t smem, void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t stream,
                                  A... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = dependent ? 1 : 0;   // otherwise plainly
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <class... P, class... A>
cudaError_t launch_dependent(bool dependent, void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t stream, A... args) {
    return launch_dependent_smem(dependent, 0, kernel, grid, block, stream, args...);
}
// A kernel that triggers at its start: as a dependent from num / den waves on.
template <class... P, class... A>
cudaError_t launch_by_waves(long long threads, int num, int den, void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t stream,
                            A... args) {
    return launch_dependent(grid_waves(reinterpret_cast<const void*>(kernel), threads, block.x, num, den), kernel, grid, block,
                            stream, args...);
}

// ---------------------------------------------------------------------------
// Storage traits: how a stored element becomes an arithmetic value.
// ---------------------------------------------------------------------------
template <typename S>
struct Storage;

template <>
struct Storage<double> {
    static constexpr bool kDeviation = false;
    static __device__ __forceinline__ double load(const double* p) { return load_state(p); }
    static __device__ __forceinline__ void store(double* p, double v) { *p = v; }
    // FP64 value of the population f (for moments/diagnostics of the stored state)
    static __device__ __forceinline__ double to_f64(double s, double) { return s; }
    static __device__ __forceinline__ double from_f64(double f, double) { return f; }
};

template <>
struct Storage<float> {
    static constexpr bool kDeviation = true;   // stores g = f - w0 in FP32
    static __device__ __forceinline__ float load(const float* p) { return load_state(p); }
    static __device__ __forceinline__ void store(float* p, float v) { *p = v; }
    static __device__ __forceinline__ double to_f64(float s, double w0) { return w0 + (double)s; }
    static __device__ __forceinline__ float from_f64(double f, double w0) { return (float)(f - w0); }
};

template <>
struct Storage<__half> {
    static constexpr bool kDeviation = true;   // stores g = f - w0
    static __device__ __forceinline__ float load(const __half* p) { return __half2float(load_state(p)); }
    static __device__ __forceinline__ void store(__half* p, float v) { *p = __float2half_rn(v); }
    static __device__ __forceinline__ double to_f64(__half s, double w0) {
        return w0 + (double)__half2float(s);
    }
    static __device__ __forceinline__ __half from_f64(double f, double w0) {
        return __double2half(f - w0);
    }
};

template <>
struct Storage<__nv_bfloat16> {
    static constexpr bool kDeviation = true;
    static __device__ __forceinline__ float load(const __nv_bfloat16* p) {
        return __bfloat162float(load_state(p));
    }
    static __device__ __forceinline__ void store(__nv_bfloat16* p, float v) {
        *p = __float2bfloat16_rn(v);
    }
    static __device__ __forceinline__ double to_f64(__nv_bfloat16 s, double w0) {
        return w0 + (double)__bfloat162float(s);
    }
    static __device__ __forceinline__ __nv_bfloat16 from_f64(double f, double w0) {
        return __double2bfloat16(f - w0);
    }
};

// ---------------------------------------------------------------------------
// Per-node diagnostics accumulated by reducing launches.
// ---------------------------------------------------------------------------
struct NodeDiag {
    double mass, jx, jy, energy, rho_min, theta_min;
};

__device__ __forceinline__ void diag_zero(NodeDiag& d) {
    d.mass = d.jx = d.jy = d.energy = 0.0;
    d.rho_min = 1e300;
    d.theta_min = 1e300;
}

// Sets PLBM_STATUS_* bits for a node whose rho or theta is non-finite or
// non-positive.  Evaluated in the kernel's own precision (FP32 kernels never
// touch the FP64 pipe here).  NaN compares false, so it lands in the first test.
template <typename R>
__device__ __forceinline__ void flag_status(const LatticeParams& P, R rho, R theta) {
    const R big = (R)3.0e38f;
    if (!(rho > (R)0 && theta > (R)0 && rho < big && theta < big)) {
        unsigned bits = 0u;
        if (!(rho == rho) || !(theta == theta) || !(rho < big) || !(theta < big)) bits |= 1u;
        if (rho <= (R)0) bits |= 2u;
        if (theta <= (R)0) bits |= 4u;
        atomicOr(P.status, bits);
    }
}

// The same for the FP64 step, on the integer pipe: a positive normal number below
// 3e38 has a high word in [1, hi(3e38)); everything else takes the FP64 comparisons.
__device__ __forceinline__ void flag_status_f64(const LatticeParams& P, double rho, double theta) {
    const unsigned top = 0x47ec363cu;   // high word of 3.0e38 (rounded down)
    const unsigned a = (unsigned)__double2hiint(rho) - 1u, b = (unsigned)__double2hiint(theta) - 1u;
    if (a >= top - 1u || b >= top - 1u) flag_status<double>(P, rho, theta);
}

// Float-float numbers: an FP32 pair hi + lo carried through error-free sums
// (TwoSum) and products (FMA), ~2^-48 relative: FP64-grade sums of FP32 data on
// the FP32 pipe (GB300's FP64 rate is two operations per SM per cycle).
struct FF {
    float hi, lo;
};
__device__ __forceinline__ FF ff_add(FF a, float b) {
    const float s = a.hi + b;
    const float t = s - a.hi;
    const float e = (a.hi - (s - t)) + (b - t);
    return {s, a.lo + e};
}
__device__ __forceinline__ FF ff_add(FF a, FF b) {
    const float s = a.hi + b.hi;
    const float t = s - a.hi;
    const float e = (a.hi - (s - t)) + (b.hi - t);
    return {s, (a.lo + b.lo) + e};
}
__device__ __forceinline__ FF ff_scale(FF a, float v) {
    const float p = a.hi * v;
    const float e = fmaf(a.hi, v, -p);
    return {p, fmaf(a.lo, v, e)};
}
// (double)v on the integer pipe: a conversion instruction takes the FP64 pipe (two lanes per SM and
// cycle), predicated off or not, so that subnormal (scaled by 2^24 first), infinite and NaN values
// are selected rather than branched to.
__device__ __forceinline__ double f64_of(float v) {
    unsigned m = __float_as_uint(v) & 0x7fffffffu;
    const unsigned sign = __float_as_uint(v) & 0x80000000u;
    unsigned off = m >= 0x7f800000u ? 0x70000000u : 0x38000000u;
    if (m < 0x00800000u) {
        m = __float_as_uint(__fmul_rn(__uint_as_float(m), 0x1p24f));
        off = m ? 0x38000000u - (24u << 20) : 0u;
    }
    return __hiloint2double((int)(sign | ((m >> 3) + off)), (int)(m << 29));
}
__device__ __forceinline__ double ff_f64(FF a) { return f64_of(a.hi) + f64_of(a.lo); }
__device__ __forceinline__ FF ff_shfl_down(FF a, int off) {
    return {__shfl_down_sync(0xffffffffu, a.hi, off), __shfl_down_sync(0xffffffffu, a.lo, off)};
}

// Per-thread diagnostics of 16/32-bit kernels: deviations from the rest state
// (mass - n, energy - n d theta0) in float-float, n the thread's node count.
struct NodeDiagF {
    FF dmass, jx, jy, denergy;
    float rho_min, theta_min, n;
};
__device__ __forceinline__ void diagf_zero(NodeDiagF& d) {
    d.dmass = d.jx = d.jy = d.denergy = FF{0.0f, 0.0f};
    d.rho_min = d.theta_min = 3.0e38f;
    d.n = 0.0f;
}

// Order-preserving int64 key of a double (total order, negatives included), so
// that FP64 minima reduce on the integer pipe.
__device__ __forceinline__ long long dkey(double v) {
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double dunkey(long long k) {
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
}
__device__ __forceinline__ long long kmin(long long a, long long b) { return a < b ? a : b; }

// Block reduction of NodeDiagF in float-float; thread 0 writes the same FP64
// record as block_reduce_diag (mass = n + dmass, energy = n d theta0 + denergy).
// DMIN: the minima are the caller's FP64 rho_min_d, theta_min_d (1e300 for no
// node), reduced as order-preserving integer keys, instead of the FP32 ones of d.
template <int NT, bool DMIN = false>
__device__ __forceinline__ void block_reduce_diagf(NodeDiagF d, double dtheta0, double* out, double rho_min_d = 0.0,
                                                   double theta_min_d = 0.0) {
    __shared__ float sh[11][NT / 32];
    __shared__ long long shk[2][NT / 32];
    long long kr = 0, kt = 0;
    if (DMIN) {
        kr = dkey(rho_min_d);
        kt = dkey(theta_min_d);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            kr = kmin(kr, __shfl_down_sync(0xffffffffu, kr, off));
            kt = kmin(kt, __shfl_down_sync(0xffffffffu, kt, off));
        }
        if ((threadIdx.x & 31) == 0) {
            shk[0][threadIdx.x >> 5] = kr;
            shk[1][threadIdx.x >> 5] = kt;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        d.dmass = ff_add(d.dmass, ff_shfl_down(d.dmass, off));
        d.jx = ff_add(d.jx, ff_shfl_down(d.jx, off));
        d.jy = ff_add(d.jy, ff_shfl_down(d.jy, off));
        d.denergy = ff_add(d.denergy, ff_shfl_down(d.denergy, off));
        d.rho_min = fminf(d.rho_min, __shfl_down_sync(0xffffffffu, d.rho_min, off));
        d.theta_min = fminf(d.theta_min, __shfl_down_sync(0xffffffffu, d.theta_min, off));
        d.n += __shfl_down_sync(0xffffffffu, d.n, off);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        sh[0][warp] = d.dmass.hi;
        sh[1][warp] = d.dmass.lo;
        sh[2][warp] = d.jx.hi;
        sh[3][warp] = d.jx.lo;
        sh[4][warp] = d.jy.hi;
        sh[5][warp] = d.jy.lo;
        sh[6][warp] = d.denergy.hi;
        sh[7][warp] = d.denergy.lo;
        sh[8][warp] = d.rho_min;
        sh[9][warp] = d.theta_min;
        sh[10][warp] = d.n;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        FF m{0.f, 0.f}, a{0.f, 0.f}, b{0.f, 0.f}, e{0.f, 0.f};
        float rmin = 3.0e38f, tmin = 3.0e38f, n = 0.0f;
        for (int w = 0; w < NT / 32; ++w) {
            m = ff_add(m, FF{sh[0][w], sh[1][w]});
            a = ff_add(a, FF{sh[2][w], sh[3][w]});
            b = ff_add(b, FF{sh[4][w], sh[5][w]});
            e = ff_add(e, FF{sh[6][w], sh[7][w]});
            rmin = fminf(rmin, sh[8][w]);
            tmin = fminf(tmin, sh[9][w]);
            n += sh[10][w];
        }
        out[0] = (double)n + ff_f64(m);
        out[1] = ff_f64(a);
        out[2] = ff_f64(b);
        out[3] = (double)n * dtheta0 + ff_f64(e);
        if (DMIN) {
            long long r = shk[0][0], t = shk[1][0];
            for (int w = 1; w < NT / 32; ++w) {
                r = kmin(r, shk[0][w]);
                t = kmin(t, shk[1][w]);
            }
            out[4] = dunkey(r);
            out[5] = dunkey(t);
        } else {
            out[4] = rmin < 3.0e38f ? (double)rmin : 1e300;
            out[5] = tmin < 3.0e38f ? (double)tmin : 1e300;
        }
    }
}

// Block reduction of NodeDiag; thread 0 writes kPartialStride doubles to out.
template <int NT>
__device__ __forceinline__ void block_reduce_diag(NodeDiag d, double* out) {
    __shared__ double sh[6][NT / 32];
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        d.mass += __shfl_down_sync(full, d.mass, off);
        d.jx += __shfl_down_sync(full, d.jx, off);
        d.jy += __shfl_down_sync(full, d.jy, off);
        d.energy += __shfl_down_sync(full, d.energy, off);
        d.rho_min = fmin(d.rho_min, __shfl_down_sync(full, d.rho_min, off));
        d.theta_min = fmin(d.theta_min, __shfl_down_sync(full, d.theta_min, off));
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        sh[0][warp] = d.mass;
        sh[1][warp] = d.jx;
        sh[2][warp] = d.jy;
        sh[3][warp] = d.energy;
        sh[4][warp] = d.rho_min;
        sh[5][warp] = d.theta_min;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double r[6] = {0, 0, 0, 0, 1e300, 1e300};
        for (int w = 0; w < NT / 32; ++w) {
            r[0] += sh[0][w];
            r[1] += sh[1][w];
            r[2] += sh[2][w];
            r[3] += sh[3][w];
            r[4] = fmin(r[4], sh[4][w]);
            r[5] = fmin(r[5], sh[5][w]);
        }
        for (int k = 0; k < 6; ++k) out[k] = r[k];
    }
}

// ---------------------------------------------------------------------------
// Source addresses of the pull: f_p(x - v_p) with periodic wrap or ghosts.
// ---------------------------------------------------------------------------
template <int Q1, int DIM>
struct PullIndex {
    int col[Q1];              // source column per x-velocity
    bool okx[Q1];             // false: the source lies in a fixed-end ghost
    bool leftx[Q1];           // ghost side when !okx
    long long row[DIM == 2 ? Q1 : 1];  // source row offset (elements) per y-velocity

    __device__ __forceinline__ void build(const LatticeParams& P, int x, int y) {
#pragma unroll
        for (int i = 0; i < Q1; ++i) {
            if (P.fixed_ends) {
                int s = x - P.v[i];
                okx[i] = (s >= 0) && (s < P.nx);
                leftx[i] = s < 0;
                col[i] = okx[i] ? s : 0;
            } else {
                int s = x + P.vxm[i];
                col[i] = (s >= P.nx) ? s - P.nx : s;
                okx[i] = true;
                leftx[i] = false;
            }
        }
        if (DIM == 2) {
#pragma unroll
            for (int j = 0; j < (DIM == 2 ? Q1 : 1); ++j) {
                int s = y + P.vym[j];
                s = (s >= P.ny) ? s - P.ny : s;
                row[j] = (long long)s * P.pitch;
            }
        } else {
            row[0] = 0;
        }
    }
};

// ---------------------------------------------------------------------------
// Direct FP64 core.
// ---------------------------------------------------------------------------
template <int Q1, int DIM>
struct DirectCore {
    static constexpr int Q = (DIM == 1) ? Q1 : Q1 * Q1;

    // f holds the pulled populations on entry and the post-collision ones on exit.
    static __device__ __forceinline__ void collide(double (&f)[Q], const LatticeParams& P,
                                                   double& rho_o, double& th_o, double& jx_o,
                                                   double& jy_o, double& e_o) {
        double S[Q1], T[Q1];
        if (DIM == 2) {
#pragma unroll
            for (int i = 0; i < Q1; ++i) {
                double s = 0.0;
#pragma unroll
                for (int j = 0; j < Q1; ++j) s += f[i * Q1 + j];
                S[i] = s;
            }
#pragma unroll
            for (int j = 0; j < Q1; ++j) {
                double t = 0.0;
#pragma unroll
                for (int i = 0; i < Q1; ++i) t += f[i * Q1 + j];
                T[j] = t;
            }
        } else {
#pragma unroll
            for (int i = 0; i < Q1; ++i) S[i] = f[i];
        }
        double rho = 0.0, jx = 0.0, ex = 0.0, jy = 0.0, ey = 0.0;
#pragma unroll
        for (int i = 0; i < Q1; ++i) {
            const double vi = (double)P.v[i];
            rho += S[i];
            jx += vi * S[i];
            ex += vi * vi * S[i];
            if (DIM == 2) {
                jy += vi * T[i];
                ey += vi * vi * T[i];
            }
        }
        const double inv = 1.0 / rho;
        const double ux = jx * inv, uy = jy * inv;
        double th = ((ex + ey) * inv - (ux * ux + uy * uy)) * (1.0 / DIM);
        rho_o = rho;
        th_o = th;
        jx_o = jx;
        jy_o = jy;
        e_o = ex + ey;
        if (P.isothermal) th = P.theta0;

        // mu_n(u, theta) by mu_{n+1} = u mu_n + n theta mu_{n-1}; r = C mu.
        double rx[Q1], ry[Q1];
        {
            double mu[Q1];
            mu[0] = 1.0;
            if (Q1 > 1) mu[1] = ux;
#pragma unroll
            for (int n = 1; n + 1 < Q1; ++n) mu[n + 1] = ux * mu[n] + (double)n * th * mu[n - 1];
#pragma unroll
            for (int i = 0; i < Q1; ++i) {
                double r = 0.0;
#pragma unroll
                for (int n = 0; n < Q1; ++n) r += P.C[i * Q1 + n] * mu[n];
                rx[i] = rho * r;  // rho folded into the x factor
            }
        }
        if (DIM == 2) {
            double mu[Q1];
            mu[0] = 1.0;
            if (Q1 > 1) mu[1] = uy;
#pragma unroll
            for (int n = 1; n + 1 < Q1; ++n) mu[n + 1] = uy * mu[n] + (double)n * th * mu[n - 1];
#pragma unroll
            for (int i = 0; i < Q1; ++i) {
                double r = 0.0;
#pragma unroll
                for (int n = 0; n < Q1; ++n) r += P.C[i * Q1 + n] * mu[n];
                ry[i] = r;
            }
        }
        const double om = P.omega;
#pragma unroll
        for (int i = 0; i < Q1; ++i) {
            if (DIM == 2) {
#pragma unroll
                for (int j = 0; j < Q1; ++j) {
                    const double feq = rx[i] * ry[j];
                    f[i * Q1 + j] = f[i * Q1 + j] + om * (feq - f[i * Q1 + j]);
                }
            } else {
                f[i] = f[i] + om * (rx[i] - f[i]);
            }
        }
    }
};

// 1 / x in FP64 by one step of Householder's third-order iteration y (1 + e + e^2),
// e = 1 - x y, from the hardware's 23-bit estimate: three FP64 instructions, within
// a few 2^-60 of the exact value before the last rounding.  Outside the normal
// range (zero, subnormal, huge, infinite, NaN) the division.
__device__ __forceinline__ double recip_f64(double x) {
    if (((unsigned)__double2hiint(x) & 0x7fffffffu) - 0x00200000u >= 0x7fa00000u) return 1.0 / x;
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// A launch with no more than a few warps per SM quarter.
__device__ __forceinline__ bool few_threads() { return (long long)gridDim.x * gridDim.y * blockDim.x < 1 << 16; }

// Sums of doubles on the integer pipe.  x = fixed_of(f, E) is f in units of 2^(E - 1080), E the largest
// biased exponent among the terms: five bits below the last place of the largest, so that a sum of up to
// 25 of them fits in 63 bits and is exact but for the rounding of each term, 2^-57 of the largest (the
// last bit of a term that may lose bits is set to 1: away from zero where it loses none, to either side
// alike otherwise, and the same for f and -f; an FP64 sum rounds each addition to 2^-53 of itself).
// f64_of_fixed rounds the sum to nearest even, by the conversion instruction, which takes the FP64 pipe, where
// there are few warps (few: their latency counts; 128^2 7.2 -> 6.7 us a step) and by integer ones otherwise
// (1024^2 175 -> 160 us).
__device__ __forceinline__ long long fixed_of(double f, int E) {
    const unsigned hi = (unsigned)__double2hiint(f), lo = (unsigned)__double2loint(f);
    const int e = (int)((hi >> 20) & 0x7ffu), d = min(E - e, 63);
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | (e ? 0x100000u : 0u)) << 32) | lo;
    const long long x = (long long)(((m << 5) >> d) | (d > 5 ? 1ull : 0ull));
    const long long s = (long long)((int)hi >> 31);
    return (x ^ s) - s;
}
__device__ __forceinline__ double f64_of_fixed(long long x, int E, bool few) {
    if (few) {
        const double d = __ll2double_rn(x);
        return x ? __hiloint2double(__double2hiint(d) + (E - 1080) * (1 << 20), __double2loint(d)) : 0.0;
    }
    const long long s = x >> 63;
    unsigned long long m = (unsigned long long)((x ^ s) - s);
    const int lz = __clzll((long long)m);
    m <<= lz & 63;
    const unsigned rem = (unsigned)m & 0x7ffu;
    unsigned long long q = m >> 11;
    q += (rem + ((unsigned)q & 1u)) > 0x400u ? 1u : 0u;
    const unsigned long long bits = q + ((unsigned long long)(unsigned)(E + 5 - lz) << 52);   // q carries the exponent's last unit
    return __longlong_as_double(x ? (long long)(bits | ((unsigned long long)s & 0x8000000000000000ull)) : 0ll);
}

// The product of two fixed-point numbers x / 2^m and y / 2^n as one over 2^(m + n - 63): the high
// word of the product, whose lost bits are replaced by their mean (to either side alike, but for products
// that have none, zero among them).
__device__ __forceinline__ long long fixed_mul(long long x, long long y, long long mean = 1) {
    return (__mul64hi(x, y) << 1) | mean;
}
// For x, y >= 0: without the signed product's corrections.
__device__ __forceinline__ long long fixed_mul_pos(long long x, long long y, long long mean = 1) {
    return (long long)(__umul64hi((unsigned long long)x, (unsigned long long)y) << 1) | mean;
}
// x times a small positive integer: two multiply instructions.
__device__ __forceinline__ long long fixed_times(long long x, unsigned c) {
    const unsigned long long lo = (unsigned long long)(unsigned)x * c;
    return (long long)(((unsigned long long)((unsigned)(x >> 32) * c) << 32) + lo);
}
// |x| in units of 2^-n for |x| < 2^(63 - n); the last bit of one that may lose bits is set to 1, as above.
__device__ __forceinline__ long long fixed_abs(double x, int n) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int e = (int)((hi >> 20) & 0x7ffu), d = min(1085 - n - e, 63);
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | (e ? 0x100000u : 0u)) << 32) | lo;
    return (long long)(((m << 10) >> d) | (e && d > 10 ? 1ull : 0ull));
}

// ---------------------------------------------------------------------------
// FP64 core of the symmetric five-velocity sets (0, +-a, +-b).  The FP64 pipe (two
// lanes per SM and cycle: 64 cycles of an SM quarter for a warp's instruction) bounds
// these steps, so what counts is the number of FP64 instructions: 71 per 2D node against
// 202 with DirectCore (general velocities and coefficients, FP64 status comparisons).
// The moment sums (47 additions in 2D) and the rule run on the integer pipe, which has
// room for 64 instructions beside an FP64 one: the sums in block fixed point (fixed_of),
// the rule in constraint form (plbm_pair.cuh, here for r itself: r_0 = 1 - 2 (E_a + E_b),
// r_(+-a) = E_a +- O_a, r_(+-b) = E_b +- O_b) in 64-bit fixed point, or, outside the range
// of that, in 16 FP64 instructions per axis instead of 31; the velocities and factors
// are constants of the lattice.  Both are nearer to the exact value than FP64 is: against
// 80-bit arithmetic, 200 steps of the 128^2 shear layer leave u_x 6e-15 and u_y 1.4e-13
// off (DirectCore 1.3e-14, 2.3e-13), 40 of a 192^2 one 1.5e-15 and 2.8e-14 (3.8e-15, 6.1e-14).
// Per step: 1024^2 D2Q25 414 us with DirectCore, 301 with all of this core in FP64, 206 with the
// sums on the integer pipe, 152 now (the FP64 pipe busy for 0.79 of it, the integer one for 0.48); 128^2 10.2, 7.95, 7.0, 6.7;
// the 1000-node D1Q5 tube 4.05 -> 3.2 us.  The identities sum r = 1, sum v^2 r = mu_2
// hold by construction, so the global sums drift less: mean density of 1024^2 after
// 40 steps 2e-16 off against 7e-15 (rounded C mu sums), energy 4e-16 against 5e-15.
// ---------------------------------------------------------------------------
template <int DIM>
struct Sym5Core {
    static constexpr int Q = DIM == 1 ? 5 : 25;

    // Products that meet a sum are formed by __dmul_rn, so that every kernel rounds alike.
    // mu_3 = u A and mu_4 = A^2 - 6 theta^2 with A = u^2 + 3 theta; sixth2 = 6 theta^2.
    static __device__ __forceinline__ void axis(const LatticeParams& P, double u, double u2, double th, double sixth2,
                                                double (&r)[5]) {
        const double A = fma(3.0, th, u2);
        const double m2 = u2 + th;
        const double m3 = __dmul_rn(u, A);
        const double m4 = fma(A, A, -sixth2);
        const double yb = fma(-P.da2, u, m3);     // O_b / kOb
        const double ya = fma(-P.dcb, yb, u);     // O_a / kOa
        const double zb = fma(-P.da2, m2, m4);    // E_b / kEb
        const double za = fma(-P.dcb, zb, m2);    // E_a / kEa
        const double Ea = __dmul_rn(za, P.dkEa), Eb = __dmul_rn(zb, P.dkEb);
        r[0] = fma(-2.0, Ea + Eb, 1.0);
        r[1] = fma(P.dkOa, ya, Ea);
        r[2] = fma(-P.dkOa, ya, Ea);
        r[3] = fma(P.dkOb, yb, Eb);
        r[4] = fma(-P.dkOb, yb, Eb);
    }

    // The same in 64-bit fixed point, for |u| < 1/2, 0 < th < 3/2 and |v| <= 3 (fixed_ok; every number then
    // fits): bits after the point in the names.  Nothing keeps fewer than 57 (an FP64 mu_4 has 50 to 52), and r
    // is 13 to 80 times nearer to the exact value before it is rounded to FP64.  O_a and E_a follow from the
    // rounded O_b and E_b, so that sum r = 1, sum v r = u and sum v^2 r = mu_2 hold without a
    // systematic error in the last place, which the steps would add up.  The odd parts are those of |u| with
    // u's sign, and zero for u = 0: a mirrored flow stays the mirrored flow and a fluid at rest exactly at rest.
    struct Theta {
        long long t61, six57;   // theta, 6 theta^2
    };
    static __device__ __forceinline__ bool fixed_ok(const LatticeParams& P, double u, double th) {
        return P.fixed_rule && ((unsigned)__double2hiint(u) & 0x7fffffffu) < 0x3fe00000u &&
               (unsigned)__double2hiint(th) < 0x3ff80000u;
    }
    static __device__ __forceinline__ Theta theta_fixed(double th) {
        Theta t;
        t.t61 = fixed_abs(th, 61);
        t.six57 = (3 * fixed_mul_pos(t.t61, t.t61)) >> 1;
        return t;
    }
    static __device__ __forceinline__ void axis_fixed(const LatticeParams& P, double ud, Theta th, bool few, double (&r)[5]) {
        const long long u60 = fixed_abs(ud, 60), u62 = u60 << 2, some = u60 ? 1 : 0;   // of |u|
        const long long m61 = fixed_mul_pos(u62, u62) + th.t61;      // mu_2
        const long long A60 = (m61 >> 1) + th.t61;                   // u^2 + 3 theta
        const long long yb59 = fixed_mul_pos(u62, A60, some) - fixed_times(u60 >> 1, P.ia2);
        const long long zb57 = fixed_mul_pos(A60, A60) - th.six57 - fixed_times(m61 >> 4, P.ia2);
        const long long Ob0 = fixed_mul(yb59, P.ikOb65, some), Eb = fixed_mul(zb57 << 1, P.ikEb65) << 1;   // 61 bits from here
        const long long w = 2 * (u60 - fixed_times(Ob0, P.ib));   // 2 a O_a
        const long long Oa0 = P.ia2 == 1 ? w >> 1 : fixed_mul(w, P.ikOa63, w ? 1 : 0);
        const long long sign = (long long)(__double2hiint(ud) >> 31);
        const long long Oa = (Oa0 ^ sign) - sign, Ob = (Ob0 ^ sign) - sign;
        const long long Ea = fixed_mul(m61 - fixed_times(Eb, P.ib2x2), P.ikEa63);
        r[0] = f64_of_fixed((1ll << 61) - 2 * (Ea + Eb), 1019, few);
        r[1] = f64_of_fixed(Ea + Oa, 1019, few);
        r[2] = f64_of_fixed(Ea - Oa, 1019, few);
        r[3] = f64_of_fixed(Eb + Ob, 1019, few);
        r[4] = f64_of_fixed(Eb - Ob, 1019, few);
    }

    // r of both axes (ry: 2D).
    static __device__ __forceinline__ void rule(const LatticeParams& P, double ux, double uy, double th, bool few,
                                                double (&rx)[5], double (&ry)[5]) {
        if (fixed_ok(P, ux, th) && (DIM == 1 || fixed_ok(P, uy, th))) {
            const Theta t = theta_fixed(th);
            axis_fixed(P, ux, t, few, rx);
            if constexpr (DIM == 2) axis_fixed(P, uy, t, few, ry);
        } else {
            const double sixth2 = __dmul_rn(__dmul_rn(6.0, th), th);
            axis(P, ux, __dmul_rn(ux, ux), th, sixth2, rx);
            if constexpr (DIM == 2) axis(P, uy, __dmul_rn(uy, uy), th, sixth2, ry);
        }
    }

    // What the moments need of the populations: rho and per axis the differences and sums of the
    // columns of opposite velocities (dp = S_1 - S_2, dq = S_3 - S_4; ep, eq: the sums over both axes).
    struct Sums {
        double rho, dpx, dqx, dpy, dqy, ep, eq;
    };
    static __device__ __forceinline__ Sums sums_f64(const double (&f)[Q]) {
        double S[5];
        Sums o;
        if constexpr (DIM == 2) {
            double T[5];
#pragma unroll
            for (int i = 0; i < 5; ++i)
                S[i] = (f[5 * i] + (f[5 * i + 1] + f[5 * i + 2])) + (f[5 * i + 3] + f[5 * i + 4]);
#pragma unroll
            for (int j = 1; j < 5; ++j) T[j] = (f[j] + (f[5 + j] + f[10 + j])) + (f[15 + j] + f[20 + j]);
            o.dpy = T[1] - T[2];
            o.dqy = T[3] - T[4];
            o.ep = T[1] + T[2];
            o.eq = T[3] + T[4];
        } else {
#pragma unroll
            for (int i = 0; i < 5; ++i) S[i] = f[i];
            o.dpy = o.dqy = o.ep = o.eq = 0.0;
        }
        const double Sp = S[1] + S[2], Sq = S[3] + S[4];
        o.rho = S[0] + Sp + Sq;
        o.dpx = S[1] - S[2];
        o.dqx = S[3] - S[4];
        o.ep = DIM == 2 ? Sp + o.ep : Sp;
        o.eq = DIM == 2 ? Sq + o.eq : Sq;
        return o;
    }

    static __device__ __forceinline__ Sums sums(const double (&f)[Q], bool few) {
        if constexpr (DIM == 2) {
            unsigned top = 0u;
#pragma unroll
            for (int p = 0; p < Q; ++p) top = max(top, (unsigned)__double2hiint(f[p]) & 0x7fffffffu);
            const int E = (int)(top >> 20);
            if (E < 64 || E > 1900) return sums_f64(f);   // NaN, infinite, near either end of the range
            long long S[5], T[5];
#pragma unroll
            for (int i = 0; i < 5; ++i)
#pragma unroll
                for (int j = 0; j < 5; ++j) {
                    const long long x = fixed_of(f[5 * i + j], E);
                    S[i] = j ? S[i] + x : x;
                    if (j) T[j] = i ? T[j] + x : x;
                }
            const long long Sp = S[1] + S[2], Sq = S[3] + S[4];
            auto out = [&](long long x) { return f64_of_fixed(x, E, few); };
            return {out(S[0] + Sp + Sq),      out(S[1] - S[2]),          out(S[3] - S[4]),         out(T[1] - T[2]),
                    out(T[3] - T[4]),         out(Sp + (T[1] + T[2])),   out(Sq + (T[3] + T[4]))};
        } else {
            return sums_f64(f);
        }
    }

    static __device__ __forceinline__ void moments(const double (&f)[Q], const LatticeParams& P, bool few, double& rho,
                                                   double& th, double& jx, double& jy, double& e, double& ux, double& uy) {
        const Sums s = sums(f, few);
        rho = s.rho;
        jx = fma(P.da, s.dpx, __dmul_rn(P.db, s.dqx));
        jy = DIM == 2 ? fma(P.da, s.dpy, __dmul_rn(P.db, s.dqy)) : 0.0;
        e = fma(P.da2, s.ep, __dmul_rn(P.db2, s.eq));
        const double inv = recip_f64(rho);
        ux = __dmul_rn(jx, inv), uy = __dmul_rn(jy, inv);
        const double ux2 = __dmul_rn(ux, ux), uy2 = __dmul_rn(uy, uy);
        th = fma(e, inv, -(DIM == 2 ? ux2 + uy2 : ux2));
        if constexpr (DIM == 2) th = __dmul_rn(th, 0.5);
    }

    // few: see f64_of_fixed; one branch around the whole, as one at each conversion costs more than it gains
    static __device__ __forceinline__ void collide(double (&f)[Q], const LatticeParams& P, double& rho_o, double& th_o,
                                                   double& jx_o, double& jy_o, double& e_o) {
        if (DIM == 2 && few_threads())   // 1D (1000 nodes): 1.80 us a step without the branch, 1.83 with it
            collide_as(f, P, true, rho_o, th_o, jx_o, jy_o, e_o);
        else
            collide_as(f, P, false, rho_o, th_o, jx_o, jy_o, e_o);
    }
    static __device__ __forceinline__ void collide_as(double (&f)[Q], const LatticeParams& P, bool few, double& rho_o,
                                                      double& th_o, double& jx_o, double& jy_o, double& e_o) {
        double rho, th, ux, uy;
        moments(f, P, few, rho, th, jx_o, jy_o, e_o, ux, uy);
        rho_o = rho;
        th_o = th;
        if (P.isothermal) th = P.theta0;
        const double om = P.omega;
        double rx[5], ry[5];
        rule(P, ux, uy, th, few, rx, ry);
        if constexpr (DIM == 2) {
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                const double X = __dmul_rn(rho, rx[i]);
#pragma unroll
                for (int j = 0; j < 5; ++j)
                    f[5 * i + j] = fma(om, fma(X, ry[j], -f[5 * i + j]), f[5 * i + j]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 5; ++i) f[i] = fma(om, fma(rho, rx[i], -f[i]), f[i]);
        }
    }
};

// ---------------------------------------------------------------------------
// Deviation FP32 core (see the file header for the algebra).
// ---------------------------------------------------------------------------
template <int Q1, int DIM>
struct DeviationCore {
    static constexpr int Q = (DIM == 1) ? Q1 : Q1 * Q1;

    // dmu_n = mu_n(u, theta) - mu_n(0, theta0), dr = C dmu, for one axis.
    static __device__ __forceinline__ void axis(const LatticeParams& P, float u, float th,
                                                float dth, float (&dr)[Q1]) {
        float dmu[Q1];
        dmu[0] = 0.0f;
        if (Q1 > 1) dmu[1] = u;
#pragma unroll
        for (int n = 1; n + 1 < Q1; ++n) {
            const float fn = (float)n;
            dmu[n + 1] = u * (P.mu0f[n] + dmu[n]) + fn * th * dmu[n - 1] + fn * dth * P.mu0f[n - 1];
        }
        // C carried as Cf + Cf_lo: a single FP32 rounding of c_ij would break the
        // moment identities of Eq. (eq:rdr) by ~1e-8 in a fixed direction, which
        // the collision turns into a systematic momentum source.
#pragma unroll
        for (int i = 0; i < Q1; ++i) {
            float r = 0.0f, rl = 0.0f;
#pragma unroll
            for (int n = 1; n < Q1; ++n) {
                r = fmaf(P.Cf[i * Q1 + n], dmu[n], r);
                rl = fmaf(P.Cf_lo[i * Q1 + n], dmu[n], rl);
            }
            dr[i] = r + rl;
        }
    }

    // g holds pulled deviations on entry and post-collision deviations on exit.
    static __device__ __forceinline__ void collide(float (&g)[Q], const LatticeParams& P,
                                                   float& drho_o, float& th_o, float& jx_o,
                                                   float& jy_o, float& e_o) {
        float S[Q1], T[Q1];
        if (DIM == 2) {
#pragma unroll
            for (int i = 0; i < Q1; ++i) {
                float s = 0.0f;
#pragma unroll
                for (int j = 0; j < Q1; ++j) s += g[i * Q1 + j];
                S[i] = s;
            }
#pragma unroll
            for (int j = 0; j < Q1; ++j) {
                float t = 0.0f;
#pragma unroll
                for (int i = 0; i < Q1; ++i) t += g[i * Q1 + j];
                T[j] = t;
            }
        } else {
#pragma unroll
            for (int i = 0; i < Q1; ++i) S[i] = g[i];
        }
        float drho = 0.0f, jx = 0.0f, ex = 0.0f, jy = 0.0f, ey = 0.0f;
#pragma unroll
        for (int i = 0; i < Q1; ++i) {
            const float vi = (float)P.v[i];
            drho += S[i];
            jx += vi * S[i];
            ex += vi * vi * S[i];
            if (DIM == 2) {
                jy += vi * T[i];
                ey += vi * vi * T[i];
            }
        }
        const float rho = 1.0f + drho;
        const float inv = 1.0f / rho;
        const float ux = jx * inv, uy = jy * inv;
        const float dthp = (((ex + ey) - (float)DIM * P.theta0f * drho) * inv - (ux * ux + uy * uy)) *
                           (1.0f / (float)DIM);
        drho_o = drho;
        th_o = P.theta0f + dthp;
        jx_o = jx;
        jy_o = jy;
        e_o = ex + ey;
        const float dth = P.isothermal ? 0.0f : dthp;
        const float th = P.theta0f + dth;

        float drx[Q1];
        axis(P, ux, th, dth, drx);
        const float om = P.omegaf;
        if (DIM == 2) {
            float dry[Q1], ry[Q1];
            axis(P, uy, th, dth, dry);
#pragma unroll
            for (int j = 0; j < Q1; ++j) ry[j] = P.w1f[j] + dry[j];
#pragma unroll
            for (int i = 0; i < Q1; ++i) {
                const float a = rho * drx[i];
                const float b = rho * P.w1f[i];
#pragma unroll
                for (int j = 0; j < Q1; ++j) {
                    const int p = i * Q1 + j;
                    const float geq = drho * P.W0f[p] + (a * ry[j] + b * dry[j]);
                    g[p] = g[p] + om * (geq - g[p]);
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < Q1; ++i) {
                const float geq = drho * P.w1f[i] + rho * drx[i];
                g[i] = g[i] + om * (geq - g[i]);
            }
        }
    }
};

// ---------------------------------------------------------------------------
// One node of the fused stream-and-collide step: pull, collide, store; the
// node's contribution to the diagnostics when REDUCE (d for FP64 storage, df
// for 16/32-bit storage).  Shared by the single-lattice kernel and the batched
// persistent kernel, so both give bit-identical states.
// ---------------------------------------------------------------------------
template <typename S, int Q1, int DIM, bool REDUCE>
__device__ __forceinline__ void node_update(const LatticeParams& P, const S* src, S* __restrict__ dst, int x, int y, NodeDiag& d, NodeDiagF& df) {
    constexpr int Q = (DIM == 1) ? Q1 : Q1 * Q1;
    PullIndex<Q1, DIM> ix;
    ix.build(P, x, y);
    const long long here = (long long)y * P.pitch + x;
    if constexpr (!Storage<S>::kDeviation && sizeof(S) == 8) {
        // FP64: direct core
        double f[Q];
#pragma unroll
        for (int i = 0; i < Q1; ++i) {
#pragma unroll
            for (int j = 0; j < (DIM == 2 ? Q1 : 1); ++j) {
                const int p = (DIM == 2) ? i * Q1 + j : i;
                f[p] = ix.okx[i] ? Storage<S>::load(src + p * P.plane + ix.row[j] + ix.col[i])
                                 : (ix.leftx[i] ? P.ghostL[p] : P.ghostR[p]);
            }
        }
        double rho, th, jx, jy, e;
        bool sym5 = false;   // uniform over a lattice
        if constexpr (Q1 == 5) {
            sym5 = P.sym5;
            if (sym5) Sym5Core<DIM>::collide(f, P, rho, th, jx, jy, e);
        }
        if (!sym5) DirectCore<Q1, DIM>::collide(f, P, rho, th, jx, jy, e);
        flag_status_f64(P, rho, th);
        if (step_late<DIM>()) step_begin();
        if (REDUCE) {
            d.mass = rho;
            d.jx = jx;
            d.jy = jy;
            d.energy = e;
            d.rho_min = rho;
            d.theta_min = th;
        }
#pragma unroll
        for (int p = 0; p < Q; ++p) Storage<S>::store(dst + p * P.plane + here, f[p]);
    } else {
        // FP32 arithmetic on deviations g = f - w0
        float g[Q];
#pragma unroll
        for (int i = 0; i < Q1; ++i) {
#pragma unroll
            for (int j = 0; j < (DIM == 2 ? Q1 : 1); ++j) {
                const int p = (DIM == 2) ? i * Q1 + j : i;
                if (ix.okx[i]) {
                    float s = Storage<S>::load(src + p * P.plane + ix.row[j] + ix.col[i]);
                    g[p] = Storage<S>::kDeviation ? s : s - P.W0f[p];
                } else {
                    g[p] = ix.leftx[i] ? P.ghostLg[p] : P.ghostRg[p];
                }
            }
        }
        float drho, th, jx, jy, e;
        DeviationCore<Q1, DIM>::collide(g, P, drho, th, jx, jy, e);
        flag_status<float>(P, 1.0f + drho, th);
        if (REDUCE) {
            df.dmass = FF{drho, 0.0f};
            df.jx = FF{jx, 0.0f};
            df.jy = FF{jy, 0.0f};
            df.denergy = FF{e, 0.0f};
            df.rho_min = 1.0f + drho;
            df.theta_min = th;
            df.n = 1.0f;
        }
#pragma unroll
        for (int p = 0; p < Q; ++p) {
            const float out = Storage<S>::kDeviation ? g[p] : g[p] + P.W0f[p];
            Storage<S>::store(dst + p * P.plane + here, out);
        }
    }
}

// ---------------------------------------------------------------------------
// The fused stream-and-collide kernel.
// grid = (ceil(nx / blockDim.x), ny), blockDim.x threads along x (kBlockX when
// REDUCE, whose per-block records assume it).
// ---------------------------------------------------------------------------
template <typename S, int Q1, int DIM, bool REDUCE>
__global__ void __launch_bounds__(kBlockX)
k_stream_collide(const __grid_constant__ LatticeParams P, const S* src, S* __restrict__ dst) {
    if (sizeof(S) < 8 || !step_late<DIM>()) step_begin();
    const int x = blockIdx.x * (REDUCE ? kBlockX : (int)blockDim.x) + threadIdx.x;
    const int y = blockIdx.y;
    step_wait();

    NodeDiag d;       // FP64 storage
    NodeDiagF df;     // 16/32-bit storage
    if (REDUCE) {
        diag_zero(d);
        diagf_zero(df);
    }
    if (x < P.nx) node_update<S, Q1, DIM, REDUCE>(P, src, dst, x, y, d, df);
    if (REDUCE) {
        const int blk = blockIdx.y * gridDim.x + blockIdx.x;
        if constexpr (!Storage<S>::kDeviation && sizeof(S) == 8)
            block_reduce_diag<kBlockX>(d, P.partials + (long long)blk * kPartialStride);
        else
            block_reduce_diagf<kBlockX>(df, (double)DIM * P.theta0, P.partials + (long long)blk * kPartialStride);
    }
}

// ---------------------------------------------------------------------------
// Several steps of a 1D lattice in one launch.  A step of a short lattice (the
// 1000-node tube) is one warp's work per SM, and of its 3.2 us only 0.6 are the
// arithmetic; the rest is the launch and the way to memory and back.  Here a warp
// loads the 32 nodes around m = 32 - 2 w steps output nodes (w = max|v|), keeps
// them in registers, pulls by shuffles and steps them `steps` times; the outer w
// lanes of each side hold no valid state after each step and are dropped.  Lanes
// beyond a fixed end hold the end's populations, which never change.  The arithmetic
// done twice is free while every warp has an SM quarter to itself; steps_per_launch
// weighs it against the launches saved.
// ---------------------------------------------------------------------------
template <typename S>
struct Node1 {   // how one node's populations live between two steps
    using A = float;
    static __device__ __forceinline__ A load(const S* p) { return Storage<S>::load(p); }
    static __device__ __forceinline__ A stored(A v) {   // the value a store and a load would give
        S s;
        Storage<S>::store(&s, v);
        return v_of(s);
    }
    static __device__ __forceinline__ A v_of(float s) { return s; }
    static __device__ __forceinline__ A v_of(__half s) { return __half2float(s); }
    static __device__ __forceinline__ A v_of(__nv_bfloat16 s) { return __bfloat162float(s); }
};
template <>
struct Node1<double> {
    using A = double;
    static __device__ __forceinline__ A load(const double* p) { return load_state(p); }
    static __device__ __forceinline__ A stored(A v) { return v; }
};

constexpr int kWarps1 = 4;   // most independent warps per block, one per SM quarter

template <typename S, int Q1, bool SYM5>
__global__ void __launch_bounds__(32 * kWarps1) k_steps1(const __grid_constant__ LatticeParams P,
                                                         const S* src, S* __restrict__ dst, int steps, int w,
                                                         int m) {
    using A = typename Node1<S>::A;
    const int lane = threadIdx.x & 31;
    const long long first = (long long)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * m;   // first output node
    if (first >= P.nx) return;
    const int x = (int)first + lane - w * steps;
    const bool inside = x >= 0 && x < P.nx;
    A f[Q1];
    step_wait();
    if (!inside && P.fixed_ends) {
#pragma unroll
        for (int i = 0; i < Q1; ++i) {
            if constexpr (sizeof(S) == 8) f[i] = x < 0 ? P.ghostL[i] : P.ghostR[i];
            else f[i] = x < 0 ? P.ghostLg[i] : P.ghostRg[i];
        }
    } else {
        int s = x % P.nx;
        s = s < 0 ? s + P.nx : s;
#pragma unroll
        for (int i = 0; i < Q1; ++i) f[i] = Node1<S>::load(src + i * P.plane + s);
    }
    for (int k = 1; k <= steps; ++k) {
        A g[Q1];
#pragma unroll
        for (int i = 0; i < Q1; ++i) g[i] = SYM5 && i == 0 ? f[0] : __shfl_sync(0xffffffffu, f[i], lane - P.v[i]);
        A rho, th, jx, jy, e;
        if constexpr (sizeof(S) == 8) {
            if constexpr (SYM5) Sym5Core<1>::collide(g, P, rho, th, jx, jy, e);
            else DirectCore<Q1, 1>::collide(g, P, rho, th, jx, jy, e);
        } else {
            A drho;
            DeviationCore<Q1, 1>::collide(g, P, drho, th, jx, jy, e);
            rho = 1.0f + drho;
        }
        if (inside || !P.fixed_ends) {
            if (lane >= w * k && lane < 32 - w * k) {
                if constexpr (sizeof(S) == 8) flag_status_f64(P, rho, th);
                else flag_status<float>(P, rho, th);
            }
#pragma unroll
            for (int i = 0; i < Q1; ++i) f[i] = Node1<S>::stored(g[i]);
        }
    }
    step_begin();   // after the arithmetic
    if (inside && lane >= w * steps && lane < w * steps + m) {
#pragma unroll
        for (int i = 0; i < Q1; ++i) Storage<S>::store(dst + i * P.plane + x, f[i]);
    }
}

inline int halo1(const LatticeParams& P) {
    int w = 0;
    for (int i = 0; i < P.q1; ++i) w = P.v[i] > w ? P.v[i] : (-P.v[i] > w ? -P.v[i] : w);
    return w;
}

template <typename S>
cudaError_t launch_steps1_t(const LatticeParams& P, const void* src, void* dst, int steps, cudaStream_t stream) {
    const int w = halo1(P), m = 32 - 2 * w * steps;
    if (P.dim != 1 || steps < 1 || m < 1) return cudaErrorInvalidValue;
    // FP64 warps do best spread over the SMs (1000 nodes 1.87 us a step against 2.00), the
    // others in few blocks (100,000 nodes 1.55 us against 3.34)
    const int warps = sizeof(S) == 8 ? 1 : kWarps1;
    const int blocks = ((P.nx + m - 1) / m + warps - 1) / warps;
    const S* s = static_cast<const S*>(src);
    S* t = static_cast<S*>(dst);
    if constexpr (sizeof(S) == 8) {
        if (P.sym5) return launch_dependent(true, k_steps1<S, 5, true>, blocks, 32 * warps, stream, P, s, t, steps, w, m);
    }
    switch (P.q1) {
        case 3: return launch_dependent(true, k_steps1<S, 3, false>, blocks, 32 * warps, stream, P, s, t, steps, w, m);
        case 4: return launch_dependent(true, k_steps1<S, 4, false>, blocks, 32 * warps, stream, P, s, t, steps, w, m);
        case 5: return launch_dependent(true, k_steps1<S, 5, false>, blocks, 32 * warps, stream, P, s, t, steps, w, m);
        case 6: return launch_dependent(true, k_steps1<S, 6, false>, blocks, 32 * warps, stream, P, s, t, steps, w, m);
        case 7: return launch_dependent(true, k_steps1<S, 7, false>, blocks, 32 * warps, stream, P, s, t, steps, w, m);
        case 8: return launch_dependent(true, k_steps1<S, 8, false>, blocks, 32 * warps, stream, P, s, t, steps, w, m);
    }
    return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// Batched persistent step over 2D lattices in the plain layout (one node per
// thread): odd row counts, FP64 storage, isothermal models and velocity sets
// other than (0, +-a, +-b), which the row-paired batched kernel does not take.
// A tile is kBlockX nodes of one row of one lattice; all such lattices' tiles
// form one list that CTA c walks as c, c + G, c + 2G, ... (G CTAs), reading
// each tile's lattice from tile_inst and that lattice's parameters from the
// device table (cached by L1).  Per node it runs node_update, as the
// single-lattice kernel does.
// ---------------------------------------------------------------------------
template <typename S, int Q1>
__global__ void __launch_bounds__(kBlockX)
k_batch_node(const LatticeParams* __restrict__ inst, const NodeSpan* __restrict__ span, int total_tiles,
             int parity, const unsigned short* __restrict__ tile_inst) {
    NodeDiag d;
    NodeDiagF df;
    for (int t = blockIdx.x; t < total_tiles; t += gridDim.x) {
        const int i = tile_inst[t];
        const NodeSpan sp = span[i];
        const LatticeParams& P = inst[i];
        const int local = t - sp.tile_begin;
        const int y = local / sp.tiles_x;
        const int x = (local - y * sp.tiles_x) * kBlockX + threadIdx.x;
        if (x < sp.nx)
            node_update<S, Q1, 2, false>(P, static_cast<const S*>(sp.f[parity]), static_cast<S*>(sp.f[parity ^ 1]),
                                         x, y, d, df);
    }
}

template <typename S>
cudaError_t launch_step_t(const LatticeParams& P, const void* src, void* dst, bool reduce,
                          cudaStream_t stream) {
    if (P.paired) return cudaErrorInvalidValue;  // row-paired layouts use k_stream_collide_pair
    // Small lattices (fewer than two blocks per SM): 32-thread blocks spread the
    // nodes over four times as many SMs (GB300's FP64 rate per SM is low).
    int bx = kBlockX;
    if (!reduce && (long long)((P.nx + kBlockX - 1) / kBlockX) * P.ny < 2LL * device_sm_count()) bx = 32;
    dim3 grid((P.nx + bx - 1) / bx, P.ny);
    dim3 block(bx);
    constexpr bool f64 = sizeof(S) == 8;
    const S* s = static_cast<const S*>(src);
    S* t = static_cast<S*>(dst);
#define PLBM_LAUNCH(Q1v, DIMv)                                                              \
    if (P.q1 == Q1v && P.dim == DIMv) {                                                     \
        const auto kernel = reduce ? k_stream_collide<S, Q1v, DIMv, true> : k_stream_collide<S, Q1v, DIMv, false>;  \
        if (f64 && (DIMv == 1 || bx == 32))                                                                        \
            return launch_dependent(DIMv == 1 || Q1v <= 5, kernel, grid, block, stream, P, s, t);                  \
        return launch_by_waves(f64 ? (long long)grid.x * grid.y * bx : (long long)P.nx * P.ny, f64 ? 3 : 5, f64 ? 1 : 6, kernel,  \
                               grid, block, stream, P, s, t);                                                      \
    }
    PLBM_LAUNCH(3, 1)
    PLBM_LAUNCH(4, 1)
    PLBM_LAUNCH(5, 1)
    PLBM_LAUNCH(6, 1)
    PLBM_LAUNCH(7, 1)
    PLBM_LAUNCH(8, 1)
    PLBM_LAUNCH(3, 2)
    PLBM_LAUNCH(4, 2)
    PLBM_LAUNCH(5, 2)
    PLBM_LAUNCH(6, 2)
    PLBM_LAUNCH(7, 2)
    PLBM_LAUNCH(8, 2)
#undef PLBM_LAUNCH
    return cudaErrorInvalidValue;
}

// Batched plain-layout step of every lattice of one (precision, q1) group.
template <typename S>
cudaError_t launch_batch_node_t(int q1, const LatticeParams* inst, const NodeSpan* span, int total_tiles,
                                int ctas, int parity, const unsigned short* tile_inst, cudaStream_t stream) {
    switch (q1) {
        case 3: k_batch_node<S, 3><<<ctas, kBlockX, 0, stream>>>(inst, span, total_tiles, parity, tile_inst); break;
        case 4: k_batch_node<S, 4><<<ctas, kBlockX, 0, stream>>>(inst, span, total_tiles, parity, tile_inst); break;
        case 5: k_batch_node<S, 5><<<ctas, kBlockX, 0, stream>>>(inst, span, total_tiles, parity, tile_inst); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename S>
cudaError_t batch_node_occupancy_t(int q1, int* blocks_per_sm) {
    switch (q1) {
        case 3: return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_batch_node<S, 3>, kBlockX, 0);
        case 4: return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_batch_node<S, 4>, kBlockX, 0);
        case 5: return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_batch_node<S, 5>, kBlockX, 0);
    }
    return cudaErrorInvalidValue;
}

}  // namespace plbm
