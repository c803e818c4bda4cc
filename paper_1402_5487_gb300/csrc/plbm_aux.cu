// Initial equilibrium, moments of the stored state, deterministic reductions and
// population import/export.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "plbm.h"
#include "plbm_pair.cuh"

namespace plbm {

cudaError_t launch_step_f64(const LatticeParams&, const void*, void*, bool, cudaStream_t);
cudaError_t launch_step_f32(const LatticeParams&, const void*, void*, bool, cudaStream_t);
cudaError_t launch_step_f16(const LatticeParams&, const void*, void*, bool, cudaStream_t);
cudaError_t launch_step_bf16(const LatticeParams&, const void*, void*, bool, cudaStream_t);

bool two_steps_f32(const LatticeParams&);
bool two_steps_f16(const LatticeParams&);
bool two_steps_bf16(const LatticeParams&);
cudaError_t launch_two_steps_f32(const LatticeParams&, const void*, void*, cudaStream_t);
cudaError_t launch_two_steps_f16(const LatticeParams&, const void*, void*, cudaStream_t);
cudaError_t launch_two_steps_bf16(const LatticeParams&, const void*, void*, cudaStream_t);
cudaError_t launch_steps1_f64(const LatticeParams&, const void*, void*, int, cudaStream_t);
cudaError_t launch_steps1_f32(const LatticeParams&, const void*, void*, int, cudaStream_t);
cudaError_t launch_steps1_f16(const LatticeParams&, const void*, void*, int, cudaStream_t);
cudaError_t launch_steps1_bf16(const LatticeParams&, const void*, void*, int, cudaStream_t);

cudaError_t launch_batch_f32(const PairParams*, int, int, int, int, int, const unsigned short*, cudaStream_t);
cudaError_t launch_batch_f16(const PairParams*, int, int, int, int, int, const unsigned short*, cudaStream_t);
cudaError_t launch_batch_bf16(const PairParams*, int, int, int, int, int, const unsigned short*, cudaStream_t);
cudaError_t batch_occupancy_f32(int, int*);
cudaError_t batch_occupancy_f16(int, int*);
cudaError_t batch_occupancy_bf16(int, int*);

cudaError_t launch_batch_node_f64(int, const LatticeParams*, const NodeSpan*, int, int, int, const unsigned short*,
                                  cudaStream_t);
cudaError_t launch_batch_node_f32(int, const LatticeParams*, const NodeSpan*, int, int, int, const unsigned short*,
                                  cudaStream_t);
cudaError_t launch_batch_node_f16(int, const LatticeParams*, const NodeSpan*, int, int, int, const unsigned short*,
                                  cudaStream_t);
cudaError_t launch_batch_node_bf16(int, const LatticeParams*, const NodeSpan*, int, int, int, const unsigned short*,
                                   cudaStream_t);
cudaError_t batch_node_occupancy_f64(int, int*);
cudaError_t batch_node_occupancy_f32(int, int*);
cudaError_t batch_node_occupancy_f16(int, int*);
cudaError_t batch_node_occupancy_bf16(int, int*);

cudaError_t launch_batch_node(int prec, int q1, const LatticeParams* inst, const NodeSpan* span, int total_tiles,
                              int ctas, int parity, const unsigned short* tile_inst, cudaStream_t stream) {
    switch (prec) {
        case kF64: return launch_batch_node_f64(q1, inst, span, total_tiles, ctas, parity, tile_inst, stream);
        case kF32: return launch_batch_node_f32(q1, inst, span, total_tiles, ctas, parity, tile_inst, stream);
        case kF16Dev: return launch_batch_node_f16(q1, inst, span, total_tiles, ctas, parity, tile_inst, stream);
        case kBF16Dev: return launch_batch_node_bf16(q1, inst, span, total_tiles, ctas, parity, tile_inst, stream);
    }
    return cudaErrorInvalidValue;
}

cudaError_t batch_node_occupancy(int prec, int q1, int* blocks_per_sm) {
    switch (prec) {
        case kF64: return batch_node_occupancy_f64(q1, blocks_per_sm);
        case kF32: return batch_node_occupancy_f32(q1, blocks_per_sm);
        case kF16Dev: return batch_node_occupancy_f16(q1, blocks_per_sm);
        case kBF16Dev: return batch_node_occupancy_bf16(q1, blocks_per_sm);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_batch(int prec, const PairParams* inst, int ninst, int total_tiles, int block_x,
                         int ctas, int parity, const unsigned short* tile_inst, cudaStream_t stream) {
    switch (prec) {
        case kF32: return launch_batch_f32(inst, ninst, total_tiles, block_x, ctas, parity, tile_inst, stream);
        case kF16Dev: return launch_batch_f16(inst, ninst, total_tiles, block_x, ctas, parity, tile_inst, stream);
        case kBF16Dev: return launch_batch_bf16(inst, ninst, total_tiles, block_x, ctas, parity, tile_inst, stream);
    }
    return cudaErrorInvalidValue;
}

cudaError_t batch_occupancy(int prec, int block_x, int* blocks_per_sm) {
    switch (prec) {
        case kF32: return batch_occupancy_f32(block_x, blocks_per_sm);
        case kF16Dev: return batch_occupancy_f16(block_x, blocks_per_sm);
        case kBF16Dev: return batch_occupancy_bf16(block_x, blocks_per_sm);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_step(int prec, const LatticeParams& P, const void* src, void* dst, bool reduce,
                        cudaStream_t stream) {
    switch (prec) {
        case kF64: return launch_step_f64(P, src, dst, reduce, stream);
        case kF32: return launch_step_f32(P, src, dst, reduce, stream);
        case kF16Dev: return launch_step_f16(P, src, dst, reduce, stream);
        case kBF16Dev: return launch_step_bf16(P, src, dst, reduce, stream);
    }
    return cudaErrorInvalidValue;
}

// 1D: a launch of k steps takes `launch` us (launch, load, store) plus k times a warp's
// arithmetic, which four warps per SM do side by side (one per SM quarter; an FP64
// instruction occupies a quarter for 64 cycles) and further ones in rounds.  The
// constants are fitted to D1Q5 {0, +-1, +-3}, periodic, us per step with one step per
// launch (graph replays) and with the k this rule takes: FP64 1000 nodes 4.04 (3.2
// before the symmetric core alone) -> 1.87, 20,000 nodes 5.46 -> 3.54, 100,000 nodes
// 18.95 -> 14.70 (k = 1); FP32 1.74 -> 0.53, 1.87 -> 0.91, 2.32 -> 1.55.  Of 420 drawn lattices (16 to 4 * 10^6 nodes,
// three to eight velocities of up to 7) none is then more than 7 % slower than by single steps and the mean is 0.57 of them
// (with one pair of constants for all numbers of velocities 1.33 at worst: eight velocities, 2.8 * 10^6 nodes).
int steps_per_launch(int prec, const LatticeParams& P) {
    if (P.dim != 1)   // plbm_fuse.cuh
        return (prec == kF32 && two_steps_f32(P)) || (prec == kF16Dev && two_steps_f16(P)) || (prec == kBF16Dev && two_steps_bf16(P)) ? 2 : 1;
    const int w = halo1(P), sms = device_sm_count();
    const double launch = 1.5, latency = prec == kF64 ? 1.5 : 0.25;
    // a round of FP32 arithmetic by the number of velocities, in k_stream_collide and in k_steps1 (80 rounds and more)
    static const double single[6] = {0.173, 0.183, 0.207, 0.269, 0.316, 0.364}, several[6] = {0.093, 0.109, 0.129, 0.153, 0.186, 0.214};
    auto time = [&](int k) {   // per step
        const int m = k == 1 ? 32 : 32 - 2 * w * k;
        const long long warps = (P.nx + m - 1) / m, rounds = (warps + 4LL * sms - 1) / (4LL * sms);
        const double round = prec == kF64 ? 1.5 : k == 1 ? single[P.q1 - 3] : several[P.q1 - 3] * (rounds < 80 ? 0.75 + rounds / 320.0 : 1.0);
        const double work = rounds * round;
        const double step = work > latency ? work : latency;
        return (launch + k * step) / k;
    };
    int best = 1;
    for (int k = 2; k <= 16 && 32 - 2 * w * k >= 2; k *= 2)   // divisors of half a captured run of 32 steps
        if (time(k) < (best == 1 ? 0.95 : 1.0) * time(best)) best = k;
    return best;
}

cudaError_t launch_steps(int prec, const LatticeParams& P, const void* src, void* dst, int steps, cudaStream_t stream) {
    if (P.dim != 1) {
        if (steps != 2) return cudaErrorInvalidValue;
        switch (prec) {
            case kF32: return launch_two_steps_f32(P, src, dst, stream);
            case kF16Dev: return launch_two_steps_f16(P, src, dst, stream);
            case kBF16Dev: return launch_two_steps_bf16(P, src, dst, stream);
        }
        return cudaErrorInvalidValue;
    }
    switch (prec) {
        case kF64: return launch_steps1_f64(P, src, dst, steps, stream);
        case kF32: return launch_steps1_f32(P, src, dst, steps, stream);
        case kF16Dev: return launch_steps1_f16(P, src, dst, steps, stream);
        case kBF16Dev: return launch_steps1_bf16(P, src, dst, steps, stream);
    }
    return cudaErrorInvalidValue;
}

// FP64 equilibrium of one node, Eq. (eq:eqdist) with Eq. (eq:rdr) per axis and
// the tensor product of Sec. 2.1.  out[p], p = ix*q1 + iy.
__device__ void node_feq_f64(const LatticeParams& P, double rho, double ux, double uy, double th,
                             double* out) {
    double rx[kMaxQ1], ry[kMaxQ1], mu[kMaxQ1];
    const int q1 = P.q1;
    for (int a = 0; a < P.dim; ++a) {
        const double u = (a == 0) ? ux : uy;
        mu[0] = 1.0;
        mu[1] = u;
        for (int n = 1; n + 1 < q1; ++n) mu[n + 1] = u * mu[n] + (double)n * th * mu[n - 1];
        for (int i = 0; i < q1; ++i) {
            double r = 0.0;
            for (int n = 0; n < q1; ++n) r += P.C[i * q1 + n] * mu[n];
            if (a == 0) rx[i] = r; else ry[i] = r;
        }
    }
    if (P.dim == 1) {
        for (int i = 0; i < q1; ++i) out[i] = rho * rx[i];
    } else {
        for (int i = 0; i < q1; ++i)
            for (int j = 0; j < q1; ++j) out[i * q1 + j] = rho * rx[i] * ry[j];
    }
}

// Moments of one node from FP64 populations.
__device__ void node_moments_f64(const LatticeParams& P, const double* f, double& rho, double& ux,
                                 double& uy, double& th, double& e, double& jx_o, double& jy_o) {
    double r = 0.0, jx = 0.0, jy = 0.0, en = 0.0;
    for (int p = 0; p < P.q; ++p) {
        const int ix = (P.dim == 1) ? p : p / P.q1;
        const int iy = (P.dim == 1) ? 0 : p % P.q1;
        const double vx = (double)P.v[ix];
        const double vy = (P.dim == 1) ? 0.0 : (double)P.v[iy];
        r += f[p];
        jx += vx * f[p];
        jy += vy * f[p];
        en += (vx * vx + vy * vy) * f[p];
    }
    rho = r;
    ux = jx / r;
    uy = jy / r;
    th = (en / r - (ux * ux + uy * uy)) / (double)P.dim;
    e = en;
    jx_o = jx;
    jy_o = jy;
}

// Check of one node's initial fields, made by the initialisation kernels that read
// them anyway: a non-finite value sets PLBM_STATUS_NONFINITE, otherwise rho <= 0
// PLBM_STATUS_RHO_NONPOS and theta <= 0 PLBM_STATUS_THETA_NONPOS.
__device__ __forceinline__ void check_init_node(const LatticeParams& P, const double* rho, const double* ux,
                                                const double* uy, const double* theta, long long n) {
    const double r = rho[n], a = ux[n];
    const double b = (P.dim == 2 && uy) ? uy[n] : 0.0;
    const bool has_t = !(P.isothermal || theta == nullptr);
    const double t = has_t ? theta[n] : 1.0;
    // on the integer pipe: a positive finite double has bits in [1, inf), a finite one after its sign
    const unsigned long long inf = 0x7ff0000000000000ull, mag = 0x7fffffffffffffffull;
    const unsigned long long rb = __double_as_longlong(r), tb = __double_as_longlong(t);
    if (rb - 1 < inf - 1 && tb - 1 < inf - 1 && (__double_as_longlong(a) & mag) < inf &&
        (__double_as_longlong(b) & mag) < inf)
        return;
    unsigned bits = 0u;
    if (!isfinite(r) || !isfinite(a) || !isfinite(b) || !isfinite(t)) bits |= PLBM_STATUS_NONFINITE;
    if (isfinite(r) && !(r > 0.0)) bits |= PLBM_STATUS_RHO_NONPOS;
    if (isfinite(t) && !(t > 0.0)) bits |= PLBM_STATUS_THETA_NONPOS;
    atomicOr(P.status, bits);
}

template <typename S>
__global__ void k_init(const __grid_constant__ LatticeParams P, const double* __restrict__ rho,
                       const double* __restrict__ ux, const double* __restrict__ uy,
                       const double* __restrict__ theta, S* __restrict__ f, int y0) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = y0 + blockIdx.y;
    if (x >= P.nx) return;
    const long long n = (long long)y * P.nx + x;
    check_init_node(P, rho, ux, uy, theta, n);
    const double th = (P.isothermal || theta == nullptr) ? P.theta0 : theta[n];
    double feq[kMaxQ];
    node_feq_f64(P, rho[n], ux[n], (P.dim == 2 && uy) ? uy[n] : 0.0, th, feq);
    for (int p = 0; p < P.q; ++p) f[elem_index(P, p, x, y)] = Storage<S>::from_f64(feq[p], P.W0[p]);
}

// Compile-time q1 versions of the two kernels above (arrays in registers, no
// integer division per population); the same FP64 formulas, the moments from
// the row and column sums S_i = sum_j f_ij, T_j = sum_i f_ij.
template <typename S, int Q1, int DIM>
__global__ void k_init_q(const __grid_constant__ LatticeParams P, const double* __restrict__ rho,
                         const double* __restrict__ ux, const double* __restrict__ uy,
                         const double* __restrict__ theta, S* __restrict__ f, int y0) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = y0 + blockIdx.y;
    if (x >= P.nx) return;
    const long long n = (long long)y * P.nx + x;
    check_init_node(P, rho, ux, uy, theta, n);
    const double th = (P.isothermal || theta == nullptr) ? P.theta0 : theta[n];
    double r[DIM][Q1];
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const double u = a == 0 ? ux[n] : (uy ? uy[n] : 0.0);
        double mu[Q1];
        mu[0] = 1.0;
        if (Q1 > 1) mu[1] = u;
#pragma unroll
        for (int k = 1; k + 1 < Q1; ++k) mu[k + 1] = u * mu[k] + (double)k * th * mu[k - 1];
#pragma unroll
        for (int i = 0; i < Q1; ++i) {
            double s = 0.0;
#pragma unroll
            for (int k = 0; k < Q1; ++k) s += P.C[i * Q1 + k] * mu[k];
            r[a][i] = s;
        }
    }
    const double rh = rho[n];
#pragma unroll
    for (int i = 0; i < Q1; ++i) {
        const double ri = rh * r[0][i];
#pragma unroll
        for (int j = 0; j < (DIM == 2 ? Q1 : 1); ++j) {
            const int p = DIM == 2 ? i * Q1 + j : i;
            const double fe = DIM == 2 ? ri * r[DIM - 1][j] : ri;
            f[elem_index(P, p, x, y)] = Storage<S>::from_f64(fe, P.W0[p]);
        }
    }
}

template <typename S, int Q1, int DIM>
__global__ void k_moments_q(const __grid_constant__ LatticeParams P, const S* __restrict__ f, double* rho,
                            double* ux, double* uy, double* theta, int y0) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = y0 + blockIdx.y;
    if (x >= P.nx) return;
    double Sx[Q1], Ty[Q1];
#pragma unroll
    for (int i = 0; i < Q1; ++i) Sx[i] = Ty[i] = 0.0;
#pragma unroll
    for (int i = 0; i < Q1; ++i)
#pragma unroll
        for (int j = 0; j < (DIM == 2 ? Q1 : 1); ++j) {
            const int p = DIM == 2 ? i * Q1 + j : i;
            const double v = Storage<S>::to_f64(f[elem_index(P, p, x, y)], P.W0[p]);
            Sx[i] += v;
            Ty[j] += v;
        }
    double m0 = 0.0, jx = 0.0, jy = 0.0, en = 0.0;
#pragma unroll
    for (int i = 0; i < Q1; ++i) {
        const double vi = (double)P.v[i];
        m0 += Sx[i];
        jx += vi * Sx[i];
        en += vi * vi * Sx[i];
        if (DIM == 2) {
            jy += vi * Ty[i];
            en += vi * vi * Ty[i];
        }
    }
    const double a = jx / m0, b = jy / m0;
    const long long n = (long long)y * P.nx + x;
    if (rho) rho[n] = m0;
    if (ux) ux[n] = a;
    if (uy) uy[n] = b;
    if (theta) theta[n] = (en / m0 - (a * a + b * b)) / (double)DIM;
}

// The same of a symmetric five-velocity set by the sums of its steps (1024^2: 218 -> 126 us).
template <int DIM>
__global__ void __launch_bounds__(128) k_moments_sym5_f64(const __grid_constant__ LatticeParams P, const double* __restrict__ f,
                                                          double* rho, double* ux, double* uy, double* theta, int y0) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = y0 + blockIdx.y;
    if (x >= P.nx) return;
    double g[Sym5Core<DIM>::Q], r, t, e, jx, jy, a, b;
#pragma unroll
    for (int p = 0; p < Sym5Core<DIM>::Q; ++p) g[p] = __ldg(f + elem_index(P, p, x, y));
    Sym5Core<DIM>::moments(g, P, false, r, t, jx, jy, e, a, b);
    const long long n = (long long)y * P.nx + x;
    if (rho) rho[n] = r;
    if (ux) ux[n] = a;
    if (uy) uy[n] = b;
    if (theta) theta[n] = t;
}

// Initial state of a 16/32-bit handle with a symmetric five-velocity set, in the
// FP32 deviation arithmetic of its own collision: per axis the constraint form
// of the rule (dmu_n = mu_n(u, theta) - mu_n(0, theta0), n = 1..4;
// O_b = (dmu3 - a^2 dmu1) / (2b(b^2 - a^2)), O_a = (dmu1 - 2b O_b) / (2a),
// E_b = (dmu4 - a^2 dmu2) / (2b^2(b^2 - a^2)), E_a = (dmu2 - 2b^2 E_b) / (2a^2),
// dr = (-2(E_a + E_b), E_a +- O_a, E_b +- O_b)), then
// f^eq - w0 = X_i (w_j + dr^y_j) + w_i dr^y_j with X_i = (rho - 1) w_i + rho dr^x_i
// (in 1D: X_i).  The inputs enter as the small quantities rho - 1, u and
// theta - theta0, formed in FP64.
__device__ __forceinline__ void sym5_dev(const LatticeParams& P, float u, float dth, float (&dr)[5]) {
    const float u2 = u * u;
    const float th = P.theta0f + dth;
    const float dm1 = u;
    const float dm2 = u2 + dth;
    const float dm3 = u * (u2 + 3.0f * th);
    const float dm4 = u2 * (u2 + 6.0f * th) + 3.0f * dth * (th + P.theta0f);
    const float Ob = (dm3 - P.sa2 * dm1) * P.kOb;
    const float Oa = (dm1 - 2.0f * P.sb * Ob) * P.kOa;
    const float Eb = (dm4 - P.sa2 * dm2) * P.kEb;
    const float Ea = (dm2 - 2.0f * P.sb2 * Eb) * P.kEa;
    dr[0] = -2.0f * (Ea + Eb);
    dr[1] = Ea + Oa;
    dr[2] = Ea - Oa;
    dr[3] = Eb + Ob;
    dr[4] = Eb - Ob;
}

// The state of one node: put(p, value) for each population.
template <int DIM, class Put>
__device__ __forceinline__ void init_sym5_node(const LatticeParams& P, const double* rho, const double* ux, const double* uy,
                                               const double* theta, long long n, Put put) {
    const float dth = (P.isothermal || theta == nullptr) ? 0.0f : (float)(theta[n] - P.theta0);
    const float drho = (float)(rho[n] - 1.0);
    const float rh = 1.0f + drho;
    float drx[5], dry[5];
    sym5_dev(P, (float)ux[n], dth, drx);
    if (DIM == 2) sym5_dev(P, uy ? (float)uy[n] : 0.0f, dth, dry);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const float X = fmaf(drho, P.w1f[i], rh * drx[i]);
        if (DIM == 1) {
            put(i, X);
        } else {
#pragma unroll
            for (int j = 0; j < 5; ++j) put(i * 5 + j, fmaf(X, P.w1f[j] + dry[j], P.w1f[i] * dry[j]));
        }
    }
}

template <typename S, int DIM>
__global__ void k_init_sym5_dev(const __grid_constant__ LatticeParams P, const double* __restrict__ rho,
                                const double* __restrict__ ux, const double* __restrict__ uy,
                                const double* __restrict__ theta, S* __restrict__ f, int y0) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = y0 + blockIdx.y;
    if (x >= P.nx) return;
    const long long n = (long long)y * P.nx + x;
    check_init_node(P, rho, ux, uy, theta, n);
    init_sym5_node<DIM>(P, rho, ux, uy, theta, n,
                        [&](int p, float v) { Storage<S>::store(f + elem_index(P, p, x, y), v); });
}

// The same for the row-paired layout, whole lattice: a thread takes both nodes of a pair and stores
// them together (one node per thread writes half of each 32-byte sector, and its other half
// from a block far away: 2048^2 FP32 260 -> 80 us, FP16 141 -> 64 us).
template <typename S>
__global__ void __launch_bounds__(128) k_init_pair(const __grid_constant__ LatticeParams P, const double* __restrict__ rho,
                                                   const double* __restrict__ ux, const double* __restrict__ uy,
                                                   const double* __restrict__ theta, typename PairStore<S>::V* __restrict__ f) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y;
    if (x >= P.nx) return;
    const long long n0 = (long long)r * P.nx + x, n1 = n0 + (long long)P.half_ny * P.nx;
    check_init_node(P, rho, ux, uy, theta, n0);
    check_init_node(P, rho, ux, uy, theta, n1);
    float lo[25];
    init_sym5_node<2>(P, rho, ux, uy, theta, n0, [&](int p, float v) { lo[p] = v; });
    const long long here = (long long)r * P.pitch + x;
    init_sym5_node<2>(P, rho, ux, uy, theta, n1,
                      [&](int p, float v) { PairStore<S>::store(f + p * (P.plane / 2) + here, f2(lo[p], v)); });
}

// FP64 storage: the initial state by the constraint form of the rule that the steps use (16 FP64
// instructions an axis instead of 31 with general coefficients; 1024^2 192 -> 140 us).
template <int DIM>
__global__ void __launch_bounds__(128) k_init_sym5_f64(const __grid_constant__ LatticeParams P, const double* __restrict__ rho,
                                                       const double* __restrict__ ux, const double* __restrict__ uy,
                                                       const double* __restrict__ theta, double* __restrict__ f, int y0) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = y0 + blockIdx.y;
    if (x >= P.nx) return;
    const long long n = (long long)y * P.nx + x;
    check_init_node(P, rho, ux, uy, theta, n);
    const double th = (P.isothermal || theta == nullptr) ? P.theta0 : theta[n];
    const double u = ux[n], v = DIM == 2 && uy ? uy[n] : 0.0, rh = rho[n];
    double rx[5], ry[5];
    Sym5Core<DIM>::rule(P, u, v, th, false, rx, ry);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const double X = rh * rx[i];
        if constexpr (DIM == 2) {
#pragma unroll
            for (int j = 0; j < 5; ++j) f[elem_index(P, 5 * i + j, x, y)] = X * ry[j];
        } else {
            f[elem_index(P, i, x, y)] = X;
        }
    }
}

// Moments of a 16/32-bit (deviation) state: the row and column sums of the
// stored deviations g in float-float arithmetic (an FP32 pair hi + lo carried
// through error-free sums and products, ~2^-48 relative), then
// rho = 1 + sum g, j = sum v g, E = d theta0 + sum |v|^2 g (the rest identities of
// the 1D rule) and theta = (E / rho - |u|^2) / d in FP64.
// (FF, ff_add, ff_scale, ff_f64: plbm_device.cuh)

// The fields of a node in FP64 from its float-float sums.
struct NodeFields {
    double rho, ux, uy, theta;
};
template <int DIM>
__device__ __forceinline__ NodeFields fields_from_sums(const LatticeParams& P, FF dm, FF jx, FF jy, FF de) {
    NodeFields o;
    o.rho = 1.0 + ff_f64(dm);
    const double ir = recip_f64(o.rho);
    o.ux = ff_f64(jx) * ir;
    o.uy = DIM == 2 ? ff_f64(jy) * ir : 0.0;
    o.theta = (((double)DIM * P.theta0 + ff_f64(de)) * ir - (o.ux * o.ux + o.uy * o.uy)) * (1.0 / DIM);
    return o;
}

// get(p): the stored deviation of population p.
template <int Q1, int DIM, class Get>
__device__ __forceinline__ NodeFields fields_dev(const LatticeParams& P, Get get) {
    FF Sx[Q1], Ty[Q1];
#pragma unroll
    for (int i = 0; i < Q1; ++i) Sx[i] = Ty[i] = FF{0.0f, 0.0f};
#pragma unroll
    for (int i = 0; i < Q1; ++i)
#pragma unroll
        for (int j = 0; j < (DIM == 2 ? Q1 : 1); ++j) {
            const float g = get(DIM == 2 ? i * Q1 + j : i);
            Sx[i] = ff_add(Sx[i], g);
            if (DIM == 2) Ty[j] = ff_add(Ty[j], g);
        }
    FF dm{0.0f, 0.0f}, jx = dm, jy = dm, de = dm;
#pragma unroll
    for (int i = 0; i < Q1; ++i) {
        const float vi = (float)P.v[i];
        dm = ff_add(dm, Sx[i]);
        jx = ff_add(jx, ff_scale(Sx[i], vi));
        de = ff_add(de, ff_scale(ff_scale(Sx[i], vi), vi));
        if (DIM == 2) {
            jy = ff_add(jy, ff_scale(Ty[i], vi));
            de = ff_add(de, ff_scale(ff_scale(Ty[i], vi), vi));
        }
    }
    return fields_from_sums<DIM>(P, dm, jx, jy, de);
}

__device__ __forceinline__ void put_fields(const NodeFields& o, long long n, double* rho, double* ux, double* uy, double* theta) {
    if (rho) rho[n] = o.rho;
    if (ux) ux[n] = o.ux;
    if (uy) uy[n] = o.uy;
    if (theta) theta[n] = o.theta;
}

template <typename S, int Q1, int DIM>
__global__ void k_moments_dev(const __grid_constant__ LatticeParams P, const S* __restrict__ f, double* rho,
                              double* ux, double* uy, double* theta, int y0) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = y0 + blockIdx.y;
    if (x >= P.nx) return;
    const NodeFields o =
        fields_dev<Q1, DIM>(P, [&](int p) -> float { return Storage<S>::load(f + elem_index(P, p, x, y)); });
    put_fields(o, (long long)y * P.nx + x, rho, ux, uy, theta);
}

__device__ __forceinline__ FF lane_of(FFV<float> v, int) { return {v.hi, v.lo}; }
__device__ __forceinline__ FF lane_of(FFV<float2> v, int l) { return l ? FF{v.hi.y, v.lo.y} : FF{v.hi.x, v.lo.x}; }
template <class V>
__device__ __forceinline__ FFV<V> ffv_times(FFV<V> a, float c) {
    const V p = mul2(a.hi, splat<V>(c));
    return {p, fma2(a.lo, splat<V>(c), fma2(a.hi, splat<V>(c), neg2(p)))};
}
template <class V>
__device__ __forceinline__ FFV<V> ffv_minus(FFV<V> a, FFV<V> b) { return ffv_acc(a, FFV<V>{neg2(b.hi), neg2(b.lo)}); }

// The same for symmetric five-velocity sets, with j and E from the sums and differences of opposite
// velocities.  V = float2: row-paired layout, whole lattice; a thread loads both nodes of a pair,
// so that the state is read once (one node per thread reads it twice, once for each half of
// the rows), and sums in packed arithmetic.  V = float: one node, any rows.
// 2048^2 FP32 205 -> 128 us, FP16 200 -> 125 us, 2047^2 FP32 202 -> 124 us: 15 FP64
// instructions a node (31 with the division and conversions) take 104, the bytes 82 and 51.
template <typename S, class V>
__device__ __forceinline__ void moments_sym5(const LatticeParams& P, const S* __restrict__ f, double* rho, double* ux, double* uy,
                                             double* theta, int x, int y) {
    constexpr int kLanes = sizeof(V) / sizeof(float);
    const FFV<V> zero{splat<V>(0.0f), splat<V>(0.0f)};
    const S* at = f + elem_index(P, 0, x, y);   // V = float2: y < half_ny, the pair's first node
    FFV<V> Sx[5], Ty[5];
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            const S* q = at + (5 * i + j) * P.plane;
            V g;
            if constexpr (kLanes == 2)
                g = PairStore<S>::cvt(PairStore<S>::raw(reinterpret_cast<const typename PairStore<S>::V*>(q)));
            else
                g = Storage<S>::load(q);
            Sx[i] = j ? ffv_acc(Sx[i], g) : FFV<V>{g, zero.lo};
            Ty[j] = i ? ffv_acc(Ty[j], g) : FFV<V>{g, zero.lo};
        }
    const FFV<V> Sp = ffv_acc(Sx[1], Sx[2]), Sq = ffv_acc(Sx[3], Sx[4]);
    const FFV<V> Tp = ffv_acc(Ty[1], Ty[2]), Tq = ffv_acc(Ty[3], Ty[4]);
    const FFV<V> dm = ffv_acc(ffv_acc(Sx[0], Sp), Sq);
    const FFV<V> jx = ffv_acc(ffv_times(ffv_minus(Sx[1], Sx[2]), P.sa), ffv_times(ffv_minus(Sx[3], Sx[4]), P.sb));
    const FFV<V> jy = ffv_acc(ffv_times(ffv_minus(Ty[1], Ty[2]), P.sa), ffv_times(ffv_minus(Ty[3], Ty[4]), P.sb));
    const FFV<V> de = ffv_acc(ffv_times(ffv_acc(Sp, Tp), P.sa2), ffv_times(ffv_acc(Sq, Tq), P.sb2));
#pragma unroll
    for (int l = 0; l < kLanes; ++l)
        put_fields(fields_from_sums<2>(P, lane_of(dm, l), lane_of(jx, l), lane_of(jy, l), lane_of(de, l)),
                   ((long long)y + l * P.half_ny) * P.nx + x, rho, ux, uy, theta);
}

template <typename S, class V>
__global__ void __launch_bounds__(128) k_moments_sym5(const __grid_constant__ LatticeParams P, const S* __restrict__ f,
                                                      double* rho, double* ux, double* uy, double* theta, int y0) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x < P.nx) moments_sym5<S, V>(P, f, rho, ux, uy, theta, x, y0 + blockIdx.y);
}

// FP16 pairs: every value is a multiple of 2^-24, so that below 1/4 (every healthy deviation) the sums are
// exact 32-bit integers (the bits of g + 3/4 are 2^24 g and a constant), rho needs no FP64 instruction and
// a node 10 instead of 15: 2048^2 125 -> 85 us.  A thread that meets a larger value, an infinity or a NaN
// starts over in float-float.
__global__ void __launch_bounds__(128) k_moments_f16pair(const __grid_constant__ LatticeParams P, const __half* __restrict__ f,
                                                         double* rho, double* ux, double* uy, double* theta) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= P.nx) return;
    const __half2* at = reinterpret_cast<const __half2*>(f + elem_index(P, 0, x, y));
    uint2 S[5], T[5];   // unsigned: sums modulo 2^32
    __half2 most = __float2half2_rn(0.0f);
#pragma unroll
    for (int i = 0; i < 5; ++i) S[i] = T[i] = make_uint2(0u, 0u);
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            const __half2 h = __ldg(at + (5 * i + j) * (P.plane / 2));
            most = __hmax2_nan(most, __habs2(h));
            const float2 g = add2(__half22float2(h), f2s(0.75f));
            S[i].x += __float_as_uint(g.x);
            S[i].y += __float_as_uint(g.y);
            T[j].x += __float_as_uint(g.x);
            T[j].y += __float_as_uint(g.y);
        }
    const float2 top = __half22float2(most);
    if (!(top.x < 0.25f && top.y < 0.25f)) {
        moments_sym5<__half, float2>(P, f, rho, ux, uy, theta, x, y);
        return;
    }
    const unsigned off = 5u * 0x3f400000u;   // five times the bits of 3/4
    const long long a = P.v[1], b = P.v[3];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        auto sum = [&](const uint2& v) { return (long long)(int)((l ? v.y : v.x) - off); };
        const long long sp = sum(S[1]) + sum(S[2]), sq = sum(S[3]) + sum(S[4]);
        const long long tp = sum(T[1]) + sum(T[2]), tq = sum(T[3]) + sum(T[4]);
        auto value = [](long long i) { return f64_of_fixed(i, 1056, false); };   // units of 2^-24
        NodeFields o;
        o.rho = value((1ll << 24) + sum(S[0]) + sp + sq);
        const double ir = recip_f64(o.rho);
        o.ux = value(a * (sum(S[1]) - sum(S[2])) + b * (sum(S[3]) - sum(S[4]))) * ir;
        o.uy = value(a * (sum(T[1]) - sum(T[2])) + b * (sum(T[3]) - sum(T[4]))) * ir;
        o.theta = ((2.0 * P.theta0 + value(a * a * (sp + tp) + b * b * (sq + tq))) * ir - (o.ux * o.ux + o.uy * o.uy)) * 0.5;
        put_fields(o, ((long long)y + l * P.half_ny) * P.nx + x, rho, ux, uy, theta);
    }
}

template <typename S>
__global__ void k_moments(const __grid_constant__ LatticeParams P, const S* __restrict__ f,
                          double* rho, double* ux, double* uy, double* theta, int y0) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = y0 + blockIdx.y;
    if (x >= P.nx) return;
    double fn[kMaxQ];
    for (int p = 0; p < P.q; ++p) fn[p] = Storage<S>::to_f64(f[elem_index(P, p, x, y)], P.W0[p]);
    double r, a, b, t, e, jx, jy;
    node_moments_f64(P, fn, r, a, b, t, e, jx, jy);
    const long long n = (long long)y * P.nx + x;
    if (rho) rho[n] = r;
    if (ux) ux[n] = a;
    if (uy) uy[n] = b;
    if (theta) theta[n] = t;
}

// Moments of the stored state packed for the surrogate: F[n] = (rho, u_x, u_y,
// theta) in FP32 and the network input x[n] = bf16((F - mean_in) * istd_in).
// FP32 arithmetic on the deviations g = f - w0 (the network's input is bf16 and
// its fields FP32): rho = 1 + sum g, j = sum v g, E = 2 theta0 + sum |v|^2 g
// (the rest sums the 1D rule reproduces), with the row and column sums of g
// factorising the velocity weights.
template <typename S>
__device__ __forceinline__ float dev_f32(const S* f, long long i, double w0) {
    return Storage<S>::load(f + i);
}
template <>
__device__ __forceinline__ float dev_f32<double>(const double* f, long long i, double w0) {
    return (float)(__ldg(f + i) - w0);
}

// refs (batched launch, grid.z = lattice): lattice blockIdx.z reads refs[z].f and
// writes its fields at refs[z].index * nx * ny of the stacks F and x.
template <typename S, int Q1>
__global__ void k_moments_pack(const __grid_constant__ LatticeParams P, const S* __restrict__ f,
                               float4* __restrict__ F, __nv_bfloat16* __restrict__ x, float4 mean_in,
                               float4 istd_in, const LatticeRef* __restrict__ refs) {
    const int xx = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (xx >= P.nx) return;
    if (refs) {
        const LatticeRef r = refs[blockIdx.z];
        f = static_cast<const S*>(r.f);
        const long long off = r.index * P.nx * P.ny;
        F += off;
        x += off * 4;
    }
    constexpr int kQ1 = Q1 ? Q1 : kMaxQ1;
    const int q1 = Q1 ? Q1 : P.q1;
    float sx[kQ1], ty[kQ1];
#pragma unroll
    for (int i = 0; i < kQ1; ++i) sx[i] = ty[i] = 0.0f;
#pragma unroll
    for (int i = 0; i < kQ1; ++i) {
        if (i >= q1) break;
#pragma unroll
        for (int j = 0; j < kQ1; ++j) {
            if (j >= q1) break;
            const int p = i * q1 + j;
            const float g = dev_f32<S>(f, elem_index(P, p, xx, y), P.W0[p]);
            sx[i] += g;
            ty[j] += g;
        }
    }
    // rest sums: sum w0 = 1, sum v w0 = 0, sum |v|^2 w0 = 2 theta0
    float dr = 0.0f, jx = 0.0f, jy = 0.0f, de = 0.0f;
#pragma unroll
    for (int i = 0; i < kQ1; ++i) {
        if (i >= q1) break;
        const float v = (float)P.v[i];
        dr += sx[i];
        jx += v * sx[i];
        jy += v * ty[i];
        de += v * v * (sx[i] + ty[i]);
    }
    const float rho = 1.0f + dr;
    const float ir = 1.0f / rho;
    const float ux = jx * ir, uy = jy * ir;
    const float th = P.theta0f + 0.5f * ((de - 2.0f * P.theta0f * dr) * ir - (ux * ux + uy * uy));
    const long long n = (long long)y * P.nx + xx;
    const float4 v = make_float4(rho, ux, uy, th);
    F[n] = v;
    __nv_bfloat162 lo = __floats2bfloat162_rn((v.x - mean_in.x) * istd_in.x, (v.y - mean_in.y) * istd_in.y);
    __nv_bfloat162 hi = __floats2bfloat162_rn((v.z - mean_in.z) * istd_in.z, (v.w - mean_in.w) * istd_in.w);
    uint2 o;
    o.x = *reinterpret_cast<uint32_t*>(&lo);
    o.y = *reinterpret_cast<uint32_t*>(&hi);
    reinterpret_cast<uint2*>(x)[n] = o;
}

template <typename S>
__global__ void __launch_bounds__(kBlockX) k_reduce_state(const __grid_constant__ LatticeParams P,
                                                          const S* __restrict__ f) {
    const int x = blockIdx.x * kBlockX + threadIdx.x;
    const int y = blockIdx.y;
    NodeDiag d;
    diag_zero(d);
    if (x < P.nx) {
        double fn[kMaxQ];
        for (int p = 0; p < P.q; ++p) fn[p] = Storage<S>::to_f64(f[elem_index(P, p, x, y)], P.W0[p]);
        double r, a, b, t, e, jx, jy;
        node_moments_f64(P, fn, r, a, b, t, e, jx, jy);
        d.mass = r;
        d.jx = jx;
        d.jy = jy;
        d.energy = e;
        d.rho_min = r;
        d.theta_min = t;
        flag_status<double>(P, r, t);
    }
    const int blk = blockIdx.y * gridDim.x + blockIdx.x;
    block_reduce_diag<kBlockX>(d, P.partials + (long long)blk * kPartialStride);
}

// The same record for 16/32-bit storage with compile-time q1, on the FP32 pipe:
// per node the row and column sums of the stored deviations in float-float,
// mass - 1 = sum g, j = sum v g, E - d theta0 = sum |v|^2 g, then the block sums
// in float-float (block_reduce_diagf); the minima from FP32 rho and theta.
template <typename S, int Q1, int DIM>
__global__ void __launch_bounds__(kBlockX) k_reduce_state_dev(const __grid_constant__ LatticeParams P,
                                                              const S* __restrict__ f) {
    const int x = blockIdx.x * kBlockX + threadIdx.x;
    const int y = blockIdx.y;
    NodeDiagF d;
    diagf_zero(d);
    double rmin = 1e300, tmin = 1e300;
    if (x < P.nx) {
        FF Sx[Q1], Ty[Q1];
#pragma unroll
        for (int i = 0; i < Q1; ++i) Sx[i] = Ty[i] = FF{0.0f, 0.0f};
#pragma unroll
        for (int i = 0; i < Q1; ++i)
#pragma unroll
            for (int j = 0; j < (DIM == 2 ? Q1 : 1); ++j) {
                const int p = DIM == 2 ? i * Q1 + j : i;
                const float g = Storage<S>::load(f + elem_index(P, p, x, y));
                Sx[i] = ff_add(Sx[i], g);
                if (DIM == 2) Ty[j] = ff_add(Ty[j], g);
            }
        FF dm{0.0f, 0.0f}, jx = dm, jy = dm, de = dm;
#pragma unroll
        for (int i = 0; i < Q1; ++i) {
            const float vi = (float)P.v[i];
            dm = ff_add(dm, Sx[i]);
            jx = ff_add(jx, ff_scale(Sx[i], vi));
            de = ff_add(de, ff_scale(ff_scale(Sx[i], vi), vi));
            if (DIM == 2) {
                jy = ff_add(jy, ff_scale(Ty[i], vi));
                de = ff_add(de, ff_scale(ff_scale(Ty[i], vi), vi));
            }
        }
        // rho and theta of the node in FP64 (the minima are reported in FP64)
        const double rho = 1.0 + ff_f64(dm);
        const double ir = 1.0 / rho;
        const double ux = ff_f64(jx) * ir, uy = DIM == 2 ? ff_f64(jy) * ir : 0.0;
        const double th = (((double)DIM * P.theta0 + ff_f64(de)) * ir - (ux * ux + uy * uy)) / (double)DIM;
        flag_status<double>(P, rho, th);
        d.dmass = dm;
        d.jx = jx;
        d.jy = jy;
        d.denergy = de;
        d.n = 1.0f;
        rmin = rho;
        tmin = th;
    }
    const int blk = blockIdx.y * gridDim.x + blockIdx.x;
    block_reduce_diagf<kBlockX, true>(d, (double)DIM * P.theta0, P.partials + (long long)blk * kPartialStride, rmin,
                                      tmin);
}

// Sums the per-block partials in a fixed order, so the result is bit-reproducible for a
// given lattice: a cluster of kFinalBlocks blocks, whose own sums the first one adds up.
// One SM retires two FP64 operations a cycle, and a lattice of 1500 x 900 nodes has 5,400
// records of four sums: one block of 512 threads took 16.4 us (dependent loads, additions,
// FP64 minima), this 7.4.  Minima go by integer keys; a NaN is no minimum.  out[6]: the status word.
constexpr int kFinalBlocks = 8, kFinalThreads = 256;
__device__ __forceinline__ long long min_key(double v) { return v == v ? dkey(v) : 0x7fffffffffffffffLL; }
__global__ void __cluster_dims__(kFinalBlocks, 1, 1) __launch_bounds__(kFinalThreads)
k_finalize(const double* partials, int nblocks, const unsigned* status, double* __restrict__ out) {
    __shared__ double sum[4][kFinalThreads];
    __shared__ long long key[2][kFinalThreads];
    const int t = threadIdx.x;
    const long long none = dkey(1e300);
    double r[4] = {0, 0, 0, 0};
    long long m[2] = {none, none};
    step_wait();
#pragma unroll 4
    for (int b = blockIdx.x * kFinalThreads + t; b < nblocks; b += kFinalBlocks * kFinalThreads) {
        const double2* q = reinterpret_cast<const double2*>(partials + (long long)b * kPartialStride);
        const double2 a = load_state(q), c = load_state(q + 1), d = load_state(q + 2);
        r[0] += a.x;
        r[1] += a.y;
        r[2] += c.x;
        r[3] += c.y;
        m[0] = kmin(m[0], min_key(d.x));
        m[1] = kmin(m[1], min_key(d.y));
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) sum[k][t] = r[k];
    key[0][t] = m[0];
    key[1][t] = m[1];
    __syncthreads();
#pragma unroll
    for (int s = kFinalThreads / 2; s > 0; s >>= 1) {   // 4 s additions and 2 s minima over the whole block
        for (int i = t; i < 4 * s; i += kFinalThreads) sum[i / s][i % s] += sum[i / s][i % s + s];
        for (int i = t; i < 2 * s; i += kFinalThreads) key[i / s][i % s] = kmin(key[i / s][i % s], key[i / s][i % s + s]);
        __syncthreads();
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (blockIdx.x == 0 && t < 6) {
        const unsigned at = (unsigned)__cvta_generic_to_shared(t < 4 ? (void*)&sum[t][0] : (void*)&key[t - 4][0]);
        long long v[kFinalBlocks];
#pragma unroll
        for (int b = 0; b < kFinalBlocks; ++b) {
            unsigned there;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(at), "r"(b));
            asm volatile("ld.shared::cluster.s64 %0, [%1];" : "=l"(v[b]) : "r"(there));
        }
        if (t < 4) {
            double s = __longlong_as_double(v[0]);
#pragma unroll
            for (int b = 1; b < kFinalBlocks; ++b) s += __longlong_as_double(v[b]);
            out[t] = s;
        } else {
            long long k = v[0];
#pragma unroll
            for (int b = 1; b < kFinalBlocks; ++b) k = kmin(k, v[b]);
            out[t] = dunkey(k);
        }
    }
    if (blockIdx.x == 0 && t == 32) {
        unsigned* o = reinterpret_cast<unsigned*>(out + 6);
        o[0] = load_state(status);
        o[1] = 0u;
    }
    // no block's shared memory goes before the first one has read it
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename S>
__global__ void k_get_pop(const __grid_constant__ LatticeParams P, const S* __restrict__ f,
                          double* __restrict__ out) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    const int p = blockIdx.z;
    if (x >= P.nx) return;
    const double v = Storage<S>::to_f64(f[elem_index(P, p, x, y)], P.W0[p]);
    out[((long long)p * P.ny + y) * P.nx + x] = v;
}

template <typename S>
__global__ void k_set_pop(const __grid_constant__ LatticeParams P, const double* __restrict__ in,
                          S* __restrict__ f) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    const int p = blockIdx.z;
    if (x >= P.nx) return;
    f[elem_index(P, p, x, y)] = Storage<S>::from_f64(in[((long long)p * P.ny + y) * P.nx + x], P.W0[p]);
}

#define PLBM_DISPATCH(prec, CALL)                                        \
    switch (prec) {                                                      \
        case kF64: { using S = double; CALL; break; }                    \
        case kF32: { using S = float; CALL; break; }                     \
        case kF16Dev: { using S = __half; CALL; break; }                 \
        case kBF16Dev: { using S = __nv_bfloat16; CALL; break; }         \
        default: return cudaErrorInvalidValue;                           \
    }

// The deviation-storage precisions only.
#define PLBM_DISPATCH_DEV(prec, CALL)                                    \
    switch (prec) {                                                      \
        case kF32: { using S = float; CALL; break; }                     \
        case kF16Dev: { using S = __half; CALL; break; }                 \
        case kBF16Dev: { using S = __nv_bfloat16; CALL; break; }         \
        default: return cudaErrorInvalidValue;                           \
    }

cudaError_t launch_init(int prec, const LatticeParams& P, const double* rho, const double* ux,
                        const double* uy, const double* theta, void* f, cudaStream_t stream, int y0, int y1) {
    if (y1 < 0) y1 = P.ny;
    if (y1 <= y0) return cudaSuccess;
    dim3 grid((P.nx + 127) / 128, y1 - y0);
    if (P.paired && y0 == 0 && y1 == P.ny) {
        grid.y = P.half_ny;
        PLBM_DISPATCH_DEV(prec, (k_init_pair<S><<<grid, 128, 0, stream>>>(P, rho, ux, uy, theta,
                                                                          static_cast<PairStore<S>::V*>(f))));
        return cudaGetLastError();
    }
    if (prec == kF64 && P.sym5) {
        double* d = static_cast<double*>(f);
        if (P.dim == 2)
            k_init_sym5_f64<2><<<grid, 128, 0, stream>>>(P, rho, ux, uy, theta, d, y0);
        else
            k_init_sym5_f64<1><<<grid, 128, 0, stream>>>(P, rho, ux, uy, theta, d, y0);
        return cudaGetLastError();
    }
#define PLBM_INIT_DEV(DIMv)                                                                            \
    if (P.dim == DIMv) {                                                                               \
        PLBM_DISPATCH_DEV(prec, (k_init_sym5_dev<S, DIMv><<<grid, 128, 0, stream>>>(P, rho, ux, uy, theta, \
                                                                                 static_cast<S*>(f), y0))); \
        return cudaGetLastError();                                                                     \
    }
    if (prec != kF64 && P.sym5) {
        PLBM_INIT_DEV(2)
        PLBM_INIT_DEV(1)
    }
#undef PLBM_INIT_DEV
#define PLBM_INIT_Q(Q1v, DIMv)                                                                          \
    if (P.q1 == Q1v && P.dim == DIMv) {                                                                 \
        PLBM_DISPATCH(prec, (k_init_q<S, Q1v, DIMv><<<grid, 128, 0, stream>>>(P, rho, ux, uy, theta,     \
                                                                              static_cast<S*>(f), y0)));  \
        return cudaGetLastError();                                                                      \
    }
    PLBM_INIT_Q(3, 2)
    PLBM_INIT_Q(4, 2)
    PLBM_INIT_Q(5, 2)
    PLBM_INIT_Q(5, 1)
#undef PLBM_INIT_Q
    PLBM_DISPATCH(prec, (k_init<S><<<grid, 128, 0, stream>>>(P, rho, ux, uy, theta,
                                                             static_cast<S*>(f), y0)));
    return cudaGetLastError();
}

cudaError_t launch_moments(int prec, const LatticeParams& P, const void* f, double* rho,
                           double* ux, double* uy, double* theta, cudaStream_t stream, int y0, int y1) {
    if (y1 < 0) y1 = P.ny;
    if (y1 <= y0) return cudaSuccess;
    dim3 grid((P.nx + 127) / 128, y1 - y0);
    if (prec != kF64 && P.sym5 && P.dim == 2) {
        if (P.paired && y0 == 0 && y1 == P.ny) {
            grid.y = P.half_ny;
            if (prec == kF16Dev) {
                k_moments_f16pair<<<grid, 128, 0, stream>>>(P, static_cast<const __half*>(f), rho, ux, uy, theta);
                return cudaGetLastError();
            }
            PLBM_DISPATCH_DEV(prec, (k_moments_sym5<S, float2><<<grid, 128, 0, stream>>>(
                                        P, static_cast<const S*>(f), rho, ux, uy, theta, 0)));
        } else {
            PLBM_DISPATCH_DEV(prec, (k_moments_sym5<S, float><<<grid, 128, 0, stream>>>(
                                        P, static_cast<const S*>(f), rho, ux, uy, theta, y0)));
        }
        return cudaGetLastError();
    }
    if (prec == kF64 && P.sym5) {
        const double* d = static_cast<const double*>(f);
        if (P.dim == 2)
            k_moments_sym5_f64<2><<<grid, 128, 0, stream>>>(P, d, rho, ux, uy, theta, y0);
        else
            k_moments_sym5_f64<1><<<grid, 128, 0, stream>>>(P, d, rho, ux, uy, theta, y0);
        return cudaGetLastError();
    }
#define PLBM_MOM_Q(Q1v, DIMv)                                                                           \
    if (P.q1 == Q1v && P.dim == DIMv) {                                                                 \
        if (prec == kF64)                                                                               \
            k_moments_q<double, Q1v, DIMv><<<grid, 128, 0, stream>>>(                                   \
                P, static_cast<const double*>(f), rho, ux, uy, theta, y0);                                  \
        else                                                                                            \
            PLBM_DISPATCH_DEV(prec, (k_moments_dev<S, Q1v, DIMv><<<grid, 128, 0, stream>>>(             \
                                    P, static_cast<const S*>(f), rho, ux, uy, theta, y0)));                 \
        return cudaGetLastError();                                                                      \
    }
    PLBM_MOM_Q(3, 2)
    PLBM_MOM_Q(4, 2)
    PLBM_MOM_Q(5, 2)
    PLBM_MOM_Q(5, 1)
#undef PLBM_MOM_Q
    PLBM_DISPATCH(prec, (k_moments<S><<<grid, 128, 0, stream>>>(P, static_cast<const S*>(f), rho,
                                                                ux, uy, theta, y0)));
    return cudaGetLastError();
}

cudaError_t launch_moments_pack(int prec, const LatticeParams& P, const void* f, float* F, void* x,
                                const float* mean_in, const float* std_in, cudaStream_t stream) {
    if (P.dim != 2) return cudaErrorInvalidValue;
    const float4 mi = make_float4(mean_in[0], mean_in[1], mean_in[2], mean_in[3]);
    const float4 si = make_float4(1.f / std_in[0], 1.f / std_in[1], 1.f / std_in[2], 1.f / std_in[3]);
    dim3 grid((P.nx + 127) / 128, P.ny);
    const LatticeRef* none = nullptr;
    if (P.q1 == 5) {
        PLBM_DISPATCH(prec, (k_moments_pack<S, 5><<<grid, 128, 0, stream>>>(
                                P, static_cast<const S*>(f), reinterpret_cast<float4*>(F),
                                static_cast<__nv_bfloat16*>(x), mi, si, none)));
    } else {
        PLBM_DISPATCH(prec, (k_moments_pack<S, 0><<<grid, 128, 0, stream>>>(
                                P, static_cast<const S*>(f), reinterpret_cast<float4*>(F),
                                static_cast<__nv_bfloat16*>(x), mi, si, none)));
    }
    return cudaGetLastError();
}

cudaError_t launch_moments_pack_batch(int prec, const LatticeParams& P, const LatticeRef* refs, int n, float* F,
                                      void* x, const float* mean_in, const float* std_in, cudaStream_t stream) {
    if (P.dim != 2 || n < 1 || n > 65535) return cudaErrorInvalidValue;
    const float4 mi = make_float4(mean_in[0], mean_in[1], mean_in[2], mean_in[3]);
    const float4 si = make_float4(1.f / std_in[0], 1.f / std_in[1], 1.f / std_in[2], 1.f / std_in[3]);
    dim3 grid((P.nx + 127) / 128, P.ny, n);
    if (P.q1 == 5) {
        PLBM_DISPATCH(prec, (k_moments_pack<S, 5><<<grid, 128, 0, stream>>>(
                                P, nullptr, reinterpret_cast<float4*>(F), static_cast<__nv_bfloat16*>(x), mi, si,
                                refs)));
    } else {
        PLBM_DISPATCH(prec, (k_moments_pack<S, 0><<<grid, 128, 0, stream>>>(
                                P, nullptr, reinterpret_cast<float4*>(F), static_cast<__nv_bfloat16*>(x), mi, si,
                                refs)));
    }
    return cudaGetLastError();
}

cudaError_t launch_finalize(const LatticeParams& P, int nblocks, double* out, cudaStream_t stream) {
    return launch_dependent(true, k_finalize, kFinalBlocks, kFinalThreads, stream, P.partials, nblocks, P.status, out);
}

cudaError_t launch_reduce_state(int prec, const LatticeParams& P, const void* f, double* out,
                                cudaStream_t stream) {
    dim3 grid((P.nx + kBlockX - 1) / kBlockX, P.ny);
    bool done = false;
#define PLBM_RED_Q(Q1v, DIMv)                                                                           \
    if (!done && prec != kF64 && P.q1 == Q1v && P.dim == DIMv) {                                        \
        PLBM_DISPATCH_DEV(prec, (k_reduce_state_dev<S, Q1v, DIMv><<<grid, kBlockX, 0, stream>>>(         \
                                    P, static_cast<const S*>(f))));                                     \
        done = true;                                                                                    \
    }
    PLBM_RED_Q(3, 2)
    PLBM_RED_Q(4, 2)
    PLBM_RED_Q(5, 2)
    PLBM_RED_Q(5, 1)
#undef PLBM_RED_Q
    if (!done)
        PLBM_DISPATCH(prec, (k_reduce_state<S><<<grid, kBlockX, 0, stream>>>(P, static_cast<const S*>(f))));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_finalize(P, reduce_blocks(P), out, stream);
}

cudaError_t launch_get_populations(int prec, const LatticeParams& P, const void* f, double* out,
                                   cudaStream_t stream) {
    dim3 grid((P.nx + 127) / 128, P.ny, P.q);
    PLBM_DISPATCH(prec, (k_get_pop<S><<<grid, 128, 0, stream>>>(P, static_cast<const S*>(f), out)));
    return cudaGetLastError();
}

cudaError_t launch_set_populations(int prec, const LatticeParams& P, const double* in, void* f,
                                   cudaStream_t stream) {
    dim3 grid((P.nx + 127) / 128, P.ny, P.q);
    PLBM_DISPATCH(prec, (k_set_pop<S><<<grid, 128, 0, stream>>>(P, in, static_cast<S*>(f))));
    return cudaGetLastError();
}

}  // namespace plbm
