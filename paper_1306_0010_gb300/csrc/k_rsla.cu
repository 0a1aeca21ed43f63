// k_rsla.cu -- grid reductions behind the reduced-speed-of-light helpers of librhd.so
// (Sections 3.1 and 3.2): the maximum gas signal speed v_max = max(|v| + c_eff) of
// Eq. algorithm:ceff, and the largest optical depth of the domain along the grid axes, which set
// Delta t_gas (Eq. algorithm:gastimestep) and the choice of chat (Eq. rsla:staticdiffreq).
//
// Every block reduces a fixed set of cells (or lines) to its maximum and a one-block kernel takes
// the maximum of the block results: the result does not depend on timing.  A NaN anywhere is
// carried to the result (the comparisons below keep it), so the host can report it.
#include <cuda_runtime.h>
#include <math.h>

#include "fp_convert.cuh"
#include "rhd_internal.h"

namespace rhd {

constexpr int RS_THREADS = 256;

// the larger of a, b, a NaN in either winning
__device__ __forceinline__ double max_nan(double a, double b) { return (b > a || b != b) ? b : a; }

// k_F of cell i: the per-cell array if given, else the opacity law kappa_F rho^p
__device__ __forceinline__ double flux_absorption(const GridParams& g, const double* kF, const double* rho,
                                                  long long i)
{
    if (kF) return kF[i];
    const double r = rho[i];
    return g.kpow == 0 ? g.kappa_F : (g.kpow == 1 ? g.kappa_F * r : (g.kappa_F * r) * r);
}

// block maximum of v into out[blockIdx.x]
__device__ __forceinline__ void block_max(double v, double* out)
{
    __shared__ double sh[RS_THREADS];
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int s = RS_THREADS / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] = max_nan(sh[threadIdx.x], sh[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = sh[0];
}

// v_max over the cells: |v| + sqrt((gamma P + (4/9) E (1 - exp(-k_F dx))) / rho) with P = rho T / (mu/k_B).
// The FP64 value (the result) costs an exponential, two square roots and two divisions on the FP64 pipe, about
// ten times what reading the cell takes; only the maximum matters, so few cells are evaluated in FP64: those
// whose FP32 value cannot be told from the maximum.  The FP32 value has a relative error below 2^-20 (truncated
// inputs and some ten roundings of 2^-24 under a square root); two values are told apart where they differ by
// 2^-18.  Each thread keeps the inputs of its largest cell so far: a cell that is clearly below it or below the
// block's maximum is passed over, one clearly above it takes its place, and one that cannot be told from it is
// evaluated at once, unless its inputs are the same.  At the end the kept cell is evaluated if it cannot be told
// from the block's maximum.  The cell with the FP64 maximum is never passed over, so the result is the FP64
// maximum itself, whatever the timing (300 x 250 x 200: 1041 us with each thread's own maximum and a bound of
// 2^-12, the call now 230 us with its host synchronisation).  NaN, infinities and values small enough to lose bits to
// FP32 underflow are evaluated at once.  NaN truncates to infinity, which as k_F would be just an opaque cell: k_F - k_F
// carries it on.
struct SignalCell {
    double r, T, E, v[3], k;
};
__device__ __forceinline__ double signal_speed(const GridParams& g, const SignalCell& s, double dx_min)
{
    const double P = s.r * s.T / g.mu_over_kB;
    const double rad = (4.0 / 9.0) * s.E * (-expm1(-s.k * dx_min));
    return sqrt(s.v[0] * s.v[0] + s.v[1] * s.v[1] + s.v[2] * s.v[2]) + sqrt((g.gamma * P + rad) / s.r);
}
__device__ __forceinline__ unsigned long long differs(double a, double b)
{
    return (unsigned long long)(__double_as_longlong(a) ^ __double_as_longlong(b));
}

// KF: kF is given (with the choice in the loop, 277 and 289 us without and with it; 230 and 231 apart)
template <bool KF>
__global__ void __launch_bounds__(RS_THREADS) signal_speed_kernel(GridParams g, const double* rho, const double* T,
                                                                  const double* E, const double* v0, const double* v1,
                                                                  const double* v2, const double* kF, double dx_min,
                                                                  long long n, double* partial)
{
    constexpr float kClear = 1.0f - 0x1p-18f;
    __shared__ unsigned block_bits;  // the block's largest finite FP32 value so far (its bits: they order like it)
    if (threadIdx.x == 0) block_bits = 0;
    __syncthreads();
    const float gam = (float)g.gamma, inv_mu = (float)(1.0 / g.mu_over_kB), dxf = (float)dx_min;
    double m = 0.0;
    float top = -1.0f;  // FP32 value of the kept cell; -1: none yet
    SignalCell keep{};
    const long long stride = (long long)gridDim.x * RS_THREADS;
    for (long long i = (long long)blockIdx.x * RS_THREADS + threadIdx.x; i < n; i += stride) {
        SignalCell c;
        c.r = rho[i];
        c.T = T[i];
        c.E = E[i];
        c.v[0] = v0 ? v0[i] : 0.0;
        c.v[1] = v1 ? v1[i] : 0.0;
        c.v[2] = v2 ? v2[i] : 0.0;
        const float rf = d2f_trunc(c.r), af = d2f_trunc(c.v[0]), bf = d2f_trunc(c.v[1]), cf = d2f_trunc(c.v[2]);
        c.k = KF ? kF[i] : 0.0;
        const float kf = KF ? d2f_trunc(c.k) : (g.kpow == 0 ? g.f_kappa_F : (g.kpow == 1 ? g.f_kappa_F * rf : (g.f_kappa_F * rf) * rf));
        const float Pf = rf * d2f_trunc(c.T) * inv_mu;
        float radf = (4.0f / 9.0f) * d2f_trunc(c.E) * (-expm1f(-kf * dxf));
        if (KF) radf += kf - kf;
        const float q = gam * Pf + radf, s32 = sqrtf(af * af + bf * bf + cf * cf) + sqrtf(q / rf);
        const float seen = __uint_as_float(*(volatile unsigned*)&block_bits);
        if (s32 < seen * kClear && q > 1e-30f) continue;
        const bool plain = s32 < 3e38f && s32 > 1e-15f && q > 1e-30f;
        if (plain && s32 > seen) atomicMax(&block_bits, __float_as_uint(s32));
        if (plain && s32 < top * kClear) continue;
        if (!KF) c.k = flux_absorption(g, nullptr, rho, i);
        if (plain && s32 * kClear > top) {
            top = s32;
            keep = c;
            continue;
        }
        if (plain && (differs(c.r, keep.r) | differs(c.T, keep.T) | differs(c.E, keep.E) | differs(c.v[0], keep.v[0]) |
                      differs(c.v[1], keep.v[1]) | differs(c.v[2], keep.v[2]) | differs(c.k, keep.k)) == 0)
            continue;
        m = max_nan(m, signal_speed(g, c, dx_min));
    }
    __syncthreads();
    if (top >= 0.0f && !(top < __uint_as_float(block_bits) * kClear)) m = max_nan(m, signal_speed(g, keep, dx_min));
    block_max(m, partial);
}

// the largest sum of k_F dx_axis along the grid lines parallel to `axis` (cells indexed
// x + nx (y + ny z)); lines along y or z: one thread per line, consecutive threads on consecutive x;
// lines along x: one warp per line, lanes on strided x, then a fixed shuffle tree
__global__ void __launch_bounds__(RS_THREADS) line_depth_kernel(GridParams g, const double* kF, const double* rho,
                                                                int axis, double dx, double* partial)
{
    const long long nx = g.n[0], ny = g.n[1], nz = g.n[2];
    double m = 0.0;
    if (axis == 0) {
        const long long lines = ny * nz;
        const int lane = threadIdx.x & 31;
        const long long warp0 = ((long long)blockIdx.x * RS_THREADS + threadIdx.x) >> 5;
        const long long nwarps = ((long long)gridDim.x * RS_THREADS) >> 5;
        for (long long l = warp0; l < lines; l += nwarps) {
            double s = 0.0;
#pragma unroll 8
            for (long long x = lane; x < nx; x += 32) s += flux_absorption(g, kF, rho, l * nx + x);
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            m = max_nan(m, s * dx);
        }
    } else {
        const long long lines = axis == 1 ? nx * nz : nx * ny;
        const long long len = axis == 1 ? ny : nz, step = axis == 1 ? nx : nx * ny;
        for (long long l = (long long)blockIdx.x * RS_THREADS + threadIdx.x; l < lines;
             l += (long long)gridDim.x * RS_THREADS) {
            const long long x = l % nx, o = l / nx;  // o: z (axis y) or y (axis z)
            long long i = axis == 1 ? x + nx * ny * o : x + nx * o;
            double s = 0.0;
#pragma unroll 8
            for (long long k = 0; k < len; ++k, i += step) s += flux_absorption(g, kF, rho, i);
            m = max_nan(m, s * dx);
        }
    }
    block_max(m, partial);
}

__global__ void max_finish_kernel(const double* partial, int nb, double* out)
{
    double m = 0.0;
    for (int i = threadIdx.x; i < nb; i += RS_THREADS) m = max_nan(m, partial[i]);
    __shared__ double sh[RS_THREADS];
    sh[threadIdx.x] = m;
    __syncthreads();
    for (int s = RS_THREADS / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] = max_nan(sh[threadIdx.x], sh[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = max_nan(*out, sh[0]);
}

// blocks of every reduction launch (the partial buffer holds this many doubles + 1 for the result)
int rsla_blocks(int num_sms) { return num_sms * 4; }

cudaError_t launch_signal_speed(const GridParams& g, const double* rho, const double* T, const double* E,
                                const double* const v[3], const double* kF, double dx_min, long long n, int nb,
                                double* partial, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(partial + nb, 0, sizeof(double), s);
    if (e != cudaSuccess) return e;
    (kF ? signal_speed_kernel<true> : signal_speed_kernel<false>)<<<nb, RS_THREADS, 0, s>>>(g, rho, T, E, v[0], v[1], v[2], kF, dx_min, n, partial);
    max_finish_kernel<<<1, RS_THREADS, 0, s>>>(partial, nb, partial + nb);
    return cudaGetLastError();
}

cudaError_t launch_max_optical_depth(const GridParams& g, const double* kF, const double* rho, const double dx[3],
                                     int nb, double* partial, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(partial + nb, 0, sizeof(double), s);
    if (e != cudaSuccess) return e;
    for (int axis = 0; axis < 3; ++axis) {
        if (g.n[axis] <= 1) continue;
        line_depth_kernel<<<nb, RS_THREADS, 0, s>>>(g, kF, rho, axis, dx[axis], partial);
        max_finish_kernel<<<1, RS_THREADS, 0, s>>>(partial, nb, partial + nb);
    }
    return cudaGetLastError();
}

}  // namespace rhd
