// k_gas.cu -- the gas step around the radiation subcycles (Section 3.1 steps 3 and 6, Section 3.4):
// the Euler equations for (rho, rho v, E_gas) with the explicit gas sources S_e,gas of
// Eq. (algorithm:source:explicit:gas) (no gravity), advanced by one van Leer predictor / corrector step:
//
//   predictor: first-order HLLC fluxes of the ghost-filled state at t^n on the faces of the grid
//              extended by two ghost layers, then W^{n+1/2} on that extended grid (half step; sources
//              from the gas and the radiation at t^n);
//   corrector: limited piecewise-linear primitives of W^{n+1/2}, HLLC fluxes on the interior faces,
//              then the full step (sources from the gas at t^{n+1/2} and the radiation at t^n);
//   correction (after the subcycles): dt/2 [S_e,gas(W^{n+1/2}, U_rad^{n+1}) - S_e,gas(W^{n+1/2}, U_rad^n)].
//
// Split grids, and FP64 grids in 1D, take each half of the step in one launch, whose face fluxes stay in
// shared memory; FP64 grids in 2D and 3D store them (each computed once, by one thread) for an update launch.
// The HLLC solver (Toro, Riemann Solvers and Numerical
// Methods for Fluid Dynamics, Sec. 10.4) uses the Davis wave-speed estimates; the left star state when
// S* = 0; HLL where the contact speed's denominator is not negative.
//
// Precision: the kernels are templates on the arithmetic type R.  FP64 grids: R = double throughout.
// Split grids: R = float for reconstruction, wave speeds and HLLC (inputs truncated to FP32 by integer
// bit operations, FP32 fluxes stored), the flux differences and the sources; the half step W^{n+1/2} is
// an FP32 intermediate; the state (rho, v, T) accumulates FP32 increments in FP64, the pattern of the
// radiation's split path.  The increments of the primitive variables follow from those of the conserved
// ones (d rho, dM, dE) without cancellation: with rho' = rho + d rho,
//     dv = (dM - v d rho) / rho',   dK = (M.dv + dM.v') / 2   (the kinetic energy's change),
//     dT = ((gamma - 1) mu/k_B (dE - dK) - T d rho) / rho',
// so each is accurate relative to the increment itself, whatever the ratio of kinetic to internal
// energy, and the FP64 state gains FP64 additions only.  Divisions are reciprocals (FP64: the hardware
// approximation refined by Newton-Raphson; FP32: the hardware approximation) times the numerator.
#include <cuda_runtime.h>
#include <math.h>

#include "dfloat.cuh"
#include "fp_convert.cuh"
#include "gas_index.h"
#include "gas_internal.h"

namespace rhd {

namespace {

constexpr int GAS_THREADS = 256;

template <typename R>
struct Prim {
    R r, v[3], P;
};

template <typename R>
__device__ __forceinline__ R flip(R x, int s)
{
    return s < 0 ? -x : x;
}

// physical constants in R
template <typename R>
struct Consts {
    R gamma, inv_gm1, inv_mu;
};
template <typename R>
__device__ __forceinline__ Consts<R> consts(const GasParams& p);
template <>
__device__ __forceinline__ Consts<double> consts<double>(const GasParams& p)
{
    return {p.gamma, p.inv_gm1, p.inv_mu};
}
template <>
__device__ __forceinline__ Consts<float> consts<float>(const GasParams& p)
{
    return {p.f_gamma, p.f_inv_gm1, p.f_inv_mu};
}

// the gas state at t^n of interior cell i, with the normal velocity components of a mirrored ghost
// cell flipped (s)
__device__ __forceinline__ Prim<double> load_prim(const GasParams& p, const GasArrays& a, long long i, const int s[3])
{
    Prim<double> w;
    w.r = a.rho[i];
    for (int d = 0; d < 3; ++d) w.v[d] = flip(a.v[d][i], s[d]);
    w.P = w.r * a.T[i] * p.inv_mu;
    return w;
}

template <typename R>
__device__ __forceinline__ R kin2(const Prim<R>& w)
{
    return w.v[0] * w.v[0] + w.v[1] * w.v[1] + w.v[2] * w.v[2];
}

// (rho, Mx, My, Mz, E_gas) of a primitive state (FP64)
__device__ __forceinline__ void to_cons(const GasParams& p, const Prim<double>& w, double U[5])
{
    U[0] = w.r;
    for (int d = 0; d < 3; ++d) U[1 + d] = w.r * w.v[d];
    U[4] = w.P * p.inv_gm1 + 0.5 * w.r * kin2(w);
}

// primitive state of U (FP64); a negative internal energy is floored to zero (returns true then).
// inv_r receives 1/rho.
__device__ __forceinline__ bool to_prim(const GasParams& p, const double U[5], Prim<double>& w, double& inv_r)
{
    w.r = U[0];
    inv_r = rcp(U[0]);
    for (int d = 0; d < 3; ++d) w.v[d] = U[1 + d] * inv_r;
    double e = U[4] - 0.5 * (U[1] * w.v[0] + U[2] * w.v[1] + U[3] * w.v[2]);
    const bool neg = e < 0.0;
    if (neg) e = 0.0;
    w.P = p.gm1 * e;
    return neg;
}

template <typename R, int D>
__device__ __forceinline__ void euler_flux(const Consts<R>& k, const Prim<R>& w, R F[5], R& E)
{
    const R u = w.v[D];
    E = w.P * k.inv_gm1 + R(0.5) * w.r * kin2(w);
    F[0] = w.r * u;
    for (int q = 0; q < 3; ++q) F[1 + q] = w.r * w.v[q] * u;
    F[1 + D] += w.P;
    F[4] = (E + w.P) * u;
}

// HLL, where the contact speed's denominator is not negative (inlined: a call's stack and registers cost the
// marching kernels 20 to 30 %, though it all but never runs)
template <typename R, int D>
__device__ __forceinline__ void hll_flux(const Consts<R>& k, const Prim<R>& L, const Prim<R>& Rt, R SL, R SR, R F[5])
{
    R FL[5], FR[5], EL, ER;
    euler_flux<R, D>(k, L, FL, EL);
    euler_flux<R, D>(k, Rt, FR, ER);
    const R UL[5] = {L.r, L.r * L.v[0], L.r * L.v[1], L.r * L.v[2], EL};
    const R UR[5] = {Rt.r, Rt.r * Rt.v[0], Rt.r * Rt.v[1], Rt.r * Rt.v[2], ER};
    const R iw = rcp(SR - SL);
    for (int q = 0; q < 5; ++q) F[q] = (SR * FL[q] - SL * FR[q] + SL * SR * (UR[q] - UL[q])) * iw;
}

// products and sums that the compiler does not contract any further
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// The flux through a face between L and Rt.  Only one side's flux is needed wherever the contact speed exists: the
// side is chosen first (supersonic: the upwind one; else the contact's), its flux formed, and the star state's jump
// added.  The products that the jump is added to are rounded by themselves.
template <typename R, int D>
__device__ __forceinline__ void hllc(const Consts<R>& k, const Prim<R>& L, const Prim<R>& Rt, R F[5])
{
    const R irL = rcp(L.r), irR = rcp(Rt.r);
    const R aL = sqrt_fast(k.gamma * L.P * irL), aR = sqrt_fast(k.gamma * Rt.P * irR);
    const R uL = L.v[D], uR = Rt.v[D];
    const R SL = fmin(uL - aL, uR - aR), SR = fmax(uL + aL, uR + aR);
    const R den = L.r * (SL - uL) - Rt.r * (SR - uR);
    const bool supL = SL >= R(0), supR = SR <= R(0);
    if (!(supL || supR || den < R(0))) {
        hll_flux<R, D>(k, L, Rt, SL, SR, F);
        return;
    }
    const R Ss = (Rt.P - L.P + L.r * uL * (SL - uL) - Rt.r * uR * (SR - uR)) * rcp(den);
    const bool left = supL || (!supR && Ss >= R(0));
    Prim<R> K;
    K.r = left ? L.r : Rt.r;
    for (int q = 0; q < 3; ++q) K.v[q] = left ? L.v[q] : Rt.v[q];
    K.P = left ? L.P : Rt.P;
    const R S = left ? SL : SR, irK = left ? irL : irR, uK = K.v[D];
    R EK, M[3];
    for (int q = 0; q < 3; ++q) M[q] = mul_rn(K.r, K.v[q]);
    EK = K.P * k.inv_gm1 + R(0.5) * K.r * kin2(K);
    F[0] = M[D];
    for (int q = 0; q < 3; ++q) F[1 + q] = q == D ? fma_rn(M[q], uK, K.P) : mul_rn(M[q], uK);
    F[4] = mul_rn(EK + K.P, uK);
    if (!(supL || supR)) {
        const R chi = K.r * (S - uK) * rcp(S - Ss);
        R Us[5];
        Us[0] = chi;
        for (int q = 0; q < 3; ++q) Us[1 + q] = chi * K.v[q];
        Us[1 + D] = chi * Ss;
        Us[4] = chi * (EK * irK + (Ss - uK) * (Ss + K.P * irK * rcp(S - uK)));
        const R UK[5] = {K.r, K.r * K.v[0], K.r * K.v[1], K.r * K.v[2], EK};
        for (int q = 0; q < 5; ++q) F[q] = F[q] + S * (Us[q] - UK[q]);
    }
}

template <typename R>
__device__ __forceinline__ R limited_slope(R dl, R dr, int lim)
{
    if (lim == 2) return R(0.5) * (dl + dr);  // no limiter
    if (dl * dr <= R(0)) return R(0);
    R m = fmin(fabs(dl), fabs(dr));                                   // minmod
    if (lim != 0) m = fmin(R(2) * m, R(0.5) * fabs(dl + dr));  // monotonized central
    return dl > R(0) ? m : -m;
}

__device__ __forceinline__ double absorption(const GasParams& p, const double* kF, long long i, double rho)
{
    if (kF) return kF[i];
    return p.kpow == 0 ? p.kappa_F : (p.kpow == 1 ? p.kappa_F * rho : (p.kappa_F * rho) * rho);
}

// S_e,gas rows of rho v and E_gas: k (G - (4/3) v E / c) and -k v.G (the terms with v only when beta tau is on)
__device__ __forceinline__ void gas_source(const GasParams& p, double k, const double v[3], double E, const double G[3],
                                           double S[5])
{
    S[0] = 0.0;
    if (p.beta_tau) {
        for (int d = 0; d < 3; ++d) S[1 + d] = k * (G[d] - (4.0 / 3.0) * v[d] * E * p.inv_c);
        S[4] = -k * (v[0] * G[0] + v[1] * G[1] + v[2] * G[2]);
    } else {
        for (int d = 0; d < 3; ++d) S[1 + d] = k * G[d];
        S[4] = 0.0;
    }
}

// split grids: the same sources in FP32 (k from the FP64 array truncated, or the law in FP32)
__device__ __forceinline__ float absorption32(const GasParams& p, const double* kF, long long i, float rho)
{
    if (kF) return d2f_trunc(kF[i]);
    return p.kpow == 0 ? p.f_kappa_F : (p.kpow == 1 ? p.f_kappa_F * rho : (p.f_kappa_F * rho) * rho);
}
__device__ __forceinline__ void gas_source32(const GasParams& p, float k, const float v[3], float E, const float G[3],
                                             float S[5])
{
    S[0] = 0.0f;
    if (p.beta_tau) {
        for (int d = 0; d < 3; ++d) S[1 + d] = k * (G[d] - (4.0f / 3.0f) * v[d] * E * p.f_inv_c);
        S[4] = -k * (v[0] * G[0] + v[1] * G[1] + v[2] * G[2]);
    } else {
        for (int d = 0; d < 3; ++d) S[1 + d] = k * G[d];
        S[4] = 0.0f;
    }
}

// Tests of FP64 values by their bits, on the integer pipes (an FP64 comparison occupies the FP64 pipe,
// which the split kernels otherwise leave to the accumulation): finite, and below zero (not -0, not NaN)
__device__ __forceinline__ bool finite_bits(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) != 0x7ff; }
__device__ __forceinline__ bool below_zero_bits(double x)
{
    const long long b = __double_as_longlong(x);
    return b < 0 && b != (long long)0x8000000000000000ull && finite_bits(x);
}

// Increments of the primitive variables from those of the conserved ones, D = (d rho, dMx, dMy, dMz,
// dE), at a state (r, v, T) in FP32: dv, dT and rho' = r + d rho (see the precision note above).
struct PrimInc {
    float r1, dv[3], dT;
};
__device__ __forceinline__ PrimInc prim_increment(const GasParams& p, float r, const float v[3], float T,
                                                  const float D[5])
{
    PrimInc o;
    o.r1 = r + D[0];
    const float inv = rcp(o.r1);
    float dK2 = 0.0f;  // 2 dK = M.dv + dM.v'
    for (int d = 0; d < 3; ++d) {
        o.dv[d] = (D[1 + d] - v[d] * D[0]) * inv;
        dK2 += r * v[d] * o.dv[d] + D[1 + d] * (v[d] + o.dv[d]);
    }
    o.dT = (p.f_gm1_mu * (D[4] - 0.5f * dK2) - T * D[0]) * inv;
    return o;
}

__device__ __forceinline__ bool finite_prim(const Prim<double>& w)
{
    return isfinite(w.r) && isfinite(w.v[0]) && isfinite(w.v[1]) && isfinite(w.v[2]) && isfinite(w.P);
}

__device__ __forceinline__ long long first_index() { return (long long)blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ long long index_stride() { return (long long)gridDim.x * blockDim.x; }

// minus the divergence of the stored face fluxes
__device__ __forceinline__ void flux_divergence(const GasParams& p, const GasArrays& a, const long long lo[3],
                                                const long long hi[3], double dU[5])
{
    for (int q = 0; q < 5; ++q) dU[q] = 0.0;
    for (int d = 0; d < 3; ++d) {
        if (p.n[d] <= 1) continue;
        for (int q = 0; q < 5; ++q) dU[q] -= (a.flux[d][q][hi[d]] - a.flux[d][q][lo[d]]) * p.inv_dx[d];
    }
}

// ---------------------------------------------------------------------------------------- a cell's steps

// half step of extended cell i (interior cell k mirrored with the signs s): W^{n+1/2} from minus the flux
// divergence dU and the sources at t^n; true if the internal energy was floored
__device__ __forceinline__ bool pred_update(const GasParams& p, const GasArrays& a, long long i, long long k,
                                            const int s[3], const double dU[5])
{
    const double hdt = 0.5 * p.dt;
    const Prim<double> W = load_prim(p, a, k, s);
    double U[5];
    to_cons(p, W, U);
    const double G[3] = {flip(a.G[0][k], s[0]), flip(a.G[1][k], s[1]), flip(a.G[2][k], s[2])};
    double S[5];
    gas_source(p, absorption(p, a.kF, k, W.r), W.v, a.E[k], G, S);
    double Uh[5], inv_r;
    for (int q = 0; q < 5; ++q) Uh[q] = U[q] + hdt * dU[q] + hdt * S[q];
    Prim<double> Wh;
    const bool neg = to_prim(p, Uh, Wh, inv_r);
    const double w5[5] = {Wh.r, Wh.v[0], Wh.v[1], Wh.v[2], Wh.P};
    for (int q = 0; q < 5; ++q) a.wh[q][i] = w5[q];
    return neg;
}

// full step of interior cell i (extended cell x), and the record the source correction needs
__device__ __forceinline__ void corr_update(const GasParams& p, const GasArrays& a, long long i, long long x,
                                            const double dU[5], unsigned long long& floors, unsigned long long& bad)
{
    const int one[3] = {1, 1, 1};
    const Prim<double> W = load_prim(p, a, i, one);
    double U[5];
    to_cons(p, W, U);
    const double rh = a.wh[0][x];
    const double vh[3] = {a.wh[1][x], a.wh[2][x], a.wh[3][x]};
    const double kh = absorption(p, a.kF, i, rh);
    const double E = a.E[i];
    const double G[3] = {a.G[0][i], a.G[1][i], a.G[2][i]};
    double S[5];
    gas_source(p, kh, vh, E, G, S);
    double U1[5], inv_r;
    for (int q = 0; q < 5; ++q) U1[q] = U[q] + p.dt * dU[q] + p.dt * S[q];
    Prim<double> W1;
    if (to_prim(p, U1, W1, inv_r)) ++floors;
    if (!finite_prim(W1)) ++bad;
    a.rho[i] = W1.r;
    for (int d = 0; d < 3; ++d) a.v[d][i] = W1.v[d];
    a.T[i] = W1.P * p.mu_over_kB * inv_r;
    a.pend[0][i] = kh;
    for (int d = 0; d < 3; ++d) a.pend[1 + d][i] = vh[d];
    a.pend[4][i] = E;
    for (int d = 0; d < 3; ++d) a.pend[5 + d][i] = G[d];
}

// limited slopes of a cell; a slope whose face values have rho <= 0 or P <= 0 is zeroed (all components)
template <typename R>
__device__ __forceinline__ void cell_slopes(const R wm[5], const R w0[5], const R wp[5], int lim, R sl[5])
{
    for (int q = 0; q < 5; ++q) sl[q] = limited_slope<R>(w0[q] - wm[q], wp[q] - w0[q], lim);
    bool bad = false;
    for (int hs = 0; hs < 2; ++hs) {
        const R sg = hs ? R(0.5) : R(-0.5);
        bad = bad || !(w0[0] + sg * sl[0] > R(0)) || !(w0[4] + sg * sl[4] > R(0));
    }
    if (bad)
        for (int q = 0; q < 5; ++q) sl[q] = R(0);
}

// the cell's state at its high (h = 1/2) or low (h = -1/2) face
template <typename R>
__device__ __forceinline__ Prim<R> face_state(const R w0[5], const R sl[5], R h)
{
    Prim<R> W;
    W.r = w0[0] + h * sl[0];
    for (int q = 0; q < 3; ++q) W.v[q] = w0[1 + q] + h * sl[1 + q];
    W.P = w0[4] + h * sl[4];
    return W;
}

// ------------------------------------------------------------- FP64 grids in 2D and 3D: a launch per direction

template <int D>
__global__ void __launch_bounds__(GAS_THREADS) gas_pred_flux_kernel(GasParams p, GasArrays a)
{
    int fe[3];
    gas_pred_faces(p, D, fe);
    const long long nf = gas_count(fe);
    const Consts<double> k = consts<double>(p);
    for (long long f = first_index(); f < nf; f += index_stride()) {
        long long iL, iR;
        int sL[3], sR[3];
        gas_pred_flux_cells(p, D, f, &iL, sL, &iR, sR);
        const Prim<double> WL = load_prim(p, a, iL, sL), WR = load_prim(p, a, iR, sR);
        double F[5];
        hllc<double, D>(k, WL, WR, F);
        for (int q = 0; q < 5; ++q) a.flux[D][q][f] = F[q];
    }
}

__global__ void __launch_bounds__(GAS_THREADS) gas_pred_update_kernel(GasParams p, GasArrays a)
{
    const long long ne = gas_count(p.m);
    unsigned long long floors = 0;
    for (long long i = first_index(); i < ne; i += index_stride()) {
        long long k, lo[3], hi[3];
        int s[3];
        bool inside;
        gas_pred_update_cells(p, i, &k, s, &inside, lo, hi);
        double dU[5];
        flux_divergence(p, a, lo, hi, dU);
        if (pred_update(p, a, i, k, s, dU) && inside) ++floors;
    }
    if (floors) atomicAdd(&a.counters[0], floors);
}

template <int D>
__global__ void __launch_bounds__(GAS_THREADS) gas_corr_flux_kernel(GasParams p, GasArrays a)
{
    int fe[3];
    gas_corr_faces(p, D, fe);
    const long long nf = gas_count(fe);
    const Consts<double> k = consts<double>(p);
    for (long long f = first_index(); f < nf; f += index_stride()) {
        // W^{n+1/2} of the cells f - 2 e_D .. f + e_D
        long long x[4];
        gas_corr_flux_cells(p, D, f, x);
        double w[4][5], sl[5];
        for (int j = 0; j < 4; ++j)
            for (int q = 0; q < 5; ++q) w[j][q] = a.wh[q][x[j]];
        cell_slopes(w[0], w[1], w[2], p.limiter, sl);
        const Prim<double> WL = face_state(w[1], sl, 0.5);
        cell_slopes(w[1], w[2], w[3], p.limiter, sl);
        const Prim<double> WR = face_state(w[2], sl, -0.5);
        double F[5];
        hllc<double, D>(k, WL, WR, F);
        for (int q = 0; q < 5; ++q) a.flux[D][q][f] = F[q];
    }
}

__global__ void __launch_bounds__(GAS_THREADS) gas_corr_update_kernel(GasParams p, GasArrays a)
{
    const long long nc = gas_count(p.n);
    unsigned long long floors = 0, bad = 0;
    for (long long i = first_index(); i < nc; i += index_stride()) {
        long long x, lo[3], hi[3];
        gas_corr_update_cells(p, i, &x, lo, hi);
        double dU[5];
        flux_divergence(p, a, lo, hi, dU);
        corr_update(p, a, i, x, dU, floors, bad);
    }
    if (floors) atomicAdd(&a.counters[0], floors);
    if (bad) atomicAdd(&a.counters[1], bad);
}

// ------------------------------------------- split grids, and FP64 grids in 1D: one launch for a half of the step
//
// A CTA takes a tile of x and y and marches its planes in z.  Each face's flux is computed by the thread of the
// cell above it (x and y: passed to the cell below through shared memory; z: kept in registers for the next
// plane), the faces that close the tile by two more warps (one for the row above it, one for the column).
// Nothing but the half step's result goes through memory: a launch for each direction that stored its faces' five
// components, and an update that read them back, moved 20 B a cell and direction there and again 20 B back.
// Same arithmetic, operation for operation.  Bound by instruction issue (HLLC and the limiter; the launches per
// direction were bound by memory).  256^3, us: five launches of fluxes and updates a half 1176 and 1467, marched 554
// and 1004; the step and its correction, 300 x 250 x 200: 2.8 ms, and the copies by five launches, -> 2.1 with the copies;
// FP64, 512 cells: 54 -> 28 us.

// the FP32 radiation state of interior cell i: the two-pass subcycles' mirror where it is current
__device__ __forceinline__ float4 load_rad32(const GasArrays& a, long long i)
{
    if (a.um32) return a.um32[i];
    return make_float4(d2f_trunc(a.E[i]), d2f_trunc(a.G[0][i]), d2f_trunc(a.G[1][i]), d2f_trunc(a.G[2][i]));
}

// split grids: the new velocity and the FP32 copies the subcycles read
__device__ __forceinline__ void store_velocity(const GasArrays& a, long long i, float r32, const double v1[3])
{
    const float f[3] = {to_f32(v1[0]), to_f32(v1[1]), to_f32(v1[2])};
    for (int d = 0; d < 3; ++d) {
        a.v[d][i] = v1[d];
        a.v32[d][i] = f[d];
    }
    if (a.gas4) a.gas4[i] = make_float4(r32, f[0], f[1], f[2]);
}

// a cell of W^n as it lies in memory (split grids: the FP32 copies), its mirrored normal components flipped
template <typename R>
struct GasCell {
    R r, v[3], T;
};
template <typename R>
__device__ __forceinline__ GasCell<R> load_cell(const GasArrays& a, long long k, int s0, int s1, int s2)
{
    if constexpr (sizeof(R) == 4)
        return {a.rho32[k], {flip(a.v32[0][k], s0), flip(a.v32[1][k], s1), flip(a.v32[2][k], s2)}, d2f_trunc(a.T[k])};
    else
        return {a.rho[k], {flip(a.v[0][k], s0), flip(a.v[1][k], s1), flip(a.v[2][k], s2)}, a.T[k]};
}
template <typename R>
__device__ __forceinline__ Prim<R> prim_of(const GasParams& p, const GasCell<R>& c)
{
    Prim<R> w;
    w.r = c.r;
    for (int d = 0; d < 3; ++d) w.v[d] = c.v[d];
    if constexpr (sizeof(R) == 4) w.P = c.r * c.T * p.f_inv_mu;
    else w.P = c.r * c.T * p.inv_mu;
    return w;
}

// W^{n+1/2} of extended cell x
template <typename R>
struct GasHalf {
    R w[5];
};
template <typename R>
__device__ __forceinline__ GasHalf<R> load_half(const GasArrays& a, long long x)
{
    if constexpr (sizeof(R) == 4) {
        const float4 h = a.wh4[x];
        return {{h.x, h.y, h.z, h.w, a.whP[x]}};
    } else {
        return {{a.wh[0][x], a.wh[1][x], a.wh[2][x], a.wh[3][x], a.wh[4][x]}};
    }
}

// dU -= (hi - lo) / dx, the difference rounded by itself (as of values that come from memory)
__device__ __forceinline__ void add_divergence(const GasParams& p, int d, float lo, float hi, float& dU)
{
    dU -= __fsub_rn(hi, lo) * p.f_inv_dx[d];
}
__device__ __forceinline__ void add_divergence(const GasParams& p, int d, double lo, double hi, double& dU)
{
    dU -= __dsub_rn(hi, lo) * p.inv_dx[d];
}

// Resident CTAs asked of the compiler.  The fluxes' chains leave half of the issue slots empty at the two CTAs that
// the unbounded kernels' registers allow; a few spilled values cost less.  256^3 and 300 x 250 x 200, us:
// predictor (95 registers unbounded) 633 and 688 at two, 575 and 586 at three, 560 and 547 at four; corrector (113)
// 955 and 1089 at two, 1013 and 1057 at three, 1211 and 1333 at four.
template <typename R, int DIM>
constexpr int gas_min_blocks(int n)
{
    return sizeof(R) == 4 && DIM > 1 ? n : 1;
}

// faces of one plane, for the cells below them
template <typename R, int DIM, int TX, int TY>
struct GasFaces {
    R x[5][TY][TX + 1];
    R y[DIM > 1 ? 5 : 1][DIM > 1 ? TY + 1 : 1][DIM > 1 ? TX : 1];
};

template <typename R, int DIM, int TX, int TY>
__device__ __forceinline__ void tile_divergence(const GasParams& p, const GasFaces<R, DIM, TX, TY>& f, int tx, int ty,
                                                const R zlo[5], const R zhi[5], R dU[5])
{
    for (int q = 0; q < 5; ++q) {
        dU[q] = R(0);
        if (p.n[0] > 1) add_divergence(p, 0, f.x[q][ty][tx], f.x[q][ty][tx + 1], dU[q]);
        if constexpr (DIM > 1) add_divergence(p, 1, f.y[q][ty][tx], f.y[q][ty + 1][tx], dU[q]);
        if constexpr (DIM > 2) add_divergence(p, 2, zlo[q], zhi[q], dU[q]);
    }
}

template <typename R, int DIM, int TX, int TY>
__global__ void __launch_bounds__((GasTile<DIM, TX, TY>::NT), gas_min_blocks<R, DIM>(4)) gas_predictor_kernel(const __grid_constant__ GasParams p,
                                                                                 const __grid_constant__ GasArrays a,
                                                                                 const GasMarch t)
{
    __shared__ GasFaces<R, DIM, TX, TY> faces[DIM > 2 ? 2 : 1];
    const GasTile<DIM, TX, TY> me(threadIdx.x);
    const Consts<R> kc = consts<R>(p);
    const int b = (int)(blockIdx.x % t.tiles), zc = (int)(blockIdx.x / t.tiles) * t.planes;
    const int ze = zc + t.planes < p.m[2] ? zc + t.planes : p.m[2];
    const int X = (b % t.tiles_x) * TX + me.tx, Y = (b / t.tiles_x) * TY + me.ty;
    const bool cell = me.cell && gas_cell_in(X, Y, p.m[0], p.m[1]);
    const bool fx = me.fx && p.n[0] > 1 && gas_xface_in(X, Y, p.m[0], p.m[1]);
    const bool fy = me.fy && gas_yface_in(X, Y, p.m[0], p.m[1]);
    // the interior cell under the thread's own, and under its low neighbours in x and y
    const GasPredColumn col = gas_pred_column(p, X, Y);
    const int sx = col.sx, sy = col.sy, sxl = col.sxl, syl = col.syl;
    const long long own = col.own, left = col.left, low = col.low, plane = (long long)p.n[0] * p.n[1];
    const bool in_xy = X >= p.g[0] && X < p.g[0] + p.n[0] && Y >= p.g[1] && Y < p.g[1] + p.n[1];
    unsigned long long floors = 0;

    int sz = 1, szn = 1;
    int z = DIM > 2 ? zc - 1 : 0;  // 3D: the plane below the chunk gives the flux through its lowest face
    long long base = DIM > 2 ? gas_pred_plane(p, plane, z, sz) : 0, base_n = 0;
    GasCell<R> cur = load_cell<R>(a, own + base, sx, sy, sz), nxt = cur;
    R zlo[5], zhi[5];
    for (int q = 0; q < 5; ++q) zlo[q] = zhi[q] = R(0);
    for (; z < ze; ++z) {
        const bool on = DIM < 3 || z >= zc;
        GasFaces<R, DIM, TX, TY>& f = faces[DIM > 2 ? z & 1 : 0];
        if constexpr (DIM > 2) {
            base_n = gas_pred_plane(p, plane, z + 1, szn);
            if (cell || z + 1 < ze) nxt = load_cell<R>(a, own + base_n, sx, sy, szn);
        }
        float4 u = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        float kf = 0.0f;
        if (on) {
            if constexpr (sizeof(R) == 4)
                if (cell) {
                    u = load_rad32(a, own + base);
                    kf = absorption32(p, a.kF, own + base, cur.r);
                }
            if (fx) {
                const GasCell<R> l = load_cell<R>(a, left + base, sxl, sy, sz);
                R F[5];
                hllc<R, 0>(kc, prim_of(p, l), prim_of(p, cur), F);
                for (int q = 0; q < 5; ++q) f.x[q][me.ty][me.tx] = F[q];
            }
            if constexpr (DIM > 1)
                if (fy) {
                    const GasCell<R> l = load_cell<R>(a, low + base, sx, syl, sz);
                    R F[5];
                    hllc<R, 1>(kc, prim_of(p, l), prim_of(p, cur), F);
                    for (int q = 0; q < 5; ++q) f.y[q][me.ty][me.tx] = F[q];
                }
        }
        if constexpr (DIM > 2)
            if (cell) hllc<R, 2>(kc, prim_of(p, cur), prim_of(p, nxt), zhi);
        if (on) {
            __syncthreads();
            if (cell) {
                R dU[5];
                tile_divergence(p, f, me.tx, me.ty, zlo, zhi, dU);
                const int at[3] = {X, Y, z};
                const long long i = gas_ravel(at, p.m);
                const bool inside = in_xy && (DIM < 3 || (z >= p.g[2] && z < p.g[2] + p.n[2]));
                if constexpr (sizeof(R) == 4) {
                    // W^{n+1/2} in FP32 from the FP32 copies of W^n and FP32 increments
                    const float fh = (float)(0.5 * p.dt);
                    float S[5], D[5];
                    const float G[3] = {flip(u.y, sx), flip(u.z, sy), flip(u.w, sz)};
                    gas_source32(p, kf, cur.v, u.x, G, S);
                    for (int q = 0; q < 5; ++q) D[q] = fh * (dU[q] + S[q]);
                    const PrimInc o = prim_increment(p, cur.r, cur.v, cur.T, D);
                    float Th = cur.T + o.dT;
                    if (Th < 0.0f) {
                        Th = 0.0f;
                        if (inside) ++floors;
                    }
                    a.wh4[i] = make_float4(o.r1, cur.v[0] + o.dv[0], cur.v[1] + o.dv[1], cur.v[2] + o.dv[2]);
                    a.whP[i] = o.r1 * Th * p.f_inv_mu;
                } else {
                    const int s[3] = {sx, sy, sz};
                    if (pred_update(p, a, i, own + base, s, dU) && inside) ++floors;
                }
            }
        }
        cur = nxt;
        base = base_n;
        sz = szn;
        for (int q = 0; q < 5; ++q) zlo[q] = zhi[q];
    }
    if (floors) atomicAdd(&a.counters[0], floors);
}

// LIM: the limiter, -1: p.limiter
template <typename R, int DIM, int TX, int TY, int LIM>
__global__ void __launch_bounds__((GasTile<DIM, TX, TY>::NT), gas_min_blocks<R, DIM>(3)) gas_corrector_kernel(const __grid_constant__ GasParams p,
                                                                                 const __grid_constant__ GasArrays a,
                                                                                 const GasMarch t)
{
    __shared__ GasFaces<R, DIM, TX, TY> faces[DIM > 2 ? 2 : 1];
    const GasTile<DIM, TX, TY> me(threadIdx.x);
    const Consts<R> kc = consts<R>(p);
    const int b = (int)(blockIdx.x % t.tiles), zc = (int)(blockIdx.x / t.tiles) * t.planes;
    const int ze = zc + t.planes < p.n[2] ? zc + t.planes : p.n[2];
    const int X = (b % t.tiles_x) * TX + me.tx, Y = (b / t.tiles_x) * TY + me.ty;
    const bool cell = me.cell && gas_cell_in(X, Y, p.n[0], p.n[1]);
    const bool fx = me.fx && p.n[0] > 1 && gas_xface_in(X, Y, p.n[0], p.n[1]);
    const bool fy = me.fy && gas_yface_in(X, Y, p.n[0], p.n[1]);
    const bool any = cell || fx || fy;
    const int lim = LIM >= 0 ? LIM : p.limiter;
    const long long row = p.m[0], plane = row * p.m[1];
    // the thread's extended cell in plane z is own + plane * z
    const long long own = gas_corr_column(p, X, Y);
    unsigned long long floors = 0, bad = 0;

    // 3D: cells z, z + 1 and z + 2 of the thread's column; the slope of z + 1 gives its states at the faces z + 1
    // and z + 2, the flux through face z + 1 closes cell z.  Two planes below the chunk start the chain.
    int z = DIM > 2 ? zc - 2 : 0;
    GasHalf<R> w0{}, w1{}, w2{};
    Prim<R> up{};  // state of cell z at its high z face
    R zlo[5], zhi[5];
    for (int q = 0; q < 5; ++q) zlo[q] = zhi[q] = R(0);
    if (any) {
        w0 = load_half<R>(a, own + plane * z);
        if constexpr (DIM > 2) w1 = load_half<R>(a, own + plane * (z + 1));
    }
    for (; z < ze; ++z) {
        const bool on = DIM < 3 || z >= zc;
        GasFaces<R, DIM, TX, TY>& f = faces[DIM > 2 ? z & 1 : 0];
        const long long x = own + plane * z;
        R sl[5];
        if constexpr (DIM > 2)
            if (cell || (any && z + 2 < ze)) w2 = load_half<R>(a, x + 2 * plane);
        if (on) {
            if (fx) {
                const GasHalf<R> a0 = load_half<R>(a, x - 2), a1 = load_half<R>(a, x - 1), a3 = load_half<R>(a, x + 1);
                cell_slopes(a0.w, a1.w, w0.w, lim, sl);
                const Prim<R> L = face_state(a1.w, sl, R(0.5));
                cell_slopes(a1.w, w0.w, a3.w, lim, sl);
                R F[5];
                hllc<R, 0>(kc, L, face_state(w0.w, sl, R(-0.5)), F);
                for (int q = 0; q < 5; ++q) f.x[q][me.ty][me.tx] = F[q];
            }
            if constexpr (DIM > 1)
                if (fy) {
                    const GasHalf<R> a0 = load_half<R>(a, x - 2 * row), a1 = load_half<R>(a, x - row),
                                     a3 = load_half<R>(a, x + row);
                    cell_slopes(a0.w, a1.w, w0.w, lim, sl);
                    const Prim<R> L = face_state(a1.w, sl, R(0.5));
                    cell_slopes(a1.w, w0.w, a3.w, lim, sl);
                    R F[5];
                    hllc<R, 1>(kc, L, face_state(w0.w, sl, R(-0.5)), F);
                    for (int q = 0; q < 5; ++q) f.y[q][me.ty][me.tx] = F[q];
                }
        }
        if constexpr (DIM > 2)
            if (cell) {
                cell_slopes(w0.w, w1.w, w2.w, lim, sl);
                if (z >= zc - 1) hllc<R, 2>(kc, up, face_state(w1.w, sl, R(-0.5)), zhi);
                up = face_state(w1.w, sl, R(0.5));
            }
        if (on) {
            __syncthreads();
            if (cell) {
                R dU[5];
                tile_divergence(p, f, me.tx, me.ty, zlo, zhi, dU);
                const int at[3] = {X, Y, z};
                const long long i = gas_ravel(at, p.n);
                if constexpr (sizeof(R) == 4) {
                    // FP32 increments (fluxes, sources at W^{n+1/2}) accumulated into the FP64 state
                    const float fdt = (float)p.dt;
                    const double rho = a.rho[i], T = a.T[i];
                    const double v[3] = {a.v[0][i], a.v[1][i], a.v[2][i]};
                    const float v32[3] = {d2f_trunc(v[0]), d2f_trunc(v[1]), d2f_trunc(v[2])};
                    const float vh[3] = {w0.w[1], w0.w[2], w0.w[3]};
                    const float kh = absorption32(p, a.kF, i, w0.w[0]);
                    const float4 u = load_rad32(a, i);
                    const float G[3] = {u.y, u.z, u.w};
                    float S[5], D[5];
                    gas_source32(p, kh, vh, u.x, G, S);
                    for (int q = 0; q < 5; ++q) D[q] = fdt * (dU[q] + S[q]);
                    const PrimInc o = prim_increment(p, d2f_trunc(rho), v32, d2f_trunc(T), D);
                    const double rho1 = rho + f2d_exact(D[0]);
                    double T1 = T + f2d_exact(o.dT);
                    if (below_zero_bits(T1)) {
                        T1 = 0.0;
                        ++floors;
                    }
                    double v1[3];
                    for (int d = 0; d < 3; ++d) v1[d] = v[d] + f2d_exact(o.dv[d]);
                    if (!(finite_bits(rho1) && finite_bits(v1[0]) && finite_bits(v1[1]) && finite_bits(v1[2]) &&
                          finite_bits(T1)))
                        ++bad;
                    const float r32 = to_f32(rho1);
                    a.rho[i] = rho1;
                    a.rho32[i] = r32;
                    a.T[i] = T1;
                    store_velocity(a, i, r32, v1);
                    a.rad4[i] = u;  // the radiation at t^n, for the correction (k_F and v^{n+1/2}: from W^{n+1/2})
                } else {
                    corr_update(p, a, i, x, dU, floors, bad);
                }
            }
        }
        w0 = w1;
        w1 = w2;
        for (int q = 0; q < 5; ++q) zlo[q] = zhi[q];
    }
    if (floors) atomicAdd(&a.counters[0], floors);
    if (bad) atomicAdd(&a.counters[1], bad);
}

// ---------------------------------------------------------------------------------------- correction

template <bool SPLIT>
__global__ void __launch_bounds__(GAS_THREADS) gas_correct_kernel(const __grid_constant__ GasParams p,
                                                                  const __grid_constant__ GasArrays a)
{
    const long long nc = gas_count(p.n);
    const double hdt = 0.5 * p.dt;
    unsigned long long floors = 0, bad = 0;
    if constexpr (SPLIT) {
        // split grids: the change of the sources in FP32 (the radiation's change as the difference of its
        // FP32 copies: its error is that of the FP32 sources themselves), its momentum and energy
        // increments accumulated into the FP64 state
        const float fh = (float)hdt;
        for (long long i = first_index(); i < nc; i += index_stride()) {
            int c[3];
            gas_unravel(i, p.n, c);
            for (int d = 0; d < 3; ++d) c[d] += p.g[d];
            const float4 h = a.wh4[gas_ravel(c, p.m)];
            const double rho = a.rho[i], T = a.T[i];
            const double v[3] = {a.v[0][i], a.v[1][i], a.v[2][i]};
            const float v32[3] = {d2f_trunc(v[0]), d2f_trunc(v[1]), d2f_trunc(v[2])};
            const float vh[3] = {h.y, h.z, h.w};
            const float kh = absorption32(p, a.kF, i, h.x);
            const float4 u0 = a.rad4[i], u1 = load_rad32(a, i);
            const float dG[3] = {u1.y - u0.y, u1.z - u0.z, u1.w - u0.w};
            float dS[5];
            gas_source32(p, kh, vh, u1.x - u0.x, dG, dS);
            const float D[5] = {0.0f, fh * dS[1], fh * dS[2], fh * dS[3], fh * dS[4]};
            const PrimInc o = prim_increment(p, d2f_trunc(rho), v32, d2f_trunc(T), D);
            double T1 = T + f2d_exact(o.dT);
            if (below_zero_bits(T1)) {
                T1 = 0.0;
                ++floors;
            }
            double v1[3];
            for (int d = 0; d < 3; ++d) v1[d] = v[d] + f2d_exact(o.dv[d]);
            if (!(finite_bits(v1[0]) && finite_bits(v1[1]) && finite_bits(v1[2]) && finite_bits(T1))) ++bad;
            a.T[i] = T1;
            store_velocity(a, i, to_f32(rho), v1);
        }
        if (floors) atomicAdd(&a.counters[0], floors);
        if (bad) atomicAdd(&a.counters[1], bad);
    } else {
        for (long long i = first_index(); i < nc; i += index_stride()) {
            const int one[3] = {1, 1, 1};
            const Prim<double> W = load_prim(p, a, i, one);
            double U[5];
            to_cons(p, W, U);
            // S_e,gas is linear in the radiation state: S(W^{n+1/2}, U_rad^{n+1}) - S(W^{n+1/2}, U_rad^n) is S of
            // the radiation's change
            const double kh = a.pend[0][i];
            const double vh[3] = {a.pend[1][i], a.pend[2][i], a.pend[3][i]};
            const double dG[3] = {a.G[0][i] - a.pend[5][i], a.G[1][i] - a.pend[6][i], a.G[2][i] - a.pend[7][i]};
            double dS[5];
            gas_source(p, kh, vh, a.E[i] - a.pend[4][i], dG, dS);
            for (int q = 1; q < 5; ++q) U[q] = U[q] + hdt * dS[q];
            Prim<double> W1;
            double inv_r;
            if (to_prim(p, U, W1, inv_r)) ++floors;
            if (!finite_prim(W1)) ++bad;
            for (int d = 0; d < 3; ++d) a.v[d][i] = W1.v[d];
            a.T[i] = W1.P * p.mu_over_kB * inv_r;
        }
        if (floors) atomicAdd(&a.counters[0], floors);
        if (bad) atomicAdd(&a.counters[1], bad);
    }
}

int blocks_for(long long n)
{
    const long long b = (n + GAS_THREADS - 1) / GAS_THREADS;
    return (int)(b < 1 ? 1 : (b > (1LL << 30) ? (1LL << 30) : b));
}

template <typename R, int DIM, int TX, int TY>
void launch_half(const GasParams& p, const GasArrays& a, bool predictor, int num_sms, cudaStream_t s)
{
    long long nb;
    const GasMarch t = gas_march(predictor ? p.m : p.n, TX, TY, num_sms, &nb);
    constexpr int NT = GasTile<DIM, TX, TY>::NT;
    if (predictor) gas_predictor_kernel<R, DIM, TX, TY><<<(unsigned)nb, NT, 0, s>>>(p, a, t);
    else if (DIM == 3 && p.limiter == 0)
        gas_corrector_kernel<R, DIM, TX, TY, DIM == 3 ? 0 : -1><<<(unsigned)nb, NT, 0, s>>>(p, a, t);
    else if (DIM == 3 && p.limiter == 1)
        gas_corrector_kernel<R, DIM, TX, TY, DIM == 3 ? 1 : -1><<<(unsigned)nb, NT, 0, s>>>(p, a, t);
    else gas_corrector_kernel<R, DIM, TX, TY, -1><<<(unsigned)nb, NT, 0, s>>>(p, a, t);
}

template <typename R>
void launch_half_1d(const GasParams& p, const GasArrays& a, bool predictor, int num_sms, cudaStream_t s)
{
    // three warps of cells and one for the last face: a warp on each of the multiprocessor's partitions, while
    // that gives every multiprocessor at most two CTAs; long lines take tiles with a smaller share of extra warps
    if (p.m[0] <= 2LL * 96 * num_sms) launch_half<R, 1, 96, 1>(p, a, predictor, num_sms, s);
    else launch_half<R, 1, 480, 1>(p, a, predictor, num_sms, s);
}

void launch_marched(const GasParams& p, const GasArrays& a, bool predictor, int num_sms, cudaStream_t s)
{
    if (!p.split) launch_half_1d<double>(p, a, predictor, num_sms, s);
    else if (p.n[2] > 1) launch_half<float, 3, 32, 8>(p, a, predictor, num_sms, s);
    else if (p.n[1] > 1) launch_half<float, 2, 32, 8>(p, a, predictor, num_sms, s);
    else launch_half_1d<float>(p, a, predictor, num_sms, s);
}

}  // namespace

bool gas_marched(const GasParams& p) { return p.split || p.n[1] <= 1; }

cudaError_t launch_gas_predictor(const GasParams& p, const GasArrays& a, int num_sms, cudaStream_t s)
{
    launch_marched(p, a, true, num_sms, s);
    return cudaGetLastError();
}

cudaError_t launch_gas_corrector(const GasParams& p, const GasArrays& a, int num_sms, cudaStream_t s)
{
    launch_marched(p, a, false, num_sms, s);
    return cudaGetLastError();
}

cudaError_t launch_gas_pred_flux(const GasParams& p, const GasArrays& a, int d, cudaStream_t s)
{
    int e[3];
    gas_pred_faces(p, d, e);
    const int nb = blocks_for(gas_count(e));
    if (d == 0) gas_pred_flux_kernel<0><<<nb, GAS_THREADS, 0, s>>>(p, a);
    else if (d == 1) gas_pred_flux_kernel<1><<<nb, GAS_THREADS, 0, s>>>(p, a);
    else gas_pred_flux_kernel<2><<<nb, GAS_THREADS, 0, s>>>(p, a);
    return cudaGetLastError();
}

cudaError_t launch_gas_pred_update(const GasParams& p, const GasArrays& a, cudaStream_t s)
{
    gas_pred_update_kernel<<<blocks_for(gas_count(p.m)), GAS_THREADS, 0, s>>>(p, a);
    return cudaGetLastError();
}

cudaError_t launch_gas_corr_flux(const GasParams& p, const GasArrays& a, int d, cudaStream_t s)
{
    int e[3];
    gas_corr_faces(p, d, e);
    const int nb = blocks_for(gas_count(e));
    if (d == 0) gas_corr_flux_kernel<0><<<nb, GAS_THREADS, 0, s>>>(p, a);
    else if (d == 1) gas_corr_flux_kernel<1><<<nb, GAS_THREADS, 0, s>>>(p, a);
    else gas_corr_flux_kernel<2><<<nb, GAS_THREADS, 0, s>>>(p, a);
    return cudaGetLastError();
}

cudaError_t launch_gas_corr_update(const GasParams& p, const GasArrays& a, cudaStream_t s)
{
    gas_corr_update_kernel<<<blocks_for(gas_count(p.n)), GAS_THREADS, 0, s>>>(p, a);
    return cudaGetLastError();
}

cudaError_t launch_gas_correct(const GasParams& p, const GasArrays& a, cudaStream_t s)
{
    if (p.split) gas_correct_kernel<true><<<blocks_for(gas_count(p.n)), GAS_THREADS, 0, s>>>(p, a);
    else gas_correct_kernel<false><<<blocks_for(gas_count(p.n)), GAS_THREADS, 0, s>>>(p, a);
    return cudaGetLastError();
}

}  // namespace rhd
