// subcycle_fp64.cuh -- the FP64 radiation subcycle on one tile (included by subcycle.cuh): the stages and
// the layout of subcycle_tile, with arithmetic arranged for this part's FP64 pipe.
//
// What bounds it: the FP64 pipe issues one warp instruction per 64 cycles and SM sub-partition (two FP64
// operations per cycle and SM), while the other pipes take sixty-odd instructions in that time.  So only
// FP64 instructions count, and what can be said in integers or FP32 is said there:
//   - limiters, upwind maxima and minima, floors and branch tests compare the values' bits;
//   - the realizability tests (|G| <= E) are screened in FP32 and run in FP64 only near the limit;
//   - fluxes and wave speeds are kept per unit chat, and chat dt / dx is one factor per direction, applied
//     with the flux difference as one fused multiply-add on the state;
//   - the closure works on f = G/E (each component once), and the HLL flux on three weights.
// At 128^3 (the throughput state) the FP64 additions, multiplications and fused multiply-adds of the fused kernel
// fell from 1537 per cell-update (and some 250 comparisons) to 882; the pair of kernels takes 750.
#pragma once

namespace rhd {

// Closure of a state: f = G/E (scaled onto |f| = 1 outside the light cone, see closure_scalars),
// s = sqrt(4 - 3 f^2), is = 1/s, i3 = 3/(2 + s), k23 = 2 (s - 1)/3, P = a I + (iE f) f^T with
// iE = i3 E.  Explicitly rounded throughout: other tiles evaluate the same cells.
struct Closure64 {
    double f[3], s, is, i3, k23, a, iE;
};

__device__ __forceinline__ Closure64 closure64(const double U[4], int p1)
{
    Closure64 k;
    const double invE = rcp3(U[0]);
#pragma unroll
    for (int d = 0; d < 3; ++d) k.f[d] = xmul(U[1 + d], invE);
    double f2 = xfma(k.f[2], k.f[2], xfma(k.f[1], k.f[1], xmul(k.f[0], k.f[0])));
    // |G| > E (an input outside the realizable set) is closed as f = 1 along G/|G|; so is a state on the
    // light cone to the rounding of f^2 (a rescaled one, a beam), whose 1 - f^2 of a few 2^-53 would
    // otherwise enter the speeds across G as its square root
    if (reaches1_d(f2)) {
        const double q = rsqrt3(f2);
#pragma unroll
        for (int d = 0; d < 3; ++d) k.f[d] = xmul(k.f[d], q);
        f2 = 1.0;
    }
    const double x4 = xfma(-3.0, f2, 4.0);  // in [1, 4]
    k.is = rsqrt3(x4);
    k.s = xmul(x4, k.is);
    k.i3 = rcp3(xfma(k.s, 1.0 / 3.0, 2.0 / 3.0));
    k.k23 = xmul(xadd(k.s, -1.0), 2.0 / 3.0);
    if (p1) {
        k.a = xmul(U[0], 1.0 / 3.0);
        k.iE = 0.0;
    } else {
        k.a = xmul(xmul(k.k23, U[0]), 0.5);
        k.iE = xmul(k.i3, U[0]);
    }
    return k;
}

// lambda_1, lambda_3 per unit chat in the direction whose component of f is fd (Eq. hyperbolic:evals13,
// as in wave_speeds)
__device__ __forceinline__ void speeds64(const Closure64& k, double fd, int fixed, double& l1, double& l3)
{
    if (fixed) {
        l3 = 0.57735026918962576451;
        l1 = -l3;
        return;
    }
    const double rad = xmul(k.k23, xfma(-xmul(fd, fd), k.i3, k.s));
    const double sr = sqrt3(max0_d(rad, 0.0));
    const double m = xmul(fd, k.is);
    l1 = xfma(-sr, k.is, m);
    l3 = xfma(sr, k.is, m);
}

// flux per unit chat, (G_D, P_D.)
template <int D>
__device__ __forceinline__ void flux64(const Closure64& k, const double U[4], double F[4])
{
    const double t = xmul(k.iE, k.f[D]);
    F[0] = U[1 + D];
#pragma unroll
    for (int q = 0; q < 3; ++q) F[1 + q] = q == D ? xfma(t, k.f[q], k.a) : xmul(t, k.f[q]);
}

// HLL flux per unit chat (Eq. hyperbolic:hllflux2) from fluxes and speeds per unit chat:
// w_L F_L + w_R F_R + w_U (U_R - U_L), the weights S+/(S+ - S-), -S-/(S+ - S-) and S+ S-/(S+ - S-)
__device__ __forceinline__ void hll64(const double UL[4], const double UR[4], const double FL[4], const double FR[4],
                                      double l1L, double l3L, double l1R, double l3R, double out[4])
{
    const double SRp = max0_d(l3L, l3R), SLm = min0_d(l1L, l1R);
    const double den = xadd(SRp, -SLm);
    double wL = 0.5, wR = 0.5, wU = 0.0;
    if (mag_bits(den) != 0) {
        const double inv = rcp3(den);
        wL = xmul(SRp, inv);
        wR = xmul(-SLm, inv);
        wU = xmul(wL, SLm);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) out[q] = xfma(wU, xadd(UR[q], -UL[q]), xfma(wL, FL[q], xmul(wR, FR[q])));
}

// Half the limited slope from the left and right differences (the reading of `limited`)
__device__ __forceinline__ double half_slope64(double dl, double dr, int lim)
{
    if (lim == LIM_NONE) return 0.25 * (dl + dr);
    const double m = minmod_d(dl, dr);
    if (lim == LIM_MC) return minmod_d(m, 0.25 * (dl + dr));  // half of minmod(2 m, (dl + dr)/2)
    return 0.5 * m;
}

// One face state of a cell in direction D: state, flux and wave speeds per unit chat (10 values)
template <int D>
__device__ __forceinline__ void face_state64(const double S[4], int p1, int fixed, double out[10])
{
    const Closure64 k = closure64(S, p1);
#pragma unroll
    for (int q = 0; q < 4; ++q) out[q] = S[q];
    flux64<D>(k, S, out + 4);
    speeds64(k, k.f[D], fixed, out[8], out[9]);
}

// The two face values of a cell in direction D from U^{m+1/2} of cells i-1, i, i+1: minus state Sm, plus
// state Sp (both the cell's value if either is not realizable; returns 1 then)
__device__ __forceinline__ int face_values64(const double um[4], const double u0[4], const double up[4], int lim,
                                             double Sm[4], double Sp[4])
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const double h = half_slope64(xadd(u0[q], -um[q]), xadd(up[q], -u0[q]), lim);
        Sm[q] = xadd(u0[q], -h);
        Sp[q] = xadd(u0[q], h);
    }
    const int fb = face_unrealizable(Sm[0], Sm[1], Sm[2], Sm[3]) || face_unrealizable(Sp[0], Sp[1], Sp[2], Sp[3]);
    if (fb) {
#pragma unroll
        for (int q = 0; q < 4; ++q) Sm[q] = Sp[q] = u0[q];
    }
    return fb;
}

// HLL from stored face states: L = plus part of record iL, R = minus part of record iR
__device__ __forceinline__ void hll_stored64(const double* base, int stride, int iL, int iR, double F[4])
{
    double UL[4], UR[4], FL[4], FR[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        UL[q] = base[(10 + q) * stride + iL];
        FL[q] = base[(14 + q) * stride + iL];
        UR[q] = base[q * stride + iR];
        FR[q] = base[(4 + q) * stride + iR];
    }
    hll64(UL, UR, FL, FR, base[18 * stride + iL], base[19 * stride + iL], base[8 * stride + iR], base[9 * stride + iR],
          F);
}

// U += h S_e,rad(U0) (Eq. algorithm:source:explicit:rad with Eq. m1:simplifiedsource): h chat kF = xF,
// h chat / c = hj; then the theta absorption of F (Eq. source:stiff:radmomentum:soln) and of E (ABSORB,
// FROZEN_T) over h
__device__ __forceinline__ void sources64(const GridParams& g, const GasCell<double>& gc, const double U0[4],
                                          double chat_h, double hj, bool has_j, double U[4])
{
    const double xF = chat_h * gc.kF;
    if (has_j) U[0] = xfma(hj, gc.j, U[0]);
    if (g.beta_tau) {
        const double w = xF * g.inv_c;
        U[0] = xfma(w, xfma(gc.v[2], U0[3], xfma(gc.v[1], U0[2], xmul(gc.v[0], U0[1]))), U[0]);
        const double m = xmul(xmul(w, 4.0 / 3.0), U0[0]);
#pragma unroll
        for (int q = 0; q < 3; ++q) U[1 + q] = xfma(m, gc.v[q], U[1 + q]);
    }
    double fF;
    if (is_one_d(g.theta_F)) fF = rcp3(xadd(1.0, xF));
    else fF = xfma(-(1.0 - g.theta_F), xF, 1.0) * rcp3(xfma(g.theta_F, xF, 1.0));
#pragma unroll
    for (int q = 1; q < 4; ++q) U[q] = xmul(U[q], fF);
    if (g.exchange == EX_ABSORB) {
        const double xP = chat_h * gc.kP;
        U[0] *= (1.0 - (1.0 - g.theta_E) * xP) * rcp3(1.0 + g.theta_E * xP);
    } else if (g.exchange == EX_FROZEN_T) {
        const double xP = chat_h * gc.kP, T2 = gc.T * gc.T;
        U[0] = (U[0] * (1.0 - (1.0 - g.theta_E) * xP) + xP * (g.a_rad * T2 * T2)) * rcp3(1.0 + g.theta_E * xP);
    }
}

// The end of the corrector for one cell: U holds U^m plus its flux differences; the explicit sources from
// U^{m+1/2} (Uhk), the theta updates, the exchange and realizability follow, then the stores at li.
__device__ __forceinline__ void finish_cell64(const GridParams& g, const GridArrays& a, GasCell<double>& gc, double chat,
                                              double dt, const double Uhk[4], double U[4], double Tn, bool has_j,
                                              bool full, bool linear, long long li, Counters& cnt)
{
    gc.T = Tn;
    sources64(g, gc, Uhk, chat * dt, chat * dt * g.inv_c, has_j, U);
    if (full) {
        // transport can leave E <= 0 (not positivity preserving); exchange on E >= E_floor
        if (!(d2f_trunc(U[0]) > g.f_E_floor * 1.001f) && U[0] < g.E_floor) U[0] = g.E_floor;
        const ExchangeOut o = exchange64(g, chat, dt, gc.rho, gc.kP, U[0], Tn);
        cnt.theta += o.theta_fb;
        cnt.newton_fb += o.newton_fb;
        cnt.iter_max = max(cnt.iter_max, (unsigned)o.iters);
    } else if (linear) {
        exchange_linear_fp64(g, chat, dt, gc.kP, U[0], Tn);
    }
    cnt.fix += realize(U, g.E_floor);
    const bool bad = !(finite_d(U[0]) && finite_d(U[1]) && finite_d(U[2]) && finite_d(U[3]) &&
                       (!(full || linear) || finite_d(Tn)));
    cnt.nonfinite += bad;
    a.Eo[li] = U[0];
    a.Go[0][li] = U[1];
    a.Go[1][li] = U[2];
    a.Go[2][li] = U[3];
    if (full || linear) a.T[li] = Tn;
}

// ------------------------------------------------------------------------------------------------
// one tile of one subcycle: planes [z0, z1) of the column tile at (x0, y0)
// ------------------------------------------------------------------------------------------------
template <int TX, int TY, int DIM>
__device__ __forceinline__ void subcycle_tile64(const GridParams& g, const GridArrays& a, double chat, double dt, int x0,
                                                int y0, int z0, int z1, double* sm, Counters& cnt)
{
    using G = Geo<TX, TY, DIM>;
    const int t = threadIdx.x;
    double* Um = sm + G::P_UM;
    double* Cc = sm + G::P_CC;
    double* Fx = sm + G::P_FX;
    double* Fy = sm + G::P_FY;
    double* Sx = sm + G::C_SX;
    double* Sy = sm + G::C_SY;
    double* Cx = sm + G::C_FX;
    double* Cy = sm + G::C_FY;
    double* Uh = sm + G::OFF_UH;
    double* stU = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(sm) + G::r_bytes(sizeof(double)));
    double* stC = stU + G::ST_C;
    const double hdt = 0.5 * dt;
    // chat dt / dx per direction (halved in the predictor)
    const double cx = chat * dt * g.inv_dx[0], cy = chat * dt * g.inv_dx[1], cz = chat * dt * g.inv_dx[2];
    const double hx = 0.5 * cx, hy = 0.5 * cy, hz = 0.5 * cz;
    const int p1 = g.closure == 1, fixed = g.speeds == 1, lim = g.limiter;
    const bool needT_pred = g.exchange == EX_FROZEN_T, has_j = a.j != nullptr;
    const long long nxy = (long long)g.n[0] * g.n[1];

    // cells of the R3 region handled by this thread, fixed for all planes
    int c_i3[G::NR3], c_off[G::NR3];
    // the tile's halo lies inside the domain in x and y: loads need no boundary remap there
    const bool xy_inside = x0 - 3 >= 0 && x0 + TX + 3 <= g.n[0] && y0 - 3 >= 0 && y0 + TY + 3 <= g.n[1];
#pragma unroll
    for (int r = 0; r < G::NR3; ++r) {
        int c = t + r * G::NT;
        int lx = 0, ly = 0;
        if (c < G::N3) G::cell_of(c, lx, ly);
        c_i3[r] = G::i3(lx, ly);
        c_off[r] = (x0 + lx) + g.n[0] * (y0 + ly);
    }

    const int tlx = t % TX, tly = t / TX;
    // fetch U^m of plane q on R3 into the staging buffer (asynchronously where no remap is needed)
    auto issue_plane = [&](int q) {
        const bool fast = xy_inside && (unsigned)q < (unsigned)g.n[2];
        const long long zoff = (long long)q * nxy;
#pragma unroll
        for (int r = 0; r < G::NR3; ++r) {
            int c = t + r * G::NT;
            if (c < G::N3) {
                if (fast) {
                    long long i = chk(zoff + c_off[r], n_cells(g));
                    cp_async8(stU + 0 * G::N3 + c, a.E + i);
                    cp_async8(stU + 1 * G::N3 + c, a.G[0] + i);
                    cp_async8(stU + 2 * G::N3 + c, a.G[1] + i);
                    cp_async8(stU + 3 * G::N3 + c, a.G[2] + i);
                } else {
                    int lx, ly;
                    G::cell_of(c, lx, ly);
                    double U[4];
                    load_U(g, a, x0 + lx, y0 + ly, q, U);
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq) stU[qq * G::N3 + c] = U[qq];
                }
            }
        }
    };
    // fetch the state (and T) of the own tile cell of corrector plane k
    const bool needT_corr = g.exchange == EX_FULL || g.exchange == EX_FROZEN_T || g.exchange == EX_LINEAR;
    auto issue_corr = [&](int k) {
        if (x0 + tlx < g.n[0] && y0 + tly < g.n[1] && (unsigned)k < (unsigned)g.n[2]) {
            long long i = lin(g, x0 + tlx, y0 + tly, k);
            cp_async8(stC + 0 * G::NT + t, a.E + i);
            cp_async8(stC + 1 * G::NT + t, a.G[0] + i);
            cp_async8(stC + 2 * G::NT + t, a.G[1] + i);
            cp_async8(stC + 3 * G::NT + t, a.G[2] + i);
            if (needT_corr) cp_async8(stC + 4 * G::NT + t, a.T + i);
        }
    };

    // per-thread z pipeline of the predictor (own R2 cells: c = t + r * NT): the state, its z-direction
    // pressures and speeds, the state after the x and y flux differences, and the lower z flux
    double zU[G::NR2][4], zP[G::NR2][3], zl[G::NR2][2], acc[G::NR2][4], zfl[G::NR2][4];
    // corrector: lower z face and the plus face state (z) of the previous plane, own tile column
    double cfl[4], zplus[10];

    const int qbeg = (DIM == 3) ? z0 - 3 : 0;
    const int qend = (DIM == 3) ? z1 + 3 : 1;
    issue_plane(qbeg);
    cp_async_commit();
#pragma unroll 1
    for (int qz = qbeg; qz < qend; ++qz) {
        // (a) U^m of plane qz on the tile plus 3-cell halo (each thread moves the cells it fetched
        //     itself, so its own wait suffices)
        cp_async_wait_all();
#pragma unroll
        for (int r = 0; r < G::NR3; ++r) {
            int c = t + r * G::NT;
            if (c < G::N3) {
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) Um[qq * G::N3 + c_i3[r]] = stU[qq * G::N3 + c];
            }
        }
        __syncthreads();
        // prefetch the next plane and the state of this iteration's corrector plane
        if (qz + 1 < qend) issue_plane(qz + 1);
        if (DIM == 3) issue_corr(qz - 3); else issue_corr(qz);
        cp_async_commit();
        // (b) closure once per cell: P and the x, y wave speeds to shared memory; z data of the
        //     own R2 cells to registers
        double nU[G::NR2][4], nP[G::NR2][3], nl[G::NR2][2];
#pragma unroll
        for (int r = 0; r < G::NR3; ++r) {
            int c = t + r * G::NT;
            if (c < G::N3) {
                const int i = c_i3[r];
                const double U[4] = {Um[i], Um[G::N3 + i], Um[2 * G::N3 + i], Um[3 * G::N3 + i]};
                const Closure64 k = closure64(U, p1);
                const double tx = xmul(k.iE, k.f[0]), ty = xmul(k.iE, k.f[1]);
                const double Pxz = xmul(tx, k.f[2]), Pyz = xmul(ty, k.f[2]);
                double l1, l3;
                speeds64(k, k.f[0], fixed, l1, l3);
                Cc[0 * G::N3 + i] = xfma(tx, k.f[0], k.a);
                Cc[1 * G::N3 + i] = xmul(tx, k.f[1]);
                Cc[2 * G::N3 + i] = Pxz;
                Cc[5 * G::N3 + i] = l1;
                Cc[6 * G::N3 + i] = l3;
                {
                    speeds64(k, k.f[1], fixed, l1, l3);
                    Cc[3 * G::N3 + i] = xfma(ty, k.f[1], k.a);
                    Cc[4 * G::N3 + i] = Pyz;
                    Cc[7 * G::N3 + i] = l1;
                    Cc[8 * G::N3 + i] = l3;
                }
                if (r < G::NR2 && c < G::N2) {
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq) nU[r][qq] = U[qq];
                    if (DIM == 3) {
                        nP[r][0] = Pxz;
                        nP[r][1] = Pyz;
                        nP[r][2] = xfma(xmul(k.iE, k.f[2]), k.f[2], k.a);
                        speeds64(k, k.f[2], fixed, nl[r][0], nl[r][1]);
                    }
                }
            }
        }
        __syncthreads();
        // (c) first-order HLL fluxes (per unit chat) on the x and y faces of the R2 rows / columns
        for (int f = t; f < G::NFX + G::NFY; f += G::NT) {
            const bool isx = f < G::NFX;
            const int fy = f - G::NFX;
            const int lx = isx ? f % (G::W2 + 1) - 2 : fy % G::W2 - 2;
            const int ly = isx ? f / (G::W2 + 1) - 2 : fy / G::W2 - 2;
            const int iR = G::i3(lx, ly), iL = iR - (isx ? 1 : G::W3);
            // rows of Cc: P_x. = 0, 1, 2; P_y. = 1, 3, 4; speeds 5, 6 and 7, 8
            const int r0 = isx ? 0 : 1, r1 = isx ? 1 : 3, r2 = isx ? 2 : 4, rl = isx ? 5 : 7, rg = isx ? 1 : 2;
            double UL[4], UR[4], F[4];
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) {
                UL[qq] = Um[qq * G::N3 + iL];
                UR[qq] = Um[qq * G::N3 + iR];
            }
            const double FL[4] = {Um[rg * G::N3 + iL], Cc[r0 * G::N3 + iL], Cc[r1 * G::N3 + iL], Cc[r2 * G::N3 + iL]};
            const double FR[4] = {Um[rg * G::N3 + iR], Cc[r0 * G::N3 + iR], Cc[r1 * G::N3 + iR], Cc[r2 * G::N3 + iR]};
            hll64(UL, UR, FL, FR, Cc[rl * G::N3 + iL], Cc[(rl + 1) * G::N3 + iL], Cc[rl * G::N3 + iR],
                  Cc[(rl + 1) * G::N3 + iR], F);
            double* dst = isx ? Fx + f : Fy + fy;
            const int st = isx ? G::NFX : G::NFY;
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) dst[qq * st] = F[qq];
        }
        __syncthreads();
        // (d) x/y flux differences of plane qz; z face (qz-1 | qz); U^{m+1/2} of plane p = qz - 1 (3D) or qz
        const int p = (DIM == 3) ? qz - 1 : qz;
        const bool do_pred = (DIM == 3) ? (qz >= z0 - 1) : true;
#pragma unroll
        for (int r = 0; r < G::NR2; ++r) {
            int c = t + r * G::NT;
            if (c < G::N2) {
                int lx = c % G::W2 - 2, ly = c / G::W2 - 2;
                double nd[4];
                const int fl = (ly + 2) * (G::W2 + 1) + (lx + 2);
#pragma unroll
                for (int qq = 0; qq < 4; ++qq)
                    nd[qq] = xfma(-hx, xadd(Fx[qq * G::NFX + fl + 1], -Fx[qq * G::NFX + fl]), nU[r][qq]);
                {
                    const int fb = (ly + 2) * G::W2 + (lx + 2);
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq)
                        nd[qq] = xfma(-hy, xadd(Fy[qq * G::NFY + fb + G::W2], -Fy[qq * G::NFY + fb]), nd[qq]);
                }
                double zfh[4] = {0.0, 0.0, 0.0, 0.0};
                if (DIM == 3 && qz > qbeg) {
                    const double FL[4] = {zU[r][3], zP[r][0], zP[r][1], zP[r][2]};
                    const double FR[4] = {nU[r][3], nP[r][0], nP[r][1], nP[r][2]};
                    hll64(zU[r], nU[r], FL, FR, zl[r][0], zl[r][1], nl[r][0], nl[r][1], zfh);
                }
                if (do_pred && (DIM != 3 || qz > qbeg + 1)) {
                    double U0[4], U[4];
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq) {
                        U0[qq] = DIM == 3 ? zU[r][qq] : nU[r][qq];
                        U[qq] = DIM == 3 ? xfma(-hz, xadd(zfh[qq], -zfl[r][qq]), acc[r][qq]) : nd[qq];
                    }
                    const GasCell<double> gc = load_gas<double, false>(g, a, x0 + lx, y0 + ly, p, needT_pred, false);
                    sources64(g, gc, U0, chat * hdt, chat * hdt * g.inv_c, has_j, U);
                    const int fx_ = realize(U, g.E_floor);
                    const bool owned = lx >= 0 && lx < TX && ly >= 0 && ly < TY && x0 + lx < g.n[0] &&
                                       y0 + ly < g.n[1] && p >= z0 && p < z1;
                    if (owned) cnt.fix += fx_;
                    const int slot = (DIM == 3) ? ((p + 3) % 3) : 0;
                    double* dst = Uh + slot * 4 * G::N2;
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq) dst[qq * G::N2 + c] = U[qq];
                }
                if (DIM == 3) {
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq) {
                        zfl[r][qq] = zfh[qq];
                        zU[r][qq] = nU[r][qq];
                        acc[r][qq] = nd[qq];
                    }
#pragma unroll
                    for (int qq = 0; qq < 3; ++qq) zP[r][qq] = nP[r][qq];
                    zl[r][0] = nl[r][0];
                    zl[r][1] = nl[r][1];
                }
            }
        }
        __syncthreads();
        // (e) corrector for plane k
        const int k = (DIM == 3) ? qz - 3 : qz;
        const bool own_col = x0 + tlx < g.n[0] && y0 + tly < g.n[1];
        // the own column's U^{m+1/2} of three consecutive planes starting at zb
        auto column = [&](int zb, double u[3][4]) {
            const int i = G::i2(tlx, tly);
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const double* sl = Uh + ((zb + m + 3) % 3) * 4 * G::N2;
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) u[m][qq] = sl[qq * G::N2 + i];
            }
        };
        double dz[4] = {0.0, 0.0, 0.0, 0.0};  // z flux difference of the own cell of plane k
        if (DIM == 3 && qz >= z0 + 1) {
            // face states (z) of cell k + 1 and the face (k | k + 1) below it; the cell under the chunk
            // (qz = z0 + 1) has only its plus state to give
            double u[3][4], Sm[4], Sp[4], fm[10], cfh[4];
            column(qz - 3, u);
            const int fb = face_values64(u[0], u[1], u[2], lim, Sm, Sp);
            if (fb && own_col && k + 1 >= z0 && k + 1 < z1) cnt.face += 1;
            if (qz >= z0 + 2) {
                face_state64<2>(Sm, p1, fixed, fm);
                hll64(zplus, fm, zplus + 4, fm + 4, zplus[8], zplus[9], fm[8], fm[9], cfh);
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) {
                    dz[qq] = xadd(cfh[qq], -cfl[qq]);  // meaningful from qz = z0 + 3 on
                    cfl[qq] = cfh[qq];
                }
            }
            face_state64<2>(Sp, p1, fixed, zplus);
        }
        const bool do_corr = (DIM == 3) ? (k >= z0 && k < z1) : true;
        if (do_corr) {
            const double* Uk = Uh + ((DIM == 3) ? ((k + 3) % 3) : 0) * 4 * G::N2;
            // (e1) face states of the tile cells and their neighbours along x and y
            for (int c = t; c < G::NSX + G::NSY; c += G::NT) {
                const bool isx = c < G::NSX;
                const int cy = c - G::NSX;
                const int lx = isx ? c % (TX + 2) - 1 : cy % TX, ly = isx ? c / (TX + 2) : cy / TX - 1;
                const int i0 = G::i2(lx, ly), di = isx ? 1 : G::W2;
                double u[3][4], Sm[4], Sp[4];
#pragma unroll
                for (int m = 0; m < 3; ++m)
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq) u[m][qq] = Uk[qq * G::N2 + i0 + (m - 1) * di];
                const int fb = face_values64(u[0], u[1], u[2], lim, Sm, Sp);
                if (fb && lx >= 0 && lx < TX && ly >= 0 && ly < TY && x0 + lx < g.n[0] && y0 + ly < g.n[1]) cnt.face += 1;
                double* dst = isx ? Sx + c : Sy + cy;
                const int st = isx ? G::NSX : G::NSY;
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    double W[4], fs[10];
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq) W[qq] = side ? Sp[qq] : Sm[qq];
                    const Closure64 kk = closure64(W, p1);
                    const double fd = isx ? kk.f[0] : kk.f[1], tt = xmul(kk.iE, fd);
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq) fs[qq] = W[qq];
                    fs[4] = isx ? W[1] : W[2];
                    fs[5] = xfma(tt, kk.f[0], isx ? kk.a : 0.0);
                    fs[6] = xfma(tt, kk.f[1], isx ? 0.0 : kk.a);
                    fs[7] = xmul(tt, kk.f[2]);
                    speeds64(kk, fd, fixed, fs[8], fs[9]);
#pragma unroll
                    for (int qq = 0; qq < 10; ++qq) dst[(10 * side + qq) * st] = fs[qq];
                }
            }
            __syncthreads();
            // (e2) HLL fluxes on the tile's x and y faces
            for (int f = t; f < G::NCX + G::NCY; f += G::NT) {
                const bool isx = f < G::NCX;
                const int fc = f - G::NCX;
                // the record of the cell on the low side
                const int iL = isx ? f % (TX + 1) + (TX + 2) * (f / (TX + 1)) : fc;
                double F[4];
                if (isx) hll_stored64(Sx, G::NSX, iL, iL + 1, F);
                else hll_stored64(Sy, G::NSY, iL, iL + TX, F);
                double* dst = isx ? Cx + f : Cy + fc;
                const int st = isx ? G::NCX : G::NCY;
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) dst[qq * st] = F[qq];
            }
            __syncthreads();
            // (e3) update of the own tile cell
            if (own_col) {
                const int gx = x0 + tlx, gy = y0 + tly;
                const bool full = g.exchange == EX_FULL, linear = g.exchange == EX_LINEAR;
                GasCell<double> gc = load_gas<double, false>(g, a, gx, gy, k, false, true);
                const long long li = lin(g, gx, gy, k);
                const int ih = G::i2(tlx, tly), fl = tly * (TX + 1) + tlx, fb = tly * TX + tlx;
                cp_async_wait_all();  // own staged copies of U^m and T for this cell
                double Uhk[4], U[4];
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) {
                    Uhk[qq] = Uk[qq * G::N2 + ih];
                    U[qq] = xfma(-cx, xadd(Cx[qq * G::NCX + fl + 1], -Cx[qq * G::NCX + fl]), stC[qq * G::NT + t]);
                    U[qq] = xfma(-cy, xadd(Cy[qq * G::NCY + fb + TX], -Cy[qq * G::NCY + fb]), U[qq]);
                    if (DIM == 3) U[qq] = xfma(-cz, dz[qq], U[qq]);
                }
                double Tn = needT_corr ? stC[4 * G::NT + t] : 0.0;
                finish_cell64(g, a, gc, chat, dt, Uhk, U, Tn, has_j, full, linear, li, cnt);
            }
        }
        __syncthreads();
    }
    cp_async_wait_all();  // no copy may outlive the tile
}

}  // namespace rhd
