// subcycle_split2d.cuh -- the split-precision subcycle of 2D grids as two kernels (included by subcycle.cuh).
//
//   predictor: U^{m+1/2} of every cell of the grid with its ghost layers (two per face of a direction that is not
//     periodic on both faces), written as FP32 float4 (E, Gx, Gy, Gz), 16 bytes a cell;
//   corrector: face states, HLL, sources, exchange and realizability of the interior cells.
// The arithmetic is that of subcycle_tile<.., DIM = 2>, operation for operation, so both give the same bits; that
// kernel remains for grids whose device has no room for U^{m+1/2}.  It evaluates the closure on 2.1 and the predictor
// on 1.7 cells for each of its tile's, and its 94 registers and 90 KB of shared memory let two CTAs in: 3516
// instructions a cell issued in 44 % of the cycles, 142 us a subcycle at 1000 x 700 (FROZEN_T, MC, arrays).  The pair
// takes 27 + 41 us there (709 and 1381 instructions a cell, five and four CTAs, 57 and 67 % issue): bound by
// instruction issue, the predictor by the latency of its first loads as well.
#pragma once

#include <type_traits>

namespace rhd {

// HLL flux of hll() with the weights chosen instead of the code: the average is weights 1, 1, 0 and 1/2
__device__ __forceinline__ float4 hll2d(float4 UL, float4 UR, float4 FL, float4 FR, float l1L, float l3L, float l1R,
                                        float l3R)
{
    const float SRp = rmax0(l3L, l3R), SLm = rmin0(l1L, l1R);
    const float den = xadd(SRp, -SLm);
    const bool two = den > 0.0f;
    const float a = two ? SRp : 1.0f, b = two ? -SLm : 1.0f, c = two ? xmul(SRp, SLm) : 0.0f, iv = two ? rcp(den) : 0.5f;
    return make_float4(xmul(xfma(c, xadd(UR.x, -UL.x), xfma(a, FL.x, xmul(b, FR.x))), iv),
                       xmul(xfma(c, xadd(UR.y, -UL.y), xfma(a, FL.y, xmul(b, FR.y))), iv),
                       xmul(xfma(c, xadd(UR.z, -UL.z), xfma(a, FL.z, xmul(b, FR.z))), iv),
                       xmul(xfma(c, xadd(UR.w, -UL.w), xfma(a, FL.w, xmul(b, FR.w))), iv));
}

constexpr int S2_TX = 32, S2_TY = 8, S2_NT = S2_TX * S2_TY;

// Both kernels: a thread per cell of the tile, which computes its low faces; the first threads also take a cell of the
// halo and the faces of the tile's top row and right column.  COMMON: M1 closure and speeds, theta_F = 1 and no
// theta update of E (FULL, EQUILIBRIUM), known at compile time.
template <bool COMMON>
__global__ void __launch_bounds__(S2_NT, 4) predictor2d_kernel(const __grid_constant__ StepParams P)
{
    constexpr int TX = S2_TX, TY = S2_TY;
    using G = GeoPred<TX, TY>;
    __shared__ float4 Um[G::N1], CX[G::N1], CY[G::N1], Fx[G::NFX], Fy[G::NFY];
    __shared__ float2 L3[G::N1];
    const GridParams& g = P.g;
    const GridArrays& a = P.a;
    const int t = threadIdx.x, tlx = t % TX, tly = t / TX;
    const float chat = P.f_chat, hdt = 0.5f * P.f_dt, idx = g.f_inv_dx[0], idy = g.f_inv_dx[1];
    const int p1 = !COMMON && g.closure == 1, fixed = !COMMON && g.speeds == 1;
    const bool needT = !COMMON && g.exchange == EX_FROZEN_T;
    const int x0 = (int)(blockIdx.x % P.tiles_x) * TX - g.pad[0], y0 = (int)(blockIdx.x / P.tiles_x) * TY - g.pad[1];
    const int gx = x0 + tlx, gy = y0 + tly;
    const bool stored = gx < g.n[0] + g.pad[0] && gy < g.n[1] + g.pad[1];
    const bool interior = gx >= 0 && gx < g.n[0] && gy >= 0 && gy < g.n[1];

    auto fetch = [&](int x, int y) {
        double U[4];
        load_U(g, a, x, y, 0, U);
        return make_float4(d2f_trunc(U[0]), d2f_trunc(U[1]), d2f_trunc(U[2]), d2f_trunc(U[3]));
    };
    auto closure = [&](int i, const float4& U) {
        const ClosureScalars<float> k = closure_scalars(U.x, U.y, U.z, U.w, chat, p1);
        float l1x, l3x, l1y, l3y;
        wave_speeds(k, U.y, chat, fixed, l1x, l3x);
        wave_speeds(k, U.z, chat, fixed, l1y, l3y);
        const float bx = xmul(k.b, U.y), bz = xmul(k.b, U.z);
        const float Pxy = xmul(chat, xmul(bx, U.z)), Pxz = xmul(chat, xmul(bx, U.w)), Pyz = xmul(chat, xmul(bz, U.w));
        i = chk(i, G::N1);
        Um[i] = U;
        CX[i] = make_float4(xmul(chat, xfma(bx, U.y, k.a)), Pxy, Pxz, l1x);
        CY[i] = make_float4(Pxy, xmul(chat, xfma(bz, U.z, k.a)), Pyz, l1y);
        L3[i] = make_float2(l3x, l3y);
    };
    const int i_own = G::i1(tlx, tly);
    const bool has_h = t < G::NH;
    int hlx = 0, hly = 0;
    if (has_h) G::halo(t, hlx, hly);
    const float4 U = fetch(gx, gy);
    const float4 Uhalo = has_h ? fetch(x0 + hlx, y0 + hly) : U;
    GasCell<float> gc;
    if (stored) gc = load_gas<float, true>(g, a, gx, gy, 0, needT, false);
    closure(i_own, U);
    if (has_h) closure(G::i1(hlx, hly), Uhalo);
    __syncthreads();
    auto xface = [&](int iL, int iR) {
        iL = chk(iL, G::N1);
        iR = chk(iR, G::N1);
        const float4 UL = Um[iL], UR = Um[iR], CL = CX[iL], CR = CX[iR];
        return hll2d(UL, UR, make_float4(xmul(chat, UL.y), CL.x, CL.y, CL.z), make_float4(xmul(chat, UR.y), CR.x, CR.y, CR.z),
                     CL.w, L3[iL].x, CR.w, L3[iR].x);
    };
    auto yface = [&](int iL, int iR) {
        iL = chk(iL, G::N1);
        iR = chk(iR, G::N1);
        const float4 UL = Um[iL], UR = Um[iR], CL = CY[iL], CR = CY[iR];
        return hll2d(UL, UR, make_float4(xmul(chat, UL.z), CL.x, CL.y, CL.z), make_float4(xmul(chat, UR.z), CR.x, CR.y, CR.z),
                     CL.w, L3[iL].y, CR.w, L3[iR].y);
    };
    const int fl = tly * (TX + 1) + tlx, fb = tly * TX + tlx;
    Fx[chk(fl, G::NFX)] = xface(i_own - 1, i_own);
    Fy[chk(fb, G::NFY)] = yface(i_own - G::W1, i_own);
    if (t < TX) {
        const int iL = G::i1(t, TY - 1);
        Fy[chk(TY * TX + t, G::NFY)] = yface(iL, iL + G::W1);
    } else if (t < TX + TY) {
        const int ly = t - TX, iL = G::i1(TX - 1, ly);
        Fx[chk(ly * (TX + 1) + TX, G::NFX)] = xface(iL, iL + 1);
    }
    __syncthreads();
    unsigned fix = 0;
    if (stored) {
        const float4 ax = Fx[fl], bx = Fx[fl + 1], ay = Fy[fb], by = Fy[fb + TX];
        const float U0[4] = {U.x, U.y, U.z, U.w};
        const float xl[4] = {ax.x, ax.y, ax.z, ax.w}, xh[4] = {bx.x, bx.y, bx.z, bx.w};
        const float yl[4] = {ay.x, ay.y, ay.z, ay.w}, yh[4] = {by.x, by.y, by.z, by.w};
        float S[4], Un[4];
        explicit_sources(g, gc, U0, chat, S);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float div = (xh[q] - xl[q]) * idx;
            div = div + (yh[q] - yl[q]) * idy;
            Un[q] = U0[q] - hdt * div + hdt * S[q];
        }
        if constexpr (COMMON) {
            // theta_updates with theta_F = 1, to the bit
            const float fF = rcp(xadd(1.0f, xmul(xmul(chat, gc.kF), hdt)));
            Un[1] *= fF;
            Un[2] *= fF;
            Un[3] *= fF;
        } else {
            theta_updates(g, gc, chat, hdt, Un);
        }
        const int f = realize(Un, g.f_E_floor);
        if (interior) fix = f;
        P.uhalf[chk((gx + g.pad[0]) + (long long)upad_extent(g, 0) * (gy + g.pad[1]), n_padded(g))] = f4(Un);
    }
    add_counter(&P.stats->n_fix, fix);
}

// Closure of two states (lanes .x, .y) as closure_scalars and wave_speeds form it, in packed FP32 operations
template <int D>
__device__ __forceinline__ void closure2d_pair(float2 E, float2 gx, float2 gy, float2 gz, float2 g2, float chat, int p1,
                                               int fixed, float2& a, float2& b, float2& l1, float2& l3)
{
    float2 invE = p_rcp(E);
    float2 f2 = p_mul(g2, p_mul(invE, invE));
    float2 invEb = invE;
    if (f2.x > 1.0f || f2.y > 1.0f) {  // beyond the light cone: see closure_scalars
        if (f2.x > 1.0f) {
            const float q = rcp(sqrt_fast(f2.x));
            invE.x = xmul(invE.x, q);
            invEb.x = xmul(invE.x, q);
            f2.x = 1.0f;
        }
        if (f2.y > 1.0f) {
            const float q = rcp(sqrt_fast(f2.y));
            invE.y = xmul(invE.y, q);
            invEb.y = xmul(invE.y, q);
            f2.y = 1.0f;
        }
    }
    const float2 s = p_sqrt(p_fma(p_s(-3.0f), f2, p_s(4.0f)));
    const float2 inv2ps = p_rcp(p_add(p_s(2.0f), s));
    const float2 sm1 = p_add(s, p_s(-1.0f));
    if (p1) {
        a = p_mul(E, p_s(1.0f / 3.0f));
        b = p_s(0.0f);
    } else {
        a = p_mul(p_mul(sm1, E), p_s(1.0f / 3.0f));
        b = p_mul(p_mul(p_s(3.0f), inv2ps), invEb);
    }
    if (fixed) {
        l3 = p_s(xmul(chat, 0.57735026918962576451f));
        l1 = p_s(-l3.x);
        return;
    }
    const float2 cs = p_mul(p_s(chat), p_rcp(s));
    const float2 fd = p_mul(D == 0 ? gx : (D == 1 ? gy : gz), invE);
    const float2 w = p_mul(p_mul(p_s(-3.0f), fd), fd);
    float2 rad = p_mul(p_mul(p_s(2.0f / 3.0f), sm1), p_fma(w, inv2ps, s));
    rad.x = rmax0(rad.x, 0.0f);
    rad.y = rmax0(rad.y, 0.0f);
    const float2 sr = p_sqrt(rad);
    l1 = p_mul(p_sub(fd, sr), cs);
    l3 = p_mul(p_add(fd, sr), cs);
}

// Face states of a cell in direction D (face_states): rec = minus state, plus state, their closure coefficients and
// wave speeds; returns 1 if the slope was zeroed
template <int D>
__device__ __forceinline__ int face_record2d(float4 um, float4 u0, float4 up, float chat, int lim, int p1, int fixed,
                                             float4 rec[4])
{
    float4 sl;
    sl.x = limited_f(u0.x - um.x, up.x - u0.x, lim);
    sl.y = limited_f(u0.y - um.y, up.y - u0.y, lim);
    sl.z = limited_f(u0.z - um.z, up.z - u0.z, lim);
    sl.w = limited_f(u0.w - um.w, up.w - u0.w, lim);
    float4 Sm = make_float4(u0.x - 0.5f * sl.x, u0.y - 0.5f * sl.y, u0.z - 0.5f * sl.z, u0.w - 0.5f * sl.w);
    float4 Sp = make_float4(u0.x + 0.5f * sl.x, u0.y + 0.5f * sl.y, u0.z + 0.5f * sl.z, u0.w + 0.5f * sl.w);
    float2 E = make_float2(Sm.x, Sp.x), gx = make_float2(Sm.y, Sp.y), gy = make_float2(Sm.z, Sp.z), gz = make_float2(Sm.w, Sp.w);
    float2 g2 = p_fma(gz, gz, p_fma(gy, gy, p_mul(gx, gx)));
    const float2 most = p_mul(p_s(1.0f + Tol<float>::face), p_mul(E, E));
    const int fb = (int)(!(E.x > 0.0f)) | (int)(g2.x > most.x) | (int)(!(E.y > 0.0f)) | (int)(g2.y > most.y);
    if (fb) {
        Sm = Sp = u0;
        E = p_s(u0.x), gx = p_s(u0.y), gy = p_s(u0.z), gz = p_s(u0.w);
        g2 = p_fma(gz, gz, p_fma(gy, gy, p_mul(gx, gx)));
    }
    float2 a, b, l1, l3;
    closure2d_pair<D>(E, gx, gy, gz, g2, chat, p1, fixed, a, b, l1, l3);
    rec[0] = Sm;
    rec[1] = Sp;
    rec[2] = make_float4(a.x, b.x, a.y, b.y);
    rec[3] = make_float4(l1.x, l3.x, l1.y, l3.y);
    return fb;
}

// dir_flux from the stored closure coefficients
template <int D>
__device__ __forceinline__ float4 flux2d(float4 U, float a, float b, float chat)
{
    const float gd = D == 0 ? U.y : U.z, bg = xmul(b, gd);
    return make_float4(xmul(chat, gd), xmul(chat, xfma(bg, U.y, D == 0 ? a : 0.0f)),
                       xmul(chat, xfma(bg, U.z, D == 1 ? a : 0.0f)), xmul(chat, xfma(bg, U.w, 0.0f)));
}

// LIMK >= 0: the limiter, EXK >= 0: the exchange mode of a grid with the M1 closure and speeds and theta_F = theta_E =
// 1, at compile time; -1: any.  1000 x 700, FROZEN_T: 67 us with the constants of the stiff sources formed by every
// thread (FP64) at three CTAs, 63 at four, 41 with the constants formed once per CTA and the mode known.
template <int LIMK, int EXK>
__global__ void __launch_bounds__(S2_NT, 4) corrector2d_kernel(const __grid_constant__ StepParams P)
{
    constexpr int TX = S2_TX, TY = S2_TY;
    using G = GeoCorr<TX, TY>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // the fluxes take the place of U^{m+1/2}, which only the records need: with that, four CTAs fit
    float4* Uk = reinterpret_cast<float4*>(smem_raw);
    float4* Cx = Uk;
    float4* Cy = Cx + G::NCX;
    float4* Sx = Cy + G::NCY;
    float4* Sy = Sx + 4 * G::NSX;
    const GridParams& g = P.g;
    const GridArrays& a = P.a;
    constexpr bool COMMON = EXK >= 0;
    const int t = threadIdx.x, tlx = t % TX, tly = t / TX;
    double* own = reinterpret_cast<double*>(Sy + 4 * G::NSY) + t;  // own[q NT]: E, Gx, Gy, Gz, T of the own cell
    const float chat = P.f_chat, dt = P.f_dt, idx = g.f_inv_dx[0], idy = g.f_inv_dx[1];
    __shared__ SplitStiffConsts sk;  // formed by one thread: some thirty FP64 operations
    const int p1 = !COMMON && g.closure == 1, fixed = !COMMON && g.speeds == 1, lim = LIMK >= 0 ? LIMK : g.limiter;
    const int ex = COMMON ? EXK : g.exchange;
    const bool full = ex == EX_FULL, linear = ex == EX_LINEAR, needT = full || linear || ex == EX_FROZEN_T;
    const int x0 = (int)(blockIdx.x % P.tiles_x) * TX, y0 = (int)(blockIdx.x / P.tiles_x) * TY;
    const int gx = x0 + tlx, gy = y0 + tly;
    const bool cell = gx < g.n[0] && gy < g.n[1];
    const long long li = chk(cell ? gx + (long long)g.n[0] * gy : 0ll, n_cells(g));
    Counters cnt = {0, 0, 0, 0, 0, 0};
    // U^{m+1/2} of the tile and two cells around it, at the stored positions (beyond ragged edges: values unused)
#pragma unroll
    for (int r = 0; r < G::NR2; ++r) {
        const int c = t + r * G::NT;
        if (c < G::N2)
            cp_async16(Uk + c, P.uhalf + chk(upad_pos(g, 0, x0 + c % G::W2 - 2) +
                                                 (long long)upad_extent(g, 0) * upad_pos(g, 1, y0 + c / G::W2 - 2),
                                             n_padded(g)));
    }
    cp_async_commit();
    GasCell<float> gc{};
    if (cell) {
        cp_async8(own + 0 * G::NT, a.E + li);
        cp_async8(own + 1 * G::NT, a.G[0] + li);
        cp_async8(own + 2 * G::NT, a.G[1] + li);
        cp_async8(own + 3 * G::NT, a.G[2] + li);
        if (needT) cp_async8(own + 4 * G::NT, a.T + li);
        gc = gas_at(g, a, li);
    }
    cp_async_commit();
    if (t == 0) sk = split_stiff_consts(g, P.chat, P.dt);
    cp_async_wait_1();
    __syncthreads();
    const int i_own = G::i2(tlx, tly);
    const float4 uh = Uk[i_own];
    auto store_rec = [](float4* S, int n, int slot, const float4 (&rec)[4]) {
        slot = chk(slot, n);
#pragma unroll
        for (int v = 0; v < 4; ++v) S[v * n + slot] = rec[v];
    };
    // the face states of the cell at i along x or y
    const std::integral_constant<int, 0> along_x;
    const std::integral_constant<int, 1> along_y;
    auto record = [&](auto dir, int i, float4 (&rec)[4]) {
        constexpr int D = decltype(dir)::value;
        const int di = D == 0 ? 1 : G::W2;
        return face_record2d<D>(Uk[chk(i - di, G::N2)], Uk[chk(i, G::N2)], Uk[chk(i + di, G::N2)], chat, lim, p1, fixed, rec);
    };
    {
        float4 rec[4];
        int fb = record(along_x, i_own, rec);
        cnt.face += (unsigned)(fb & (int)cell);
        store_rec(Sx, G::NSX, G::sx(tlx, tly), rec);
        fb = record(along_y, i_own, rec);
        cnt.face += (unsigned)(fb & (int)cell);
        store_rec(Sy, G::NSY, G::sy(tlx, tly), rec);
        if (t < 2 * TX) {
            const int ly = t < TX ? -1 : TY, lx = t % TX, i = G::i2(lx, ly);
            record(along_y, i, rec);
            store_rec(Sy, G::NSY, G::sy(lx, ly), rec);
        } else if (t < G::NHR) {
            const int hh = t - 2 * TX, ly = hh >> 1, lx = (hh & 1) ? TX : -1, i = G::i2(lx, ly);
            record(along_x, i, rec);
            store_rec(Sx, G::NSX, G::sx(lx, ly), rec);
        }
    }
    __syncthreads();
    auto hll_x = [&](int iL, int iR) {
        iL = chk(iL, G::NSX);
        iR = chk(iR, G::NSX);
        const float4 UL = Sx[G::NSX + iL], UR = Sx[iR], cL = Sx[2 * G::NSX + iL], cR = Sx[2 * G::NSX + iR];
        const float4 LL = Sx[3 * G::NSX + iL], LR = Sx[3 * G::NSX + iR];
        return hll2d(UL, UR, flux2d<0>(UL, cL.z, cL.w, chat), flux2d<0>(UR, cR.x, cR.y, chat), LL.z, LL.w, LR.x, LR.y);
    };
    auto hll_y = [&](int iL, int iR) {
        iL = chk(iL, G::NSY);
        iR = chk(iR, G::NSY);
        const float4 UL = Sy[G::NSY + iL], UR = Sy[iR], cL = Sy[2 * G::NSY + iL], cR = Sy[2 * G::NSY + iR];
        const float4 LL = Sy[3 * G::NSY + iL], LR = Sy[3 * G::NSY + iR];
        return hll2d(UL, UR, flux2d<1>(UL, cL.z, cL.w, chat), flux2d<1>(UR, cR.x, cR.y, chat), LL.z, LL.w, LR.x, LR.y);
    };
    const int fl = tly * (TX + 1) + tlx, fb = tly * TX + tlx;
    Cx[chk(fl, G::NCX)] = hll_x(G::sx(tlx - 1, tly), G::sx(tlx, tly));
    Cy[chk(fb, G::NCY)] = hll_y(G::sy(tlx, tly - 1), G::sy(tlx, tly));
    if (t < TX) Cy[chk(TY * TX + t, G::NCY)] = hll_y(G::sy(t, TY - 1), G::sy(t, TY));
    else if (t < TX + TY) Cx[chk((t - TX) * (TX + 1) + TX, G::NCX)] = hll_x(G::sx(TX - 1, t - TX), G::sx(TX, t - TX));
    cp_async_wait_all();
    __syncthreads();
    if (cell) {
        const float4 ax = Cx[fl], bx = Cx[fl + 1], ay = Cy[fb], by = Cy[fb + TX];
        const float Uh[4] = {uh.x, uh.y, uh.z, uh.w};
        const float xl[4] = {ax.x, ax.y, ax.z, ax.w}, xh[4] = {bx.x, bx.y, bx.z, bx.w};
        const float yl[4] = {ay.x, ay.y, ay.z, ay.w}, yh[4] = {by.x, by.y, by.z, by.w};
        const double U0[4] = {own[0], own[G::NT], own[2 * G::NT], own[3 * G::NT]};
        double Tn = needT ? own[4 * G::NT] : 0.0, Un[4];
        gc.T = Tn;
        float S[4], d[4];
        explicit_sources(g, gc, Uh, chat, S);
        // FP32 increment relative to the FP64 state; the stiff sources in double-float
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float div = (xh[q] - xl[q]) * idx;
            div = div + (yh[q] - yl[q]) * idy;
            d[q] = -dt * div + dt * S[q];
        }
        split_stiff<EXK>(g, a, sk, chat, dt, gc, U0, d, Tn, Un, cnt);
        // realizability: cheap FP32 screen, exact FP64 test only near the limit
        const float ef = d2f_trunc(Un[0]);
        float g2f = 0.f;
#pragma unroll
        for (int q = 1; q < 4; ++q) {
            const float gq = d2f_trunc(Un[q]);
            g2f += gq * gq;
        }
        if (!(ef > g.f_E_floor * 1.001f) || g2f > 0.9999f * ef * ef) cnt.fix += realize(Un, g.E_floor);
        cnt.nonfinite += !(finite_d(Un[0]) && finite_d(Un[1]) && finite_d(Un[2]) && finite_d(Un[3]) &&
                           (!(full || linear) || finite_d(Tn)));
        a.Eo[li] = Un[0];
        a.Go[0][li] = Un[1];
        a.Go[1][li] = Un[2];
        a.Go[2][li] = Un[3];
        if (full || linear) a.T[li] = Tn;
    }
    add_counter(&P.stats->n_fix, cnt.fix);
    add_counter(&P.stats->n_face, cnt.face);
    add_counter(&P.stats->n_theta, cnt.theta);
    add_counter(&P.stats->n_newton_fb, cnt.newton_fb);
    add_counter(&P.stats->n_nonfinite, cnt.nonfinite);
    max_counter(&P.stats->newton_iter_max, cnt.iter_max);
}
constexpr size_t corrector2d_smem()
{
    using G = GeoCorr<S2_TX, S2_TY>;
    static_assert(G::N2 <= G::NCX + G::NCY, "U^{m+1/2} fits in the fluxes' place");
    return 16 * (size_t)(G::NCX + G::NCY + 4 * G::NSX + 4 * G::NSY) + 8 * (size_t)(5 * G::NT);
}

}  // namespace rhd
