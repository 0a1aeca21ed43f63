// subcycle_fp64_pair.cuh -- the FP64 subcycle of 2D and 3D grids and ensembles as two kernels (included by
// subcycle.cuh after subcycle_fp64.cuh): a predictor that writes U^{m+1/2} of the grid with its ghost
// layers, and a corrector that reads it back, as in the split path's pair.
//
// Why two kernels: the FP64 pipe is the bound (subcycle_fp64.cuh), and the fused kernel spends it on the
// predictor of a 2-cell halo and on the closure of a 3-cell one (1.6 and 1.9 times a 16 x 16 tile, and six
// extra planes per z chunk); memory traffic, which the pair adds (32 B a cell written and read), is idle.
// Layout: 256 threads, one per cell of a w x h tile (w h <= 256); a tile's halo adds only what its faces
// need: in the predictor the closure of 2 (w + h) cells for one direction each, in the corrector one face
// state (of two) of 2 (w + h) cells, in both w + h faces, all in whole warps.  w and h are run-time values
// chosen for the grid (pair64_plan): index arithmetic is on the idle integer pipes, so a tile shape that
// fits the grid costs nothing.  Two CTAs per SM (128 registers; a few spills, also free) fill each other's
// barrier and load gaps.
#pragma once

namespace rhd {

constexpr int P64_NT = 256;
// shared-memory capacities over the tile shapes 8 <= w, h <= 32, w h <= 256
constexpr int P64_N1 = 340;   // (w + 2)(h + 2)
constexpr int P64_N2 = 432;   // (w + 4)(h + 4)
constexpr int P64_NF = 288;   // (w + 1) h, w (h + 1)
constexpr int P64_NE = 40;    // w + h
// doubles: two planes of U^m, closure data (9), x and y fluxes
constexpr int P64_PRED_DOUBLES = 8 * P64_N1 + 9 * P64_N1 + 8 * P64_NF;
// doubles: two planes of U^{m+1/2}, x and y plus-side records (9), minus records beyond the high edges,
// x and y fluxes, the own cell's state and T
constexpr int P64_CORR_DOUBLES = 8 * P64_N2 + 18 * P64_NF + 9 * P64_NE + 8 * P64_NF + 5 * P64_NT;
constexpr size_t pair64_pred_smem() { return sizeof(double) * (size_t)P64_PRED_DOUBLES; }
constexpr size_t pair64_corr_smem() { return sizeof(double) * (size_t)P64_CORR_DOUBLES; }

// The fluxes (rows 1 .. 3; row 0 is S[1 + dir]) and wave speeds of a face state in direction dir, per unit chat
struct Rec64 {
    double S[4], P[3], l1, l3;
};
__device__ __forceinline__ Rec64 face_rec64(const double S[4], int dir, int p1, int fixed)
{
    Rec64 r;
    const Closure64 k = closure64(S, p1);
    const double fd = dir == 0 ? k.f[0] : (dir == 1 ? k.f[1] : k.f[2]), t = xmul(k.iE, fd);
#pragma unroll
    for (int q = 0; q < 4; ++q) r.S[q] = S[q];
#pragma unroll
    for (int q = 0; q < 3; ++q) r.P[q] = xfma(t, k.f[q], q == dir ? k.a : 0.0);
    speeds64(k, fd, fixed, r.l1, r.l3);
    return r;
}
__device__ __forceinline__ void hll_rec64(const Rec64& L, const Rec64& R, int dir, double F[4])
{
    const double gL = dir == 0 ? L.S[1] : (dir == 1 ? L.S[2] : L.S[3]);
    const double gR = dir == 0 ? R.S[1] : (dir == 1 ? R.S[2] : R.S[3]);
    const double FL[4] = {gL, L.P[0], L.P[1], L.P[2]}, FR[4] = {gR, R.P[0], R.P[1], R.P[2]};
    hll64(L.S, R.S, FL, FR, L.l1, L.l3, R.l1, R.l3, F);
}
__device__ __forceinline__ void put_rec64(double* base, int stride, int i, const Rec64& r)
{
#pragma unroll
    for (int q = 0; q < 4; ++q) base[q * stride + i] = r.S[q];
#pragma unroll
    for (int q = 0; q < 3; ++q) base[(4 + q) * stride + i] = r.P[q];
    base[7 * stride + i] = r.l1;
    base[8 * stride + i] = r.l3;
}
__device__ __forceinline__ Rec64 get_rec64(const double* base, int stride, int i)
{
    Rec64 r;
#pragma unroll
    for (int q = 0; q < 4; ++q) r.S[q] = base[q * stride + i];
#pragma unroll
    for (int q = 0; q < 3; ++q) r.P[q] = base[(4 + q) * stride + i];
    r.l1 = base[7 * stride + i];
    r.l3 = base[8 * stride + i];
    return r;
}

// Predictor over the w x h tile at (x0, y0) of the stored U^{m+1/2} (coordinates in [-pad, n + pad)), planes
// [z0, z1) (3D; 2D: the one plane).  uh: 4 doubles (E, Gx, Gy, Gz) per stored cell.
template <int DIM>
__device__ __forceinline__ void predictor_tile64(const GridParams& g, const GridArrays& a, double* uh, double chat,
                                                 double dt, int x0, int y0, int w, int h, int z0, int z1, double* sm,
                                                 Counters& cnt)
{
    const int t = threadIdx.x;
    double* Um0 = sm;                      // Um0[(4 buf + q) N1 + i]
    double* Cc = Um0 + 8 * P64_N1;         // P_xx, P_xy, P_xz, P_yy, P_yz, l1x, l3x, l1y, l3y
    double* Fx = Cc + 9 * P64_N1;
    double* Fy = Fx + 4 * P64_NF;
    const double hdt = 0.5 * dt;
    const double hx = chat * hdt * g.inv_dx[0], hy = chat * hdt * g.inv_dx[1], hz = chat * hdt * g.inv_dx[2];
    const int p1 = g.closure == 1, fixed = g.speeds == 1;
    const bool needT = g.exchange == EX_FROZEN_T, has_j = a.j != nullptr;
    const int w1 = w + 2, n1 = w1 * (h + 2);
    const int ex = g.n[0] + g.pad[0], ey = g.n[1] + g.pad[1];  // the stored range ends here
    const long long nxy = (long long)g.n[0] * g.n[1];
    const int lx = t % w, ly = t / w, gx = x0 + lx, gy = y0 + ly;
    // cells whose closure is needed: the stored ones and the next beyond them
    const bool own = t < w * h && gx <= ex && gy <= ey;
    const bool emit_cell = t < w * h && gx < ex && gy < ey;
    const bool own_interior = gx >= 0 && gx < g.n[0] && gy >= 0 && gy < g.n[1];
    const int i_own = (lx + 1) + w1 * (ly + 1);
    // halo cells: rows -1 and h (their y data), columns -1 and w (their x data)
    const bool has_h = t < 2 * (w + h), h_isx = t >= 2 * w;
    const int e = t - 2 * w;
    const int hlx = h_isx ? (e < h ? -1 : w) : (t < w ? t : t - w), hly = h_isx ? (e < h ? e : e - h) : (t < w ? -1 : h);
    const int i_h = has_h ? (hlx + 1) + w1 * (hly + 1) : 0;
    const bool h_need = has_h && x0 + hlx <= ex && y0 + hly <= ey;
    // faces beyond the high edges: the h right x faces, then the w top y faces
    const bool has_e = t < w + h, e_isx = t < h;
    const int elx = e_isx ? w : t - h, ely = e_isx ? t : h;
    const bool xy_inside = x0 - 1 >= 0 && x0 + w + 1 <= g.n[0] && y0 - 1 >= 0 && y0 + h + 1 <= g.n[1];
    // the cells of the tile + 1 region that this thread stages
    int c_x[2], c_y[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int c = t + r * P64_NT;
        c_x[r] = x0 + c % w1 - 1;
        c_y[r] = y0 + c / w1 - 1;
    }
    auto issue_plane = [&](int q, int buf) {
        const bool fast = xy_inside && (unsigned)q < (unsigned)g.n[2];
        double* Ub = Um0 + 4 * P64_N1 * buf;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int c = t + r * P64_NT;
            if (c < n1) {
                const int cc = chk(c, P64_N1);
                if (fast) {
                    const long long i = chk((long long)q * nxy + c_x[r] + (long long)g.n[0] * c_y[r], n_cells(g));
                    cp_async8(Ub + cc, a.E + i);
                    cp_async8(Ub + P64_N1 + cc, a.G[0] + i);
                    cp_async8(Ub + 2 * P64_N1 + cc, a.G[1] + i);
                    cp_async8(Ub + 3 * P64_N1 + cc, a.G[2] + i);
                } else if (c_x[r] <= ex && c_y[r] <= ey) {
                    double U[4];
                    load_U(g, a, c_x[r], c_y[r], q, U);
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq) Ub[qq * P64_N1 + cc] = U[qq];
                }
            }
        }
    };
    double zU[4], zP[3], zl1 = 0.0, zl3 = 0.0, acc[4], zfl[4] = {0.0, 0.0, 0.0, 0.0};
    const int qbeg = DIM == 3 ? z0 - 1 : 0, qend = DIM == 3 ? z1 + 1 : 1;
    issue_plane(qbeg, 0);
    cp_async_commit();
#pragma unroll 1
    for (int q = qbeg; q < qend; ++q) {
        const int buf = (q - qbeg) & 1;
        const double* Um = Um0 + 4 * P64_N1 * buf;
        cp_async_wait_all();
        __syncthreads();
        if (q + 1 < qend) issue_plane(q + 1, buf ^ 1);
        cp_async_commit();
        // planes q = qbeg and qend - 1 only lend their z data
        const bool flat = DIM == 3 && (q == qbeg || q == qend - 1);
        const int p = DIM == 3 ? q - 1 : q;
        const bool emit = emit_cell && (DIM != 3 || q > qbeg + 1);
        GasCell<double> gc;
        if (emit) gc = load_gas<double, false>(g, a, gx, gy, p, needT, false);
        // closure of the own cell, and of one halo cell in its direction
        double nU[4], nP[3], nl1 = 0.0, nl3 = 0.0;
        if (own) {
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) nU[qq] = Um[qq * P64_N1 + i_own];
            const Closure64 k = closure64(nU, p1);
            const double tx = xmul(k.iE, k.f[0]), ty = xmul(k.iE, k.f[1]);
            nP[0] = xmul(tx, k.f[2]);
            nP[1] = xmul(ty, k.f[2]);
            if (!flat) {
                double l1, l3;
                Cc[i_own] = xfma(tx, k.f[0], k.a);
                Cc[P64_N1 + i_own] = xmul(tx, k.f[1]);
                Cc[2 * P64_N1 + i_own] = nP[0];
                Cc[3 * P64_N1 + i_own] = xfma(ty, k.f[1], k.a);
                Cc[4 * P64_N1 + i_own] = nP[1];
                speeds64(k, k.f[0], fixed, l1, l3);
                Cc[5 * P64_N1 + i_own] = l1;
                Cc[6 * P64_N1 + i_own] = l3;
                speeds64(k, k.f[1], fixed, l1, l3);
                Cc[7 * P64_N1 + i_own] = l1;
                Cc[8 * P64_N1 + i_own] = l3;
            }
            if (DIM == 3) {
                nP[2] = xfma(xmul(k.iE, k.f[2]), k.f[2], k.a);
                speeds64(k, k.f[2], fixed, nl1, nl3);
            }
        }
        if (h_need && !flat) {
            const double U[4] = {Um[i_h], Um[P64_N1 + i_h], Um[2 * P64_N1 + i_h], Um[3 * P64_N1 + i_h]};
            const Closure64 k = closure64(U, p1);
            const double fd = h_isx ? k.f[0] : k.f[1], tt = xmul(k.iE, fd);
            double l1, l3;
            speeds64(k, fd, fixed, l1, l3);
            // the same roundings as the own cells' rows
            if (h_isx) {
                Cc[i_h] = xfma(tt, k.f[0], k.a);
                Cc[P64_N1 + i_h] = xmul(tt, k.f[1]);
                Cc[2 * P64_N1 + i_h] = xmul(tt, k.f[2]);
                Cc[5 * P64_N1 + i_h] = l1;
                Cc[6 * P64_N1 + i_h] = l3;
            } else {
                Cc[P64_N1 + i_h] = xmul(xmul(k.iE, k.f[0]), k.f[1]);
                Cc[3 * P64_N1 + i_h] = xfma(tt, k.f[1], k.a);
                Cc[4 * P64_N1 + i_h] = xmul(tt, k.f[2]);
                Cc[7 * P64_N1 + i_h] = l1;
                Cc[8 * P64_N1 + i_h] = l3;
            }
        }
        __syncthreads();
        // first-order HLL fluxes: the x face left of the own cell, the y face below it, the faces beyond
        auto face = [&](bool isx, int flx, int fly) {
            const int iR = chk((flx + 1) + w1 * (fly + 1), P64_N1), iL = chk(iR - (isx ? 1 : w1), P64_N1);
            const int r0 = isx ? 0 : 1, r1 = isx ? 1 : 3, r2 = isx ? 2 : 4, rl = isx ? 5 : 7, rg = isx ? 1 : 2;
            double UL[4], UR[4], F[4];
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) {
                UL[qq] = Um[qq * P64_N1 + iL];
                UR[qq] = Um[qq * P64_N1 + iR];
            }
            const double FL[4] = {Um[rg * P64_N1 + iL], Cc[r0 * P64_N1 + iL], Cc[r1 * P64_N1 + iL], Cc[r2 * P64_N1 + iL]};
            const double FR[4] = {Um[rg * P64_N1 + iR], Cc[r0 * P64_N1 + iR], Cc[r1 * P64_N1 + iR], Cc[r2 * P64_N1 + iR]};
            hll64(UL, UR, FL, FR, Cc[rl * P64_N1 + iL], Cc[(rl + 1) * P64_N1 + iL], Cc[rl * P64_N1 + iR],
                  Cc[(rl + 1) * P64_N1 + iR], F);
            double* dst = isx ? Fx + chk(flx + (w + 1) * fly, P64_NF) : Fy + chk(flx + w * fly, P64_NF);
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) dst[qq * P64_NF] = F[qq];
        };
        if (!flat) {
            if (own && gy < ey) face(true, lx, ly);
            if (own && gx < ex) face(false, lx, ly);
            if (has_e && x0 + elx <= ex && y0 + ely <= ey) face(e_isx, elx, ely);
        }
        __syncthreads();
        // own cell: flux differences, the z face (q - 1 | q), U^{m+1/2} of plane p.  No barrier follows:
        // what the next plane writes to shared memory, it writes after its first barrier.
        if (own) {
            double nd[4];
            if (emit_cell && !flat) {
                const int fl = lx + (w + 1) * ly, fb = lx + w * ly;
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) {
                    nd[qq] = xfma(-hx, xadd(Fx[qq * P64_NF + fl + 1], -Fx[qq * P64_NF + fl]), nU[qq]);
                    nd[qq] = xfma(-hy, xadd(Fy[qq * P64_NF + fb + w], -Fy[qq * P64_NF + fb]), nd[qq]);
                }
            } else {
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) nd[qq] = nU[qq];
            }
            double zfh[4] = {0.0, 0.0, 0.0, 0.0};
            if (DIM == 3 && q > qbeg) {
                const double FL[4] = {zU[3], zP[0], zP[1], zP[2]}, FR[4] = {nU[3], nP[0], nP[1], nP[2]};
                hll64(zU, nU, FL, FR, zl1, zl3, nl1, nl3, zfh);
            }
            if (emit) {
                double U0[4], U[4];
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) {
                    U0[qq] = DIM == 3 ? zU[qq] : nU[qq];
                    U[qq] = DIM == 3 ? xfma(-hz, xadd(zfh[qq], -zfl[qq]), acc[qq]) : nd[qq];
                }
                sources64(g, gc, U0, chat * hdt, chat * hdt * g.inv_c, has_j, U);
                const int fx_ = realize(U, g.E_floor);
                if (own_interior && p >= 0 && p < g.n[2]) cnt.fix += fx_;
                const long long po = chk((long long)(gx + g.pad[0]) +
                                             (long long)upad_extent(g, 0) * ((long long)(gy + g.pad[1]) +
                                                                             (long long)upad_extent(g, 1) * (p + (DIM == 3 ? g.pad[2] : 0))),
                                         n_padded(g));
                reinterpret_cast<double2*>(uh)[2 * po] = make_double2(U[0], U[1]);
                reinterpret_cast<double2*>(uh)[2 * po + 1] = make_double2(U[2], U[3]);
            }
            if (DIM == 3) {
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) {
                    zfl[qq] = zfh[qq];
                    zU[qq] = nU[qq];
                    acc[qq] = nd[qq];
                }
#pragma unroll
                for (int qq = 0; qq < 3; ++qq) zP[qq] = nP[qq];
                zl1 = nl1;
                zl3 = nl3;
            }
        }
    }
    cp_async_wait_all();
    __syncthreads();
}

// Corrector over the w x h interior tile at (x0, y0), planes [z0, z1) (3D; 2D: the one plane)
template <int DIM>
__device__ __forceinline__ void corrector_tile64(const GridParams& g, const GridArrays& a, const double* uh, double chat,
                                                 double dt, int x0, int y0, int w, int h, int z0, int z1, double* sm,
                                                 Counters& cnt)
{
    const int t = threadIdx.x;
    double2* UA = reinterpret_cast<double2*>(sm);  // (E, Gx) of the tile + 2 region, two plane buffers
    double2* UB = UA + 2 * P64_N2;                 // (Gy, Gz)
    double* Sx = sm + 8 * P64_N2;                  // plus records of cells -1 .. w - 1 along x
    double* Sy = Sx + 9 * P64_NF;                  // of cells -1 .. h - 1 along y
    double* Se = Sy + 9 * P64_NF;                  // minus records of column w, then of row h
    double* Cx = Se + 9 * P64_NE;
    double* Cy = Cx + 4 * P64_NF;
    double* oD = Cy + 4 * P64_NF + t;              // oD[q NT]: the own cell's E, Gx, Gy, Gz, T
    const double cx = chat * dt * g.inv_dx[0], cy = chat * dt * g.inv_dx[1], cz = chat * dt * g.inv_dx[2];
    const int p1 = g.closure == 1, fixed = g.speeds == 1, lim = g.limiter;
    const bool needT = g.exchange == EX_FULL || g.exchange == EX_FROZEN_T || g.exchange == EX_LINEAR;
    const bool has_j = a.j != nullptr, full = g.exchange == EX_FULL, linear = g.exchange == EX_LINEAR;
    const int w2 = w + 4, n2 = w2 * (h + 4);
    const long long px = upad_extent(g, 0), pz = px * upad_extent(g, 1), nxy = (long long)g.n[0] * g.n[1];
    const int lx = t % w, ly = t / w, gx = x0 + lx, gy = y0 + ly;
    const bool own_col = t < w * h && gx < g.n[0] && gy < g.n[1];
    const bool own = t < w * h && gx <= g.n[0] && gy <= g.n[1];  // its low faces are needed
    const int i_own = (lx + 2) + w2 * (ly + 2);
    // low halo: column -1 (plus records along x), row -1 (along y); high halo: column w, row h (minus)
    const bool has_l = t < w + h, l_isx = t < h;
    const int u = P64_NT - 1 - t;
    const bool has_u = u < w + h, u_isx = u < h;
    const int i_l = l_isx ? 1 + w2 * (t + 2) : (t - h + 2) + w2;
    const int i_u = u_isx ? (w + 2) + w2 * (u + 2) : (u - h + 2) + w2 * (h + 2);
    const bool l_need = has_l && (l_isx ? y0 + t < g.n[1] : x0 + t - h < g.n[0]);
    const bool u_need = has_u && (u_isx ? x0 + w <= g.n[0] && y0 + u < g.n[1] : y0 + h <= g.n[1] && x0 + u - h < g.n[0]);
    // stored positions of the cells this thread stages (beyond the high edges of ragged tiles clamped or
    // wrapped; those values are never used)
    long long c_pos[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int c = t + r * P64_NT;
        c_pos[r] = upad_pos(g, 0, x0 + c % w2 - 2) + px * upad_pos(g, 1, y0 + c / w2 - 2);
    }
    auto zpos = [&](int k) { return DIM == 3 ? (long long)upad_pos(g, 2, k) * pz : 0ll; };
    auto issue_plane = [&](int k, int buf) {
        const long long zo = zpos(k);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int c = t + r * P64_NT;
            if (c < n2) {
                const double* src = uh + 4 * chk(zo + c_pos[r], n_padded(g));
                const int cc = chk(c, P64_N2);
                cp_async16(UA + buf * P64_N2 + cc, src);
                cp_async16(UB + buf * P64_N2 + cc, src + 2);
            }
        }
    };
    const long long colo = upad_pos(g, 0, gx) + px * upad_pos(g, 1, gy);
    auto column = [&](int k, double U[4]) {
        const double2* s = reinterpret_cast<const double2*>(uh + 4 * chk(colo + zpos(k), n_padded(g)));
        const double2 A = s[0], B = s[1];
        U[0] = A.x;
        U[1] = A.y;
        U[2] = B.x;
        U[3] = B.y;
    };
    // z pipeline of the own column: the plus record of the previous cell, the lower z flux, U^{m+1/2} at k + 1
    Rec64 zp;
    double cfl[4], uk1[4];
    if (DIM == 3 && own_col) {
        double um2[4], um1[4], u0[4], Sm[4], Sp[4];
        column(z0 - 2, um2);
        column(z0 - 1, um1);
        column(z0, u0);
        column(z0 + 1, uk1);
        face_values64(um2, um1, u0, lim, Sm, Sp);
        zp = face_rec64(Sp, 2, p1, fixed);
        const int fb = face_values64(um1, u0, uk1, lim, Sm, Sp);
        if (fb) cnt.face += 1;
        hll_rec64(zp, face_rec64(Sm, 2, p1, fixed), 2, cfl);
        zp = face_rec64(Sp, 2, p1, fixed);
    }
    issue_plane(z0, 0);
    cp_async_commit();
#pragma unroll 1
    for (int k = z0; k < z1; ++k) {
        const int buf = (k - z0) & 1;
        const double2* PA = UA + buf * P64_N2;
        const double2* PB = UB + buf * P64_N2;
        double uk2[4];
        if (DIM == 3 && own_col) column(k + 2, uk2);
        cp_async_wait_all();
        __syncthreads();
        const long long li = chk(own_col ? (long long)gx + (long long)g.n[0] * gy + (long long)k * nxy : 0ll, n_cells(g));
        GasCell<double> gc;
        if (own_col) {
            cp_async8(oD + 0 * P64_NT, a.E + li);
            cp_async8(oD + 1 * P64_NT, a.G[0] + li);
            cp_async8(oD + 2 * P64_NT, a.G[1] + li);
            cp_async8(oD + 3 * P64_NT, a.G[2] + li);
            if (needT) cp_async8(oD + 4 * P64_NT, a.T + li);
            gc = load_gas<double, false>(g, a, gx, gy, k, false, true);
        }
        cp_async_commit();
        if (k + 1 < z1) issue_plane(k + 1, buf ^ 1);
        cp_async_commit();
        auto cell = [&](int i, double U[4]) {
            const double2 A = PA[i], B = PB[i];
            U[0] = A.x;
            U[1] = A.y;
            U[2] = B.x;
            U[3] = B.y;
        };
        // the two face values of the cell at i in the direction whose neighbours are di away
        auto values = [&](int i, int di, double Sm[4], double Sp[4]) {
            double um[4], u0[4], up[4];
            cell(chk(i - di, P64_N2), um);
            cell(chk(i, P64_N2), u0);
            cell(chk(i + di, P64_N2), up);
            return face_values64(um, u0, up, lim, Sm, Sp);
        };
        // (1) face records: the own cell's plus records to shared memory, its minus records kept; the halo's
        Rec64 mx, my;
        if (own) {
            double Sm[4], Sp[4];
            int fb = values(i_own, 1, Sm, Sp);
            if (fb && own_col) cnt.face += 1;
            if (gy < g.n[1]) {
                put_rec64(Sx, P64_NF, chk(lx + 1 + (w + 1) * ly, P64_NF), face_rec64(Sp, 0, p1, fixed));
                mx = face_rec64(Sm, 0, p1, fixed);
            }
            fb = values(i_own, w2, Sm, Sp);
            if (fb && own_col) cnt.face += 1;
            if (gx < g.n[0]) {
                put_rec64(Sy, P64_NF, chk(lx + w * (ly + 1), P64_NF), face_rec64(Sp, 1, p1, fixed));
                my = face_rec64(Sm, 1, p1, fixed);
            }
        }
        if (l_need || u_need) {
            const bool isx = l_need ? l_isx : u_isx;
            double Sm[4], Sp[4], S[4];
            values(l_need ? i_l : i_u, isx ? 1 : w2, Sm, Sp);
#pragma unroll
            for (int q = 0; q < 4; ++q) S[q] = l_need ? Sp[q] : Sm[q];
            const Rec64 r = face_rec64(S, isx ? 0 : 1, p1, fixed);
            if (l_need) put_rec64(isx ? Sx : Sy, P64_NF, chk(isx ? (w + 1) * t : t - h, P64_NF), r);
            else put_rec64(Se, P64_NE, chk(u, P64_NE), r);
        }
        double dz[4] = {0.0, 0.0, 0.0, 0.0};
        if (DIM == 3 && own_col) {
            double uk[4], Sm[4], Sp[4], cfh[4];
            cell(i_own, uk);
            const int fb = face_values64(uk, uk1, uk2, lim, Sm, Sp);
            if (fb && k + 1 < z1) cnt.face += 1;
            hll_rec64(zp, face_rec64(Sm, 2, p1, fixed), 2, cfh);
            zp = face_rec64(Sp, 2, p1, fixed);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                dz[q] = xadd(cfh[q], -cfl[q]);
                cfl[q] = cfh[q];
                uk1[q] = uk2[q];
            }
        }
        __syncthreads();
        // (2) fluxes: the x face left of the own cell, the y face below it, the faces beyond the high edges
        if (own) {
            double F[4];
            if (gy < g.n[1]) {
                hll_rec64(get_rec64(Sx, P64_NF, chk(lx + (w + 1) * ly, P64_NF)), mx, 0, F);
#pragma unroll
                for (int q = 0; q < 4; ++q) Cx[q * P64_NF + chk(lx + (w + 1) * ly, P64_NF)] = F[q];
            }
            if (gx < g.n[0]) {
                hll_rec64(get_rec64(Sy, P64_NF, chk(lx + w * ly, P64_NF)), my, 1, F);
#pragma unroll
                for (int q = 0; q < 4; ++q) Cy[q * P64_NF + chk(lx + w * ly, P64_NF)] = F[q];
            }
        }
        if (u_need) {
            const int s = chk(u_isx ? w + (w + 1) * u : (u - h) + w * h, P64_NF);  // plus record and face alike
            double F[4];
            hll_rec64(get_rec64(u_isx ? Sx : Sy, P64_NF, s), get_rec64(Se, P64_NE, u), u_isx ? 0 : 1, F);
#pragma unroll
            for (int q = 0; q < 4; ++q) (u_isx ? Cx : Cy)[q * P64_NF + s] = F[q];
        }
        __syncthreads();
        // (3) update of the own cell.  No barrier follows: what the next plane writes to shared memory, it
        // writes after its first barrier (oD is this thread's own).
        cp_async_wait_1();  // the own cell's group; the next plane's may still be pending
        if (own_col) {
            const int fl = lx + (w + 1) * ly, fb = lx + w * ly;
            double Uhk[4], U[4];
            cell(i_own, Uhk);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                U[q] = xfma(-cx, xadd(Cx[q * P64_NF + fl + 1], -Cx[q * P64_NF + fl]), oD[q * P64_NT]);
                U[q] = xfma(-cy, xadd(Cy[q * P64_NF + fb + w], -Cy[q * P64_NF + fb]), U[q]);
                if (DIM == 3) U[q] = xfma(-cz, dz[q], U[q]);
            }
            double Tn = needT ? oD[4 * P64_NT] : 0.0;
            finish_cell64(g, a, gc, chat, dt, Uhk, U, Tn, has_j, full, linear, li, cnt);
        }
    }
    cp_async_wait_all();
    __syncthreads();
}

template <int DIM>
__global__ void __launch_bounds__(P64_NT, 2) predictor64_kernel(const __grid_constant__ StepParams P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Tile64& s = P.t64;
    const int tile = blockIdx.x;
    const int x0 = (tile % s.ptx) * s.pw - P.g.pad[0], y0 = (tile / s.ptx) * s.ph - P.g.pad[1];
    const int pz = DIM == 3 ? P.g.pad[2] : 0;
    const int z0 = (int)blockIdx.y * s.pz - pz, z1 = min(z0 + s.pz, P.g.n[2] + pz);
    Counters cnt = {0, 0, 0, 0, 0, 0, 0};
    predictor_tile64<DIM>(P.g, P.a, P.uhalf64, P.chat, P.dt, x0, y0, s.pw, s.ph, z0, z1,
                          reinterpret_cast<double*>(smem_raw), cnt);
    add_counter(&P.stats->n_fix, cnt.fix);
}

template <int DIM>
__global__ void __launch_bounds__(P64_NT, 2) corrector64_kernel(const __grid_constant__ StepParams P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Tile64& s = P.t64;
    const int tile = blockIdx.x;
    const int x0 = (tile % s.ctx) * s.cw, y0 = (tile / s.ctx) * s.ch;
    const int z0 = (int)blockIdx.y * s.cz, z1 = min(z0 + s.cz, P.g.n[2]);
    Counters cnt = {0, 0, 0, 0, 0, 0, 0};
    corrector_tile64<DIM>(P.g, P.a, P.uhalf64, P.chat, P.dt, x0, y0, s.cw, s.ch, z0, z1,
                          reinterpret_cast<double*>(smem_raw), cnt);
    add_counter(&P.stats->n_fix, cnt.fix);
    add_counter(&P.stats->n_face, cnt.face);
    add_counter(&P.stats->n_theta, cnt.theta);
    add_counter(&P.stats->n_newton_fb, cnt.newton_fb);
    add_counter(&P.stats->n_nonfinite, cnt.nonfinite);
    max_counter(&P.stats->newton_iter_max, cnt.iter_max);
}

// persistent ensemble kernels (3D grids): CTAs pull (grid, tile, z chunk) items, each grid with its own plan
template <bool PRED>
__global__ void __launch_bounds__(P64_NT, 2) ensemble64_kernel(const __grid_constant__ EnsembleParams P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ long long item_s;
    __shared__ __align__(16) EnsembleGrid eg;
    double* sm = reinterpret_cast<double*>(smem_raw);
    Counters cnt = {0, 0, 0, 0, 0, 0, 0};
    long long local;
#pragma unroll 1
    while (ens_next<PRED>(P, eg, &item_s, &local)) {
        const Tile64& s = eg.t64;
        const int tx = PRED ? s.ptx : s.ctx, nt = tx * (PRED ? s.pty : s.cty);
        const int txy = (int)(local % nt), tz = (int)(local / nt);
        if constexpr (PRED) {
            const int z0 = tz * s.pz - eg.g.pad[2], z1 = min(z0 + s.pz, eg.g.n[2] + eg.g.pad[2]);
            predictor_tile64<3>(eg.g, eg.a, eg.uhalf64, P.chat, eg.dt, (txy % tx) * s.pw - eg.g.pad[0],
                                (txy / tx) * s.ph - eg.g.pad[1], s.pw, s.ph, z0, z1, sm, cnt);
        } else {
            const int z0 = tz * s.cz, z1 = min(z0 + s.cz, eg.g.n[2]);
            corrector_tile64<3>(eg.g, eg.a, eg.uhalf64, P.chat, eg.dt, (txy % tx) * s.cw, (txy / tx) * s.ch, s.cw, s.ch,
                                z0, z1, sm, cnt);
        }
    }
    add_counter(&P.stats->n_fix, cnt.fix);
    if constexpr (!PRED) {
        add_counter(&P.stats->n_face, cnt.face);
        add_counter(&P.stats->n_theta, cnt.theta);
        add_counter(&P.stats->n_newton_fb, cnt.newton_fb);
        add_counter(&P.stats->n_nonfinite, cnt.nonfinite);
        max_counter(&P.stats->newton_iter_max, cnt.iter_max);
    }
}

}  // namespace rhd
