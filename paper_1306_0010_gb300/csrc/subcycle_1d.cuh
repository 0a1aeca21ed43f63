// subcycle_1d.cuh -- the radiation subcycle of 1D grids (both precisions), several subcycles per launch
// (included by subcycle.cuh).
//
// What bounds it: latency.  A short 1D grid is a few hundred warps' worth of work on 608 SM sub-partitions,
// and a subcycle is one long dependent chain: an FP64 instruction holds a lone warp for 65 cycles whatever
// the number of active lanes, so one thread per cell took 20.5 us a subcycle in FP64 (12.5 us split,
// launch gaps and loads among it) at any N up to 2048.  Two things shorten that:
//   - a CTA keeps its cells in shared memory for `steps` subcycles: it loads its tile with a halo of
//     3 steps cells on each side and redoes the halo's (shrinking) work itself, on SMs that are idle
//     anyway, so a launch, its loads and its tail are paid once per eight subcycles and CTAs never wait
//     for one another;
//   - two threads per cell (TPC = 2, on different sub-partitions) share the corrector's two face states,
//     the longest part of the chain.
// Measured at N = 512, FP64 (radiative equilibrium): 20.8 -> 12.1 us a subcycle; N = 2048, split, Marshak:
// 12.3 -> 5.9 us.  Grids of more tiles than SMs run one subcycle per launch with one thread per cell: there
// throughput counts, and the halo's work is no longer free.
//
// Every cell's arithmetic is that of the tile kernels' formulas above (closure_scalars, wave_speeds, hll,
// theta_updates, exchange), whatever the tile and the number of subcycles per launch.
#pragma once

namespace rhd {

constexpr int LINE_NT = 128;

template <typename R>
struct LineSmem {
    double U[4][LINE_NT];     // the state of the region's cells
    R Um[4][LINE_NT];         // its copy in R, the closure's rows P_xx, P_xy, P_xz and wave speeds
    R C[5][LINE_NT];
    R F[4][LINE_NT];          // flux of the face below cell c
    R Uh[4][LINE_NT];         // U^{m+1/2}
    R S[10][LINE_NT];         // plus face states (state, flux, speeds)
};

// One face state of a cell (side 0: minus, 1: plus) as in face_states<0>; returns 1 if the slope was zeroed
template <typename R>
__device__ __forceinline__ int face_state_side(const R um[4], const R u0[4], const R up[4], int side, R chat, int lim,
                                               int p1, int fixed, R out[10])
{
    R Sm[4], Sp[4];
    const R h = R(0.5);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const R sl = limited(u0[q] - um[q], up[q] - u0[q], lim);
        Sm[q] = u0[q] - h * sl;
        Sp[q] = u0[q] + h * sl;
    }
    const int fb = face_unrealizable(Sm[0], Sm[1], Sm[2], Sm[3]) || face_unrealizable(Sp[0], Sp[1], Sp[2], Sp[3]);
    R S[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        S[q] = fb ? u0[q] : (side ? Sp[q] : Sm[q]);
        out[q] = S[q];
    }
    const ClosureScalars<R> k = closure_scalars(S[0], S[1], S[2], S[3], chat, p1);
    dir_flux<0>(k, S, chat, out + 4);
    wave_speeds(k, S[1], chat, fixed, out[8], out[9]);
    return fb;
}

template <typename R, int TPC>
__global__ void __launch_bounds__(LINE_NT) line_kernel(const __grid_constant__ LineParams P)
{
    constexpr int W = LINE_NT / TPC;
    constexpr bool SPLIT = sizeof(R) == 4;
    __shared__ LineSmem<R> sm;
    const GridParams& g = P.g;
    const GridArrays& a = P.a;
    const int c = threadIdx.x % W, half = threadIdx.x / W;
    const int n = g.n[0], halo = 3 * P.steps, xr = (int)blockIdx.x * P.tile - halo, x = xr + c;
    const bool owned = c >= halo && c < halo + P.tile && x < n;
    const bool wraps = g.bc_lo[0] == BC_PERIODIC && g.bc_hi[0] == BC_PERIODIC;
    const R chat = SPLIT ? (R)P.f_chat : (R)P.chat, dt = SPLIT ? (R)P.f_dt : (R)P.dt;
    const R hdt = R(0.5) * dt, idx = (R)g.inv_dx[0];
    const R E_floor = SPLIT ? (R)g.f_E_floor : (R)g.E_floor;
    const int p1 = g.closure == 1, fixed = g.speeds == 1, lim = g.limiter;
    const bool full = g.exchange == EX_FULL, linear = g.exchange == EX_LINEAR;
    const bool needT = full || linear || g.exchange == EX_FROZEN_T;
    Counters cnt = {0, 0, 0, 0, 0, 0, 0};
    SplitStiffConsts sk;
    if constexpr (SPLIT) sk = split_stiff_consts(g, P.chat, P.dt);

    // Cells whose new state is right after subcycle s: [lo(s), hi(s)).  The region loses three cells a
    // subcycle on each side, except at a boundary that is not periodic, whose ghost cells (three, all in
    // the region) are filled again from the interior before every subcycle.
    const int c_first = -xr, c_end = n - xr;  // the domain's first cell and the one past its last
    const bool low_bc = !wraps && c_first >= 3, high_bc = !wraps && c_end + 3 <= W;
    const bool ghost = !wraps && ((x >= -3 && x < 0) || (x >= n && x < n + 3));
    const bool any_ghost = !wraps && (xr < 0 || xr + W > n);

    GasCell<R> gc = load_gas<R, SPLIT>(g, a, x, 0, 0, needT, full && !SPLIT);
    double T = gc.T;
    {
        double U[4];
        load_U(g, a, x, 0, 0, U);
        if (half == 0)
#pragma unroll
            for (int q = 0; q < 4; ++q) sm.U[q][c] = U[q];
    }
#pragma unroll 1
    for (int s = 0; s < P.steps; ++s) {
        if (s > 0 && any_ghost) {
            __syncthreads();
            if (ghost && half == 0) {
                int pos[3] = {x, 0, 0}, sg[3] = {1, 1, 1};
                const int df = remap_cell(g, pos, sg, true);
                double U[4];
                if (df >= 0) {
                    const double* d = df == 0 && a.dir_dev ? a.dir_dev + 4 * s : (df == 0 ? g.dir_lo[0] : g.dir_hi[0]);
#pragma unroll
                    for (int q = 0; q < 4; ++q) U[q] = d[q];
                } else {
                    const int cs = min(max(pos[0] - xr, 0), W - 1);
#pragma unroll
                    for (int q = 0; q < 4; ++q) U[q] = sm.U[q][cs];
                    if (sg[0] < 0) U[1] = -U[1];
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) sm.U[q][c] = U[q];
            }
        }
        // closure of every cell
        if (half == 0) {
            R U[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) sm.Um[q][c] = U[q] = to_r<R>(sm.U[q][c]);
            const ClosureScalars<R> k = closure_scalars(U[0], U[1], U[2], U[3], chat, p1);
            R l1, l3;
            wave_speeds(k, U[1], chat, fixed, l1, l3);
            sm.C[0][c] = k.a + k.b * U[1] * U[1];
            sm.C[1][c] = k.b * U[1] * U[2];
            sm.C[2][c] = k.b * U[1] * U[3];
            sm.C[3][c] = l1;
            sm.C[4][c] = l3;
        }
        __syncthreads();
        // first-order HLL flux of the face (c - 1 | c)
        if (half == 0 && c > 0) {
            R UL[4], UR[4], FL[4], FR[4], F[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                UL[q] = sm.Um[q][c - 1];
                UR[q] = sm.Um[q][c];
            }
            FL[0] = chat * UL[1];
            FR[0] = chat * UR[1];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                FL[1 + q] = chat * sm.C[q][c - 1];
                FR[1 + q] = chat * sm.C[q][c];
            }
            hll(UL, UR, FL, FR, sm.C[3][c - 1], sm.C[4][c - 1], sm.C[3][c], sm.C[4][c], F);
#pragma unroll
            for (int q = 0; q < 4; ++q) sm.F[q][c] = F[q];
        }
        __syncthreads();
        // U^{m+1/2}
        if (half == 0) {
            R U0[4], U[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) U[q] = U0[q] = sm.Um[q][c];
            if (c > 0 && c < W - 1) {
                R div[4], S[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) div[q] = (sm.F[q][c + 1] - sm.F[q][c]) * idx;
                explicit_sources(g, gc, U0, chat, S);
#pragma unroll
                for (int q = 0; q < 4; ++q) U[q] = U0[q] - hdt * div[q] + hdt * S[q];
                theta_updates(g, gc, chat, hdt, U);
                const int fx = realize(U, E_floor);
                if (owned) cnt.fix += fx;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) sm.Uh[q][c] = U[q];
        }
        __syncthreads();
        // face states of the cell: minus kept, plus to shared memory
        R Sm[10], Uhk[4];
        if (c > 0 && c < W - 1) {
            R um[4], up[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                um[q] = sm.Uh[q][c - 1];
                Uhk[q] = sm.Uh[q][c];
                up[q] = sm.Uh[q][c + 1];
            }
            if (TPC == 2) {
                const int fb = face_state_side(um, Uhk, up, half, chat, lim, p1, fixed, Sm);
                if (fb && owned && half == 0) cnt.face += 1;
                if (half == 1)
#pragma unroll
                    for (int q = 0; q < 10; ++q) sm.S[q][c] = Sm[q];
            } else {
                R fs[20];
                const int fb = face_states<0>(um, Uhk, up, chat, lim, p1, fixed, fs);
                if (fb && owned) cnt.face += 1;
#pragma unroll
                for (int q = 0; q < 10; ++q) {
                    Sm[q] = fs[q];
                    sm.S[q][c] = fs[10 + q];
                }
            }
        }
        __syncthreads();
        // HLL flux of the face (c - 1 | c)
        if (half == 0 && c > 1 && c < W - 1) {
            R L[10], F[4];
#pragma unroll
            for (int q = 0; q < 10; ++q) L[q] = sm.S[q][c - 1];
            hll(L, Sm, L + 4, Sm + 4, L[8], L[9], Sm[8], Sm[9], F);
#pragma unroll
            for (int q = 0; q < 4; ++q) sm.F[q][c] = F[q];
        }
        __syncthreads();
        // the new state
        const int lo = low_bc ? c_first : max(3 * (s + 1), wraps ? 0 : c_first);
        const int hi = high_bc ? c_end : min(W - 3 * (s + 1), wraps ? W : c_end);
        if (half == 0 && c >= lo && c < hi) {
            R div[4], S[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) div[q] = (sm.F[q][c + 1] - sm.F[q][c]) * idx;
            explicit_sources(g, gc, Uhk, chat, S);
            Counters dummy = {0, 0, 0, 0, 0, 0, 0};
            Counters& ct = owned ? cnt : dummy;
            double U[4];
            gc.T = T;
            if constexpr (SPLIT) {
                double U0[4];
                float d[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    U0[q] = sm.U[q][c];
                    d[q] = -dt * div[q] + dt * S[q];
                }
                split_stiff(g, a, sk, P.f_chat, P.f_dt, gc, U0, d, T, U, ct);
                const float ef = d2f_trunc(U[0]);
                float g2f = 0.f;
#pragma unroll
                for (int q = 1; q < 4; ++q) {
                    const float gq = d2f_trunc(U[q]);
                    g2f += gq * gq;
                }
                if (!(ef > g.f_E_floor * 1.001f) || g2f > 0.9999f * ef * ef) ct.fix += realize(U, g.E_floor);
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q) U[q] = sm.U[q][c] - dt * div[q] + dt * S[q];
                theta_updates(g, gc, chat, dt, U);
                if (full) {
                    // transport can leave E <= 0 (not positivity preserving); exchange on E >= E_floor
                    if (U[0] < g.E_floor) U[0] = g.E_floor;
                    const ExchangeOut o = exchange_fp64(g, P.chat, P.dt, gc.rho, gc.kP, U[0], T);
                    ct.theta += o.theta_fb;
                    ct.newton_fb += o.newton_fb;
                    ct.iter_max = max(ct.iter_max, (unsigned)o.iters);
                } else if (linear) {
                    exchange_linear_fp64(g, P.chat, P.dt, gc.kP, U[0], T);
                }
                ct.fix += realize(U, g.E_floor);
            }
            if (owned)
                cnt.nonfinite += !(finite_d(U[0]) && finite_d(U[1]) && finite_d(U[2]) && finite_d(U[3]) &&
                                   (!(full || linear) || finite_d(T)));
#pragma unroll
            for (int q = 0; q < 4; ++q) sm.U[q][c] = U[q];
        }
    }
    if (half == 0 && owned) {
        const int i = chk(x, n_cells(g));
        a.Eo[i] = sm.U[0][c];
#pragma unroll
        for (int q = 0; q < 3; ++q) a.Go[q][i] = sm.U[1 + q][c];
        if (full || linear) P.To[i] = T;
    }
    add_counter(&P.stats->n_fix, cnt.fix);
    add_counter(&P.stats->n_face, cnt.face);
    add_counter(&P.stats->n_theta, cnt.theta);
    add_counter(&P.stats->n_newton_fb, cnt.newton_fb);
    add_counter(&P.stats->n_nonfinite, cnt.nonfinite);
    max_counter(&P.stats->newton_iter_max, cnt.iter_max);
}

}  // namespace rhd
