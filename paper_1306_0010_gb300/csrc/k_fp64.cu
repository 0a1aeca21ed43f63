// k_fp64.cu -- FP64 instantiations of the fused subcycle kernel and of the ensemble kernel.
#include <algorithm>

#include "subcycle.cuh"

namespace rhd {

template <typename R, int TX, int TY, int DIM, bool SPLIT>
static cudaError_t launch_tile_kernel(const StepParams& p, cudaStream_t s)
{
    const size_t smem = tile_smem_bytes<R, TX, TY, DIM, SPLIT>();
    auto k = subcycle_kernel<R, TX, TY, DIM, SPLIT>;
    static SmemLimitOnce smem_once;
    cudaError_t e = smem_once.set(k, smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)(p.tiles_x * p.tiles_y), DIM == 3 ? (unsigned)((p.g.n[2] + p.z_chunk - 1) / p.z_chunk) : 1u);
    k<<<grid, Geo<TX, TY, DIM>::NT, smem, s>>>(p);
    return cudaGetLastError();
}

template <typename R, int TX, int TY, bool SPLIT>
static cudaError_t launch_ens_kernel(const EnsembleParams& p, int n_ctas, cudaStream_t s)
{
    const size_t smem = tile_smem_bytes<R, TX, TY, 3, SPLIT>();
    auto k = ensemble_kernel<R, TX, TY, SPLIT>;
    static SmemLimitOnce smem_once;
    cudaError_t e = smem_once.set(k, smem);
    if (e != cudaSuccess) return e;
    k<<<n_ctas, TX * TY, smem, s>>>(p);
    return cudaGetLastError();
}

template <typename R, int TX, int TY, bool SPLIT>
static int ens_occupancy()
{
    const size_t smem = tile_smem_bytes<R, TX, TY, 3, SPLIT>();
    auto k = ensemble_kernel<R, TX, TY, SPLIT>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 1;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, TX * TY, smem) != cudaSuccess || n < 1) return 1;
    return n;
}

void tile_shape(int precision, int nact, int* tx, int* ty)
{
    if (nact == 1) {
        *tx = 122;  // the name of 1D grids' one configuration, in files too (their tiles: line_plan)
        *ty = 1;
    } else if (precision == 0) {
        // one CTA of 256 threads per SM (255 registers each): against 16x8 tiles (two CTAs of 128) it
        // recomputes the predictor on 1.89 instead of 2.41 times the tile's cells, which the FP64 pipe pays
        *tx = 16;
        *ty = 16;
    } else {
        *tx = 32;
        *ty = 8;
    }
}

void ensemble_tile_shape(int precision, int* tx, int* ty)
{
    // the tiles ensemble_kernel is instantiated with (launch_ensemble_fp64, launch_ensemble_split)
    *tx = precision == 0 ? 16 : 32;
    *ty = precision == 0 ? 16 : 8;
}

bool tile_supported(int precision, int nact, int tx, int ty)
{
    int dx, dy;
    tile_shape(precision, nact, &dx, &dy);
    if (tx == dx && ty == dy) return true;
    if (nact != 3) return false;
    if (precision == 0) return false;
    return (tx == 32 && ty == 16) || (tx == 64 && ty == 8);
}

// 1D grids.  Two threads per cell and up to eight subcycles per launch (a tile of 64 - 6 x 8 = 16 cells of the
// 64 a CTA holds) while the tiles find an SM each (split: a quarter, the FP32 pipes take several warps);
// the longest run of subcycles that does, since the halo's redone work is on idle SMs.  Beyond that (8816
// cells in FP64, 35264 split) one thread per cell and one subcycle per launch, where the cells beyond a
// tile cost a twentieth and not three quarters of the work.  A line with one periodic end alone has ghost cells
// from its far end, which only the state in memory holds: one subcycle per launch.
LinePlan line_plan(const GridParams& g, bool split, int n_sms)
{
    const long long most = (long long)n_sms * (split ? 4 : 1);
    const bool half_periodic = (g.bc_lo[0] == BC_PERIODIC) != (g.bc_hi[0] == BC_PERIODIC);
    for (int steps = half_periodic ? 1 : 8; steps >= 1; --steps) {
        const int tile = LINE_NT / 2 - 6 * steps;
        if ((g.n[0] + tile - 1) / tile <= most) return {2, steps};
    }
    return {1, 1};
}

LineParams line_params(const StepParams& p, int steps, int tpc, double* To)
{
    LineParams l;
    l.g = p.g;
    l.a = p.a;
    l.To = To;
    l.chat = p.chat;
    l.dt = p.dt;
    l.f_chat = p.f_chat;
    l.f_dt = p.f_dt;
    l.steps = steps;
    l.tile = LINE_NT / tpc - 6 * steps;
    l.stats = p.stats;
    return l;
}

cudaError_t launch_line_fp64(const LineParams& p, int tpc, cudaStream_t s)
{
    const unsigned nb = (unsigned)((p.g.n[0] + p.tile - 1) / p.tile);
    if (tpc == 2) line_kernel<double, 2><<<nb, LINE_NT, 0, s>>>(p);
    else line_kernel<double, 1><<<nb, LINE_NT, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_line(const LineParams& p, bool split, int tpc, cudaStream_t s)
{
    return split ? launch_line_split(p, tpc, s) : launch_line_fp64(p, tpc, s);
}

cudaError_t launch_subcycle_fp64(const StepParams& p, cudaStream_t s)
{
    switch (p.g.nact) {
    case 1: return cudaErrorInvalidValue;  // 1D grids: launch_line
    case 2: return launch_tile_kernel<double, 16, 16, 2, false>(p, s);
    default: return launch_tile_kernel<double, 16, 16, 3, false>(p, s);
    }
}

// ------------------------------------------------------------------------------------------------ pair
// FP64 instructions of a tile's plane in units of one warp, counted from subcycle_fp64_pair.cuh (own
// cells, halo cells, faces beyond the edges; whole warps), and the share of a plane that starting a z
// chunk costs.
namespace {
struct PairCost {
    double own, halo, face, start;
};
constexpr PairCost kPred3 = {180.0, 40.0, 23.0, 0.6}, kPred2 = {140.0, 40.0, 23.0, 0.0};
constexpr PairCost kCorr3 = {432.0, 56.0, 23.0, 0.4}, kCorr2 = {305.0, 56.0, 23.0, 0.0};

double plane_cost(const PairCost& c, bool predictor, int w, int h)
{
    const int edge = (w + h + 31) / 32, halo = predictor ? (2 * (w + h) + 31) / 32 : 2 * edge;
    return c.own * ((w * h + 31) / 32) + c.halo * halo + c.face * edge;
}

// Tile shape and planes per CTA for an ex x ey x ez range: the fewest FP64 instructions on the busiest SM.
// An SM's time is the sum over its CTAs (the pipe is shared), with a tenth more where it has only one to
// fill the gaps between its phases.  128^3: 16 x 16 x 19 (448 CTAs, three per SM; with 32 planes per CTA one
// SM in three would have half the work), 1157 + 2292 us a subcycle, 4960 for the fused kernel.
void best_split(const PairCost& c, bool predictor, int ex, int ey, int ez, int n_sms, int z_fixed, bool shared,
                int* bw, int* bh, int* bz)
{
    double best = -1.0;
    for (int w = 8; w <= 32; ++w)
        for (int h = 8; h <= 32 && w * h <= 256; ++h) {
            if (w * h < 192 && w < ex && h < ey) continue;
            const long long tiles = (long long)((ex + w - 1) / w) * ((ey + h - 1) / h);
            const double pc = plane_cost(c, predictor, w, h);
            for (int nz = 1; nz <= ez; ++nz) {
                const int z = z_fixed > 0 ? std::min(z_fixed, ez) : (ez + nz - 1) / nz;
                const long long ctas = tiles * ((ez + z - 1) / z);
                const long long per_sm = (ctas + n_sms - 1) / n_sms;
                const double load = shared ? (double)ctas : (double)per_sm * (per_sm == 1 ? 1.1 : 1.0);
                const double cost = load * pc * (z + c.start);
                if (best < 0.0 || cost < best * 0.999) {
                    best = cost;
                    *bw = w;
                    *bh = h;
                    *bz = z;
                }
                if (z_fixed > 0 || z <= 4 || per_sm > 24) break;
            }
        }
}
}  // namespace

Tile64 pair64_plan(const GridParams& g, int n_sms, int z_chunk, bool shared_queue)
{
    Tile64 s;
    const bool d3 = g.nact == 3;
    const int e[3] = {upad_extent(g, 0), upad_extent(g, 1), d3 ? upad_extent(g, 2) : 1};
    best_split(d3 ? kPred3 : kPred2, true, e[0], e[1], e[2], n_sms, z_chunk, shared_queue, &s.pw, &s.ph, &s.pz);
    best_split(d3 ? kCorr3 : kCorr2, false, g.n[0], g.n[1], d3 ? g.n[2] : 1, n_sms, z_chunk, shared_queue, &s.cw, &s.ch,
               &s.cz);
    s.ptx = (e[0] + s.pw - 1) / s.pw;
    s.pty = (e[1] + s.ph - 1) / s.ph;
    s.ctx = (g.n[0] + s.cw - 1) / s.cw;
    s.cty = (g.n[1] + s.ch - 1) / s.ch;
    return s;
}

template <typename K>
static cudaError_t launch_pair64(K k, size_t smem, SmemLimitOnce& once, dim3 grid, const StepParams& p, cudaStream_t s)
{
    cudaError_t e = once.set(k, smem);
    if (e != cudaSuccess) return e;
    k<<<grid, P64_NT, smem, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_predictor64(const StepParams& p, cudaStream_t s)
{
    static SmemLimitOnce once;
    const Tile64& t = p.t64;
    const int ez = p.g.nact == 3 ? upad_extent(p.g, 2) : 1;
    const dim3 grid((unsigned)(t.ptx * t.pty), (unsigned)((ez + t.pz - 1) / t.pz));
    return p.g.nact == 3 ? launch_pair64(predictor64_kernel<3>, pair64_pred_smem(), once, grid, p, s)
                         : launch_pair64(predictor64_kernel<2>, pair64_pred_smem(), once, grid, p, s);
}

cudaError_t launch_corrector64(const StepParams& p, cudaStream_t s)
{
    static SmemLimitOnce once;
    const Tile64& t = p.t64;
    const int nz = p.g.nact == 3 ? p.g.n[2] : 1;
    const dim3 grid((unsigned)(t.ctx * t.cty), (unsigned)((nz + t.cz - 1) / t.cz));
    return p.g.nact == 3 ? launch_pair64(corrector64_kernel<3>, pair64_corr_smem(), once, grid, p, s)
                         : launch_pair64(corrector64_kernel<2>, pair64_corr_smem(), once, grid, p, s);
}

cudaError_t launch_ensemble_pair64(const EnsembleParams& p, bool predictor, int n_ctas, cudaStream_t s)
{
    static SmemLimitOnce once;
    const size_t smem = predictor ? pair64_pred_smem() : pair64_corr_smem();
    auto k = predictor ? ensemble64_kernel<true> : ensemble64_kernel<false>;
    cudaError_t e = once.set(k, smem);
    if (e != cudaSuccess) return e;
    k<<<n_ctas, P64_NT, smem, s>>>(p);
    return cudaGetLastError();
}

int ensemble_ctas_per_sm_pair64()
{
    int n = 0;
    auto k = ensemble64_kernel<false>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pair64_corr_smem()) != cudaSuccess) return 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, P64_NT, pair64_corr_smem()) != cudaSuccess || n < 1) return 1;
    return n;
}

cudaError_t launch_ensemble_fp64(const EnsembleParams& p, int n_ctas, cudaStream_t s)
{
    return launch_ens_kernel<double, 16, 16, false>(p, n_ctas, s);
}

int ensemble_ctas_per_sm_fp64() { return ens_occupancy<double, 16, 16, false>(); }

// The stiff exchange integrated once per gas step (Section 3.1 step 2, the paper's placement of S_i): in
// every cell, E floored at E_floor, then the FULL quartic theta scheme of the subcycles (exchange_fp64,
// Eqs. source:energyupdate - source:polynomial) over dt = Delta t_gas, then |G| <= E by rescaling G.
// FP64 on every grid: it runs once per gas step, not per subcycle.  One thread per cell, grid-stride.
__global__ void __launch_bounds__(256) gas_exchange_kernel(const __grid_constant__ GasExchangeParams P)
{
    Counters cnt = {0, 0, 0, 0, 0, 0, 0};
    const GridParams& g = P.g;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += (long long)gridDim.x * blockDim.x) {
        double E = P.E[i], T = P.T[i];
        const double rho = P.rho[i];
        const double kP = P.kP ? P.kP[i] : kappa_law(g.kappa_P, g.kpow, rho);
        if (!(d2f_trunc(E) > g.f_E_floor * 1.001f) && E < g.E_floor) E = g.E_floor;
        const ExchangeOut o = exchange_fp64(g, P.chat, P.dt, rho, kP, E, T);
        cnt.theta += o.theta_fb;
        cnt.newton_fb += o.newton_fb;
        cnt.iter_max = max(cnt.iter_max, (unsigned)o.iters);
        double G[3] = {P.G[0][i], P.G[1][i], P.G[2][i]};
        const double U[4] = {E, G[0], G[1], G[2]};
        if (!surely_realizable(U)) {
            const double g2 = G[0] * G[0] + G[1] * G[1] + G[2] * G[2];
            if (g2 > E * E) {
                const double sc = E / sqrt(g2);
                G[0] *= sc;
                G[1] *= sc;
                G[2] *= sc;
                cnt.fix += 1;
            }
        }
        cnt.nonfinite += !(finite_d(E) && finite_d(T) && finite_d(G[0]) && finite_d(G[1]) && finite_d(G[2]));
        P.E[i] = E;
        P.T[i] = T;
        P.G[0][i] = G[0];
        P.G[1][i] = G[1];
        P.G[2][i] = G[2];
    }
    add_counter(&P.stats->n_fix, cnt.fix);
    add_counter(&P.stats->n_theta, cnt.theta);
    add_counter(&P.stats->n_newton_fb, cnt.newton_fb);
    add_counter(&P.stats->n_nonfinite, cnt.nonfinite);
    max_counter(&P.stats->newton_iter_max, cnt.iter_max);
}

cudaError_t launch_gas_exchange(const GasExchangeParams& p, int num_sms, cudaStream_t s)
{
    const long long blocks = std::min<long long>((p.n + 255) / 256, (long long)num_sms * 8);
    gas_exchange_kernel<<<(unsigned)std::max<long long>(blocks, 1), 256, 0, s>>>(p);
    return cudaGetLastError();
}

// Out-of-range index record of this module's kernels (debug builds; the release build has none and
// reports 0): copied to *out on stream s and, with reset, zeroed after the copy.
cudaError_t oob_read_fp64(OobRecord* out, int reset, cudaStream_t s)
{
#ifdef RHD_BOUNDS_CHECK
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_oob);
    if (e != cudaSuccess) return e;
    if (out && (e = cudaMemcpyAsync(out, p, sizeof(OobRecord), cudaMemcpyDeviceToHost, s)) != cudaSuccess)
        return e;
    return reset ? cudaMemsetAsync(p, 0, sizeof(OobRecord), s) : cudaSuccess;
#else
    (void)reset;
    (void)s;
    if (out) *out = OobRecord{0, 0, 0, 0, 0};
    return cudaSuccess;
#endif
}
bool bounds_checked_fp64()
{
#ifdef RHD_BOUNDS_CHECK
    return true;
#else
    return false;
#endif
}

}  // namespace rhd
