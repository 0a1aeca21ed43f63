// Host enumeration of what the marching gas kernels (k_gas.cu) access, through the functions of gas_index.h that they
// call: for every thread of every CTA of a march, each index it loads or stores must lie inside its array, each cell
// must be updated exactly once, and each face an update takes from shared memory must have been written there by an
// active thread.  Prints "ok <marches>" or the first violations (exit status 1).
#include <cstdio>
#include <vector>

#include "gas_index.h"

using namespace rhd;

static int fail_count = 0;
static const int* grid_n;

static void check(bool ok, const char* what, long long v, long long extent)
{
    if (ok || fail_count++ >= 5) return;
    std::printf("violation: %s = %lld of %lld for n = (%d, %d, %d)\n", what, v, extent, grid_n[0], grid_n[1], grid_n[2]);
}
static void in(long long v, long long extent, const char* what) { check(v >= 0 && v < extent, what, v, extent); }

struct Role {
    bool cell, fx, fy;
};
template <typename Tile>
static Role role(const GasParams& p, const Tile& me, int X, int Y, const int* e)
{
    return {me.cell && gas_cell_in(X, Y, e[0], e[1]), me.fx && p.n[0] > 1 && gas_xface_in(X, Y, e[0], e[1]),
            me.fy && gas_yface_in(X, Y, e[0], e[1])};
}

template <int DIM, int TX, int TY>
static void check_march(const GasParams& p, bool predictor, int num_sms)
{
    using Tile = GasTile<DIM, TX, TY>;
    const int* e = predictor ? p.m : p.n;
    const long long ncell = gas_count(p.n), next = gas_count(p.m), total = gas_count(e), row = p.m[0], plane = row * p.m[1];
    long long blocks;
    const GasMarch t = gas_march(e, TX, TY, num_sms, &blocks);
    check(t.planes >= 1, "planes", t.planes, 1);
    std::vector<int> updated((size_t)total, 0);
    for (long long blk = 0; blk < blocks; ++blk) {
        const int b = (int)(blk % t.tiles), zc = (int)(blk / t.tiles) * t.planes;
        const int ze = zc + t.planes < e[2] ? zc + t.planes : e[2];
        const int X0 = (b % t.tiles_x) * TX, Y0 = (b / t.tiles_x) * TY;
        bool wx[TY][TX + 1] = {}, wy[TY + 1][TX] = {};  // faces written (the same in every plane)
        for (int th = 0; th < Tile::NT; ++th) {
            const Tile me(th);
            const Role r = role(p, me, X0 + me.tx, Y0 + me.ty, e);
            if (r.fx) {
                in(me.tx, TX + 1, "x face column");
                in(me.ty, TY, "x face row");
                wx[me.ty][me.tx] = true;
            }
            if (r.fy) {
                in(me.tx, TX, "y face column");
                in(me.ty, TY + 1, "y face row");
                wy[me.ty][me.tx] = true;
            }
        }
        for (int th = 0; th < Tile::NT; ++th) {
            const Tile me(th);
            const int X = X0 + me.tx, Y = Y0 + me.ty;
            const Role r = role(p, me, X, Y, e);
            if (r.cell) {
                if (p.n[0] > 1) check(wx[me.ty][me.tx] && wx[me.ty][me.tx + 1], "x faces of a cell", X, e[0]);
                if (DIM > 1) check(wy[me.ty][me.tx] && wy[me.ty + 1][me.tx], "y faces of a cell", Y, e[1]);
            }
            const auto update = [&](int z) {
                const int at[3] = {X, Y, z};
                const long long i = gas_ravel(at, e);
                in(i, total, "updated cell");
                if (i >= 0 && i < total) ++updated[(size_t)i];
            };
            if (predictor) {
                const GasPredColumn c = gas_pred_column(p, X, Y);
                const long long nxy = (long long)p.n[0] * p.n[1];
                int s;
                int z = DIM > 2 ? zc - 1 : 0;
                long long base = DIM > 2 ? gas_pred_plane(p, nxy, z, s) : 0, base_n = 0;
                in(c.own + base, ncell, "predictor own");
                for (; z < ze; ++z) {
                    const bool on = DIM < 3 || z >= zc;
                    if (DIM > 2) {
                        base_n = gas_pred_plane(p, nxy, z + 1, s);
                        if (r.cell || z + 1 < ze) in(c.own + base_n, ncell, "predictor next");
                    }
                    if (on && r.fx) in(c.left + base, ncell, "predictor left");
                    if (on && r.fy) in(c.low + base, ncell, "predictor low");
                    if (on && r.cell) update(z);
                    base = base_n;
                }
            } else {
                const bool any = r.cell || r.fx || r.fy;
                const long long own = gas_corr_column(p, X, Y);
                int z = DIM > 2 ? zc - 2 : 0;
                if (any) in(own + plane * z, next, "corrector first");
                if (any && DIM > 2) in(own + plane * (z + 1), next, "corrector second");
                for (; z < ze; ++z) {
                    const bool on = DIM < 3 || z >= zc;
                    const long long x = own + plane * z;
                    if (DIM > 2 && (r.cell || (any && z + 2 < ze))) in(x + 2 * plane, next, "corrector next");
                    if (on && r.fx)
                        for (int d : {-2, -1, 1}) in(x + d, next, "corrector x neighbour");
                    if (on && r.fy)
                        for (int d : {-2, -1, 1}) in(x + d * row, next, "corrector y neighbour");
                    if (on && r.cell) update(z);
                }
            }
        }
    }
    for (long long i = 0; i < total; ++i) check(updated[(size_t)i] == 1, "updates of a cell", updated[(size_t)i], 1);
}

int main()
{
    const int shapes[][3] = {{1, 1, 1},   {3, 1, 1},   {91, 1, 1},  {92, 1, 1},  {93, 1, 1},  {97, 1, 1},  {481, 1, 1},
                             {3, 3, 1},   {28, 4, 1},  {29, 5, 1},  {33, 9, 1},  {64, 16, 1}, {3, 3, 3},   {5, 3, 7},
                             {28, 4, 8},  {29, 5, 9},  {32, 8, 16}, {33, 9, 17}, {31, 7, 40}, {60, 12, 5}};
    int marches = 0;
    for (const auto& n : shapes)
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b)
                for (int sms : {1, 8, 152})
                    for (bool predictor : {true, false}) {
                        const int lo[3] = {a, b, (a + b) % 4}, hi[3] = {b, (a + 1) % 4, a};
                        GasParams p{};
                        gas_set_geometry(p, n, lo, hi);
                        grid_n = n;
                        if (n[2] > 1) check_march<3, 32, 8>(p, predictor, sms);
                        else if (n[1] > 1) check_march<2, 32, 8>(p, predictor, sms);
                        else {
                            check_march<1, 96, 1>(p, predictor, sms);
                            check_march<1, 480, 1>(p, predictor, sms);
                        }
                        ++marches;
                    }
    if (fail_count) {
        std::printf("%d violations\n", fail_count);
        return 1;
    }
    std::printf("ok %d\n", marches);
    return 0;
}
