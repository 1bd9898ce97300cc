// cx_tile.cu -- the register-tile pass (cx_tile.cuh): which tiles and how many
// time steps a pass takes, and the dispatch to its kernels.
#include <math.h>

#include "cx_internal.h"

namespace cx {
namespace tile {
// defined in cx_tile_kernels.cuh, instantiated in cx_tile_inst.cu
template <int LAW, int MOB>
cudaError_t launch_tile_lm(const TileLaunch &a, const TilePlan &p, bool per_step, cudaStream_t st);
}  // namespace tile

cudaError_t launch_tile(int law, int mob, bool per_step, const TileLaunch &a, const TilePlan &p,
                        cudaStream_t st)
{
    if (law == CX_CHEMO_RECEPTOR)
        return mob == CX_MOBILITY_CENTRAL
                   ? tile::launch_tile_lm<CX_CHEMO_RECEPTOR, CX_MOBILITY_CENTRAL>(a, p, per_step, st)
                   : tile::launch_tile_lm<CX_CHEMO_RECEPTOR, CX_MOBILITY_UPWIND>(a, p, per_step, st);
    return mob == CX_MOBILITY_CENTRAL
               ? tile::launch_tile_lm<CX_CHEMO_CONSTANT, CX_MOBILITY_CENTRAL>(a, p, per_step, st)
               : tile::launch_tile_lm<CX_CHEMO_CONSTANT, CX_MOBILITY_UPWIND>(a, p, per_step, st);
}

namespace {

// The tile shapes that are compiled, with the time of one stage per cell of a
// tile on a busy SM (ns): the fewer rows a thread holds, the larger its share
// of y-faces that the thread below evaluates too.
struct Shape {
    int lx, r, threads;
    double ns;
};
const Shape kShapes[] = {{16, 2, 128, 0.200}, {16, 2, 256, 0.200}, {16, 2, 512, 0.200},
                         {16, 4, 128, 0.185}, {16, 4, 256, 0.185}, {16, 4, 512, 0.185},
                         {16, 6, 256, 0.175}, {16, 6, 512, 0.175},
                         {32, 6, 256, 0.175}, {32, 6, 512, 0.175}};
const int kSteps[] = {1, 2, 3, 4, 5, 6, 7, 8, 10, 12, 16, 32, 64, 128, 256, 512, 1024};

}  // namespace

// The modelled time per step of the best tiles (us), HUGE_VAL if none fits.
// The model: a pass costs a launch (1.5 us), the latency of each stage per
// round of resident blocks (barrier and dependence chain, 0.1 us, and 0.06 us
// per row of a thread over the warps of a scheduler that hide it; 0.4 us more
// where the stage draws sigma), and the SM's share of the tiles at the rates of
// kShapes, plus 0.2 ns per cell for loads and stores that another block's
// stages hide, 0.35 ns for those of a lone block.  Against the measured passes
// of 64^2 .. 2048^2 it is within about 15 %.
double plan_tiles(const TileGrid *grids, int count, int sms, bool heun, bool per_step,
                  long long steps, TilePlan *best)
{
    const double draw_us = per_step ? (heun ? 0.2 : 0.4) : 0.0;
    const double draw_ns = per_step ? (heun ? 0.10 : 0.20) : 0.0;
    double least = HUGE_VAL;
    for (const Shape &s : kShapes) {
        for (int k : kSteps) {
            if (k > steps && k > 1) break;
            TilePlan p;
            p.steps = k;
            p.lx = s.lx;
            p.r = s.r;
            p.threads = s.threads;
            p.heun = heun;
            double tiles = 0.0;
            for (int i = 0; i < count && tiles >= 0.0; ++i) {
                // tiles that keep less than a quarter of their cells do not pay
                // (and a single grid's tile rows have to fit its launch)
                const bool fits = (grids[i].nx <= p.width() || 2 * (p.width() - 2 * p.halo_x()) >= p.width()) &&
                                  (grids[i].ny <= p.height() || 2 * (p.height() - 2 * p.halo_y()) >= p.height()) &&
                                  tiles_y(grids[i].ny, p) <= 65535;
                if (fits)
                    tiles += (double)grids[i].count * tiles_x(grids[i].nx, p) * tiles_y(grids[i].ny, p);
                else
                    tiles = -1.0;
            }
            if (tiles < 0.0) continue;
            const int resident = 512 / s.threads;
            double q = tiles / sms;  // tiles of the busiest SM
            q = q <= 2.0 * resident ? ceil(q) : q + 0.5;
            const double cells = (double)p.width() * p.height();
            const double warps = s.threads / 128.0 * fmin(resident, ceil(q));  // per scheduler
            const double latency = 0.1 + 0.06 * s.r / warps + draw_us;
            const double us = 1.5 + ceil(q / resident) * p.halo_y() * latency +
                              q * cells * 1e-3 * (p.halo_y() * (s.ns + draw_ns) + (resident == 1 ? 0.35 : 0.2));
            // passes of a call of `steps` steps are of equal length
            const long long passes = (steps + k - 1) / k;
            const double per = us * (double)passes / (double)steps;
            if (per < least) {
                least = per;
                *best = p;
            }
        }
    }
    return least;
}

}  // namespace cx
