// cx_strip.cu -- several stages per pass of FP64 strips (grids one row high, as
// in the 1D front-speed study of Sec. 4.2) with a static sigma.
//
// What bounds a strip in FP64 is a scheduler's FP64 unit: a warp instruction
// holds it for 64 cycles, whatever the number of active lanes.  So the strip
// is cut as finely as it can be: one cell per lane and one warp per block, the
// warps spread over all schedulers, each taking `stages` stages in registers
// on its 32 cells and writing the ones that its missing neighbours have not
// reached (as the register tiles of cx_tile.cuh, with which it shares the
// tiling of the pass).  A face is evaluated by the lane right of it and passed
// to the left one; its sum of sigma is kept from stage to stage.  20 strips of
// 400 cells, constant law: 5.9 us per step by the march (its four-cell lanes
// keep 20 SMs busy), 0.88 by this kernel.
#include <math.h>

#include "cx_batch_types.cuh"

namespace cx {
namespace {

using namespace stencil;
using batch::InstDev;

template <int LAW, int MOB, bool HEUN>
__device__ __forceinline__ void strip_stages(const Ptrs<double> &P, int nx, const KV<double> &k,
                                             int stages, int halo, int tile)
{
    const int lane = threadIdx.x;
    const int x0 = tile * (32 - 2 * halo), x = x0 + lane;
    const long long c = pair_col(x);
    const bool inside = x < nx;
    double b = 0.0, n = 0.0, s = 0.0, ub = 0.0, un = 0.0;
    if (inside) {
        b = Vec<double>::load1(P.b + c);
        n = Vec<double>::load1(P.n + c);
        s = Vec<double>::load1(P.s + c);
    }
    const double s2 = add_rn(__shfl_up_sync(kFull, s, 1), s);
    // no flux through the faces left and right of the cell (the face left of nx
    // lies in no lane if the strip ends with the warp)
    const bool wall = x == 0 || x >= nx, wallE = x + 1 >= nx;
    for (int st = 0; st < stages; ++st) {
        const bool second = HEUN && (st & 1);
        if (HEUN && !second) {
            ub = b;
            un = n;
        }
        const double bL = __shfl_up_sync(kFull, b, 1), nL = __shfl_up_sync(kFull, n, 1);
        double ph, g;
        face_s2<LAW, MOB>(s2, nL, n, bL, b, k, ph, g);
        if (wall) ph = g = 0.0;
        double phE = __shfl_down_sync(kFull, ph, 1), gE = __shfl_down_sync(kFull, g, 1);
        if (wallE) phE = gE = 0.0;
        const double r = mul_rn(n, b);
        double ob = fma_rn(k.cA, sub_rn(phE, ph, k.m1), fma_rn(k.cR, r, b));
        double on = fma_rn(k.ncG, sub_rn(gE, g, k.m1), fma_rn(k.ncN, r, n));
        if (second) {
            ob = mul_rn(k.half, add_rn(ub, ob));
            on = mul_rn(k.half, add_rn(un, on));
        }
        b = ob;
        n = on;
    }
    // the first and the last tile lie against the walls
    const int w0 = tile == 0 ? 0 : x0 + halo, w1 = x0 + 32 >= nx ? nx : x0 + 32 - halo;
    if (x >= w0 && x < w1) {
        P.bo[c] = b;
        P.no[c] = n;
    }
}

template <int LAW, int MOB, bool HEUN>
__global__ void __launch_bounds__(32)
    strip_kernel(Ptrs<double> P, int nx, KV<double2> k, int stages, int halo)
{
    pass_wait();
    strip_stages<LAW, MOB, HEUN>(P, nx, scalar_kv<double>(k), stages, halo, blockIdx.x);
}

template <int LAW, int MOB, bool HEUN>
__global__ void __launch_bounds__(32)
    batch_strip_kernel(const InstDev<double> *__restrict__ inst, int parity, int stages, int halo,
                       const __grid_constant__ TileRuns runs)
{
    // the table is not written while a pass may be queued
    const batch::TileAt w = batch::tile_of_block(runs, blockIdx.x);
    const InstDev<double> &I = inst[w.place];
    if (!w.across && !tile_needed(w.tile, I.nx, 32, halo)) return;
    const KV<double> k = scalar_kv<double>(make_kv(I.k));
    pass_wait();
    const Ptrs<double> P{I.b[parity], I.n[parity], I.s, nullptr, nullptr, I.b[parity ^ 1],
                         I.n[parity ^ 1]};
    strip_stages<LAW, MOB, HEUN>(P, I.nx, k, stages, halo, w.tile);
}

template <int LAW, int MOB, bool HEUN>
cudaError_t launch_v(const TileLaunch &a, const TilePlan &p, cudaStream_t st)
{
    if (a.inst)
        return launch_pass(batch_strip_kernel<LAW, MOB, HEUN>, a.runs->run[a.runs->n].first, 32, 0, st,
                           (const InstDev<double> *)a.inst, a.parity, p.stages(), p.halo_x(), *a.runs);
    const StepArgs &g = *a.grid;
    const Ptrs<double> P{(const double *)g.b, (const double *)g.n, (const double *)g.s, nullptr,
                         nullptr, (double *)g.bo, (double *)g.no};
    return launch_pass(strip_kernel<LAW, MOB, HEUN>, tiles_x(g.nx, p), 32, 0, st, P, g.nx,
                       make_kv(coef_t<double>(g.k)), p.stages(), p.halo_x());
}

template <int LAW, int MOB>
cudaError_t launch_lm(const TileLaunch &a, const TilePlan &p, cudaStream_t st)
{
    return p.heun ? launch_v<LAW, MOB, true>(a, p, st) : launch_v<LAW, MOB, false>(a, p, st);
}

}  // namespace

cudaError_t launch_strip(int law, int mob, const TileLaunch &a, const TilePlan &p, cudaStream_t st)
{
    if (law == CX_CHEMO_RECEPTOR)
        return mob == CX_MOBILITY_CENTRAL ? launch_lm<CX_CHEMO_RECEPTOR, CX_MOBILITY_CENTRAL>(a, p, st)
                                          : launch_lm<CX_CHEMO_RECEPTOR, CX_MOBILITY_UPWIND>(a, p, st);
    return mob == CX_MOBILITY_CENTRAL ? launch_lm<CX_CHEMO_CONSTANT, CX_MOBILITY_CENTRAL>(a, p, st)
                                      : launch_lm<CX_CHEMO_CONSTANT, CX_MOBILITY_UPWIND>(a, p, st);
}

// Passes of strips (every grid one row high): the tiles are 32 cells wide, the
// steps per pass the ones with the least modelled time per step.  A stage
// takes 16 (constant law) or 21 (receptor) FP64 instructions of 64 cycles per
// warp of a scheduler, a pass 2 us more.  The march spends four times as much
// on a warp's 128 cells, and little less for the faces it does not evaluate
// twice; it stays ahead on strips that fill the GPU several times over.
double plan_strips(const TileGrid *grids, int count, int sms, int law, bool heun, long long steps,
                   TilePlan *best, double *march)
{
    const double stage = (law == CX_CHEMO_RECEPTOR ? 21.0 : 16.0) * 64.0 / 2070.0;
    const int per_step = heun ? 2 : 1;
    double least = HUGE_VAL, warps = 0.0;
    for (int k : {1, 2, 4, 8}) {
        TilePlan p;
        p.steps = k;
        p.lx = 8;
        p.r = 1;
        p.threads = 32;
        p.heun = heun;
        if ((k > steps && k > 1) || p.halo_x() > 8) break;
        double tiles = 0.0;
        for (int i = 0; i < count; ++i) tiles += (double)grids[i].count * tiles_x(grids[i].nx, p);
        const double us = 2.0 + ceil(tiles / (4.0 * sms)) * p.stages() * stage;
        const double per = us * (double)((steps + k - 1) / k) / (double)steps;
        if (per < least) {
            least = per;
            *best = p;
        }
    }
    for (int i = 0; i < count; ++i) warps += (double)grids[i].count * ((grids[i].nx + 127) / 128);
    *march = per_step * (2.0 + ceil(warps / (4.0 * sms)) * 4.0 * stage);
    return least;
}

}  // namespace cx
