// cx_tile_kernels.cuh -- the register-tile kernels of a single grid and of a
// batch (cx_tile.cuh) and their launch templates, for an FP32 state.
// Included only by cx_tile_inst.cu, which the build compiles once per
// (chemotaxis law, mobility); cx_tile.cu chooses the tiles and dispatches.
#pragma once

#include "cx_batch_types.cuh"
#include "cx_tile.cuh"

namespace cx {
namespace tile {

using namespace stencil;
using batch::InstDev;
using batch::inst_noise;

// 512 threads hold an SM's registers at 128 each: one block of 512 per SM or
// two of 256.
constexpr int kMaxThreads = 512;

// The halo of a pass of `stages` stages along x: whole groups of four cells.
__device__ __forceinline__ int x_halo(int stages) { return (stages + kCells - 1) / kCells * kCells; }

// Tile (tx, ty) of a grid, `steps` time steps.
template <int LAW, int MOB, int NOISE, bool HEUN, int LX, int R>
__device__ __forceinline__ void one_tile(const Ptrs<float> &P, int nx, int ny, long long pitch,
                                         const KV<float2> &k, const NoiseT<float> &nz, int steps,
                                         int tx, int ty)
{
    extern __shared__ __align__(16) unsigned char smem[];
    Cells<float> *sm = reinterpret_cast<Cells<float> *>(smem);
    constexpr int W = LX * kCells;
    const int H = (int)(blockDim.x / LX) * R, stages = HEUN ? 2 * steps : steps;
    TileBox box;
    tile_span(tx, nx, W, x_halo(stages), box.x, box.wx0, box.wx1);
    tile_span(ty, ny, H, stages, box.y, box.wy0, box.wy1);
    // every cell of the tile and the faces around it lie inside the grid
    if (box.x > 0 && box.y > 0 && box.x + W < nx && box.y + H < ny)
        tile_stages<float, LAW, MOB, NOISE, HEUN, LX, R, false>(P, nx, ny, pitch, k, nz, steps, box, sm);
    else
        tile_stages<float, LAW, MOB, NOISE, HEUN, LX, R, true>(P, nx, ny, pitch, k, nz, steps, box, sm);
}

template <int LAW, int MOB, int NOISE, bool HEUN, int LX, int R>
__global__ void __launch_bounds__(kMaxThreads, 1)
    tile_kernel(Ptrs<float> P, int nx, int ny, long long pitch, KV<float2> k, NoiseT<float> nz,
                int steps)
{
    pass_wait();
    one_tile<LAW, MOB, NOISE, HEUN, LX, R>(P, nx, ny, pitch, k, nz, steps, blockIdx.x, blockIdx.y);
}

// One tile of an instance of a batch.
template <int LAW, int MOB, int NOISE, bool HEUN, int LX, int R>
__global__ void __launch_bounds__(kMaxThreads, 1)
    batch_tile_kernel(const InstDev<float> *__restrict__ inst, int parity, int steps,
                      const long long *step_base, int step_off,
                      const __grid_constant__ TileRuns runs)
{
    // the table is not written while a pass may be queued
    const batch::TileAt w = batch::tile_of_block(runs, blockIdx.x);
    const InstDev<float> &I = inst[w.place];
    const int stages = HEUN ? 2 * steps : steps;
    const int across = w.across ? w.across : tile_count(I.nx, LX * kCells, x_halo(stages));
    const int ty = batch::quotient(w.tile, across), tx = w.tile - ty * across;
    if (!w.across && !tile_needed(ty, I.ny, (int)(blockDim.x / LX) * R, stages)) return;
    const KV<float2> k = make_kv(I.k);
    pass_wait();
    const Ptrs<float> P{I.b[parity], I.n[parity], I.s, nullptr, nullptr, I.b[parity ^ 1],
                        I.n[parity ^ 1]};
    const NoiseT<float> nz =
        NOISE ? inst_noise(I, (uint64_t)(*step_base + step_off)) : NoiseT<float>{};
    one_tile<LAW, MOB, NOISE, HEUN, LX, R>(P, I.nx, I.ny, I.pitch, k, nz, steps, tx, ty);
}

template <int LAW, int MOB, int NOISE, bool HEUN, int LX, int R>
cudaError_t launch_v(const TileLaunch &a, const TilePlan &p, cudaStream_t st)
{
    const size_t smem = tile_smem<float, R>(p.threads);
    if (a.inst) {
        auto kern = batch_tile_kernel<LAW, MOB, NOISE, HEUN, LX, R>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        return launch_pass(kern, a.runs->run[a.runs->n].first, p.threads, smem, st,
                           (const InstDev<float> *)a.inst, a.parity, p.steps, a.nz.step_base,
                           a.nz.step_off, *a.runs);
    }
    const StepArgs &g = *a.grid;
    const KV<float2> k = make_kv(coef_t<float>(g.k));
    NoiseT<float> nz;
    nz.seed = g.sg.seed;
    nz.step = (uint64_t)g.step;
    nz.dist = g.sg.dist;
    nz.sigma0 = (float)g.sg.sigma0;
    nz.amp = (float)g.sg.amp;
    set_noise_keys(nz);
    const Ptrs<float> P{(const float *)g.b, (const float *)g.n, (const float *)g.s, nullptr, nullptr,
                        (float *)g.bo, (float *)g.no};
    auto kern = tile_kernel<LAW, MOB, NOISE, HEUN, LX, R>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_pass(kern, dim3(tiles_x(g.nx, p), tiles_y(g.ny, p)), p.threads, smem, st, P, g.nx,
                       g.ny, g.pitch, k, nz, p.steps);
}

template <int LAW, int MOB, int NOISE, bool HEUN>
cudaError_t launch_shape(const TileLaunch &a, const TilePlan &p, cudaStream_t st)
{
    if (p.lx == 16 && p.r == 2) return launch_v<LAW, MOB, NOISE, HEUN, 16, 2>(a, p, st);
    if (p.lx == 16 && p.r == 4) return launch_v<LAW, MOB, NOISE, HEUN, 16, 4>(a, p, st);
    if (p.lx == 16 && p.r == 6) return launch_v<LAW, MOB, NOISE, HEUN, 16, 6>(a, p, st);
    if (p.lx == 32 && p.r == 6) return launch_v<LAW, MOB, NOISE, HEUN, 32, 6>(a, p, st);
    return cudaErrorInvalidValue;
}

// One (law, mobility) combination: every noise mode and scheme.
template <int LAW, int MOB>
cudaError_t launch_tile_lm(const TileLaunch &a, const TilePlan &p, bool per_step, cudaStream_t st)
{
    if (per_step)
        return p.heun ? launch_shape<LAW, MOB, 1, true>(a, p, st) : launch_shape<LAW, MOB, 1, false>(a, p, st);
    return p.heun ? launch_shape<LAW, MOB, 0, true>(a, p, st) : launch_shape<LAW, MOB, 0, false>(a, p, st);
}

}  // namespace tile
}  // namespace cx
