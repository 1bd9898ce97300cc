// cx_batch_types.cuh -- device-side records of a batch (cx_batch.cu,
// cx_batch_kernels.cuh): the per-instance table entry and the state of the
// resident kernel's grid barrier.
#pragma once

#include "cx_stencil.cuh"

namespace cx {
namespace batch {

using stencil::CoefT;

template <typename T> struct InstDev {
    T *b[2];
    T *n[2];
    const T *s;
    int nx, ny;
    long long pitch;
    CoefT<T> k;
    float fth;     // FP32 envelope threshold (diagnostics)
    double bth;    // FP64 envelope threshold
    // per-step noise: sigma = sigma0 (1 + amp Delta(seed, cell, step)), Delta
    // of law `dist`, by the recipe of the state's precision
    uint64_t seed;
    T sigma0, amp;
    int dist;
};

// The per-step noise of instance I at time step `step`, as a single grid
// with the same seed draws it.
template <typename T>
__device__ __forceinline__ stencil::NoiseT<T> inst_noise(const InstDev<T> &I, uint64_t step)
{
    stencil::NoiseT<T> nz{};
    nz.seed = I.seed;
    nz.step = step;
    nz.dist = I.dist;
    nz.sigma0 = I.sigma0;
    nz.amp = I.amp;
    if constexpr (sizeof(T) == 4) nz.set_keys();
    return nz;
}

// t / d for t >= 0, d >= 1.  (t + 1/2) / d lies 1 / 2d or more from an integer and
// the fast division is off by 2 ulp, less than that while t < 2^20.  Every block
// of a pass begins with it (129 different grids of up to 311 x 149, 256 steps:
// 1243 us with integer divisions, 1237 so).
__device__ __forceinline__ int quotient(int t, int d)
{
    return t < (1 << 20) ? (int)__fdividef((float)t + 0.5f, (float)d) : t / d;
}

// What block `blk` of a pass over z works on: the instance's place in the table,
// which of its tiles, and how many of them lie side by side (0: see TileRuns).
struct TileAt {
    int place, tile, across;
};
__device__ __forceinline__ TileAt tile_of_block(const TileRuns &z, int blk)
{
    int k = 0, last = z.n - 1;
    if (z.n > 8) {  // (fewer lie together, in the first lines of the parameters)
        const int i = blk >> z.shift;
        k = z.index[i];
        last = z.index[i + 1];
    }
    while (k < last) {
        const int mid = (k + last + 1) / 2;
        if (blk < z.run[mid].first) last = mid - 1;
        else k = mid;
    }
    const TileRun r = z.run[k];
    const int t = blk - r.first, i = quotient(t, r.tiles);
    return TileAt{r.place + i, t - i * r.tiles, r.across};
}

// State of the resident kernel's grid-wide barrier (cx_batch_kernels.cuh).
struct GridBarrier {
    unsigned count, gen;
    int err, pad;
};

}  // namespace batch
}  // namespace cx
