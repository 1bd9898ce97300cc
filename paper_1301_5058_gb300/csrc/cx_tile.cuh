// cx_tile.cuh -- the register tile: a block holds a tile of the grid in
// registers, takes several explicit stages of Eq. ka-chem-model on it and
// writes the cells that its missing surroundings have not reached.
//
// Geometry.  LX lanes side by side hold 4 LX columns (4 adjacent cells of R
// consecutive rows per thread), blockDim.x / LX of these thread rows stand on
// one another.  A stage needs the cells around a thread's: x-neighbours come
// from the adjacent lanes by shuffles, the rows below and above from the
// threads below and above through shared memory (every thread publishes its
// first and last row; two buffers, so one barrier per stage).  The block
// starts from the state of the pass's start, so a cell is right after s
// stages if it lies at least s cells inside every tile edge that is not a
// wall; the tiles overlap by that much and each writes its valid part.
// What the outermost lanes and rows compute from missing neighbours spoils
// one more cell per stage and is never written.
//
// Each stage evaluates exactly the operations of the one-stage march
// (cx_stencil.cuh) on the same operands, so a pass of s stages is bit for
// bit the s passes it replaces.
//
// What bounds it.  A small grid stepped by the marches waits: for the launch
// of every pass, and for a handful of warps' dependence chains.  Here a pass
// of 8 steps costs one launch and every SM holds a tile; what is left is the
// FMA pipes (a paired FP32 instruction takes two of a scheduler's cycles, 37
// operations per cell and stage; a busy SM takes about 47 cycles per warp and
// cell) and the overlap, which grows with the steps per pass and shrinks with
// the tile: 64 x 32 cells x 8 steps at 256^2 keeps 38 %, 128 x 48 x 4 at 2048^2
// 78 %.  Euler, static sigma, us per step, marches -> tiles: 64^2 1.5 -> 0.67,
// 256^2 2.7 -> 0.74, 512^2 3.1 -> 1.2, 1024^2 4.5 -> 2.8, 2048^2 10.1 -> 9.0;
// Heun with per-step sigma 256^2 4.4 -> 2.1, 1024^2 19.1 -> 8.3, 2048^2
// 37.1 -> 25.0; 96 instances of 256^2 38 -> 14.6.  Four shapes: 2 rows per
// thread make the smallest tiles (most SMs at work), 4 and 6 rows waste less on
// y-faces that two threads both evaluate (a share of 1/(2 R)); 6 rows of 64
// columns stand beside those of 128 because a tall tile fits some grids better
// (96 instances of 256^2 14.6 -> 13.4 us per step, 1501 x 1037 5.0 -> 4.7).  A static
// sigma's face sums are kept in shared memory from stage to stage (3-5 %).
#pragma once

#include "cx_stencil.cuh"

namespace cx {
namespace stencil {

// Where a tile lies: its first column and row, and the columns and rows that
// it writes.
struct TileBox {
    int x, y, wx0, wx1, wy0, wy1;
};

// Tile i of a row (or column) of n cells, tiles of `size` cells overlapping
// by 2 halo: the first and the last lie against the walls and need no halo
// there.
__device__ __forceinline__ void tile_span(int i, int n, int size, int halo, int &origin, int &w0,
                                          int &w1)
{
    origin = i * (size - 2 * halo);
    w0 = i == 0 ? 0 : origin + halo;
    w1 = origin + size >= n ? n : origin + size - halo;
}

// Bytes of shared memory of a block of `threads` threads: the published rows
// (b and n, first and last, two buffers) and two values per cell of the tile:
// the face sums of a static sigma, or two buffers of a sigma that is redrawn
// every step.
template <typename T, int R> constexpr size_t tile_smem(int threads)
{
    return sizeof(Cells<T>) * (size_t)threads * (8 + 2 * R);
}

template <typename T, int LAW, int MOB, int NOISE, bool HEUN, int LX, int R, bool EDGE>
__device__ __forceinline__ void tile_stages(const Ptrs<T> &P, int nx, int ny, long long pitch,
                                            const KV<P2<T>> &k, NoiseT<T> nz, int steps,
                                            const TileBox &box, Cells<T> *smem)
{
    const int th = threadIdx.x, nth = blockDim.x;
    const int lx = th % LX, ty = th / LX, nty = nth / LX;
    const int x0 = box.x + lx * kCells, y0 = box.y + ty * R;
    // the threads below and above (at the tile's edges itself: what depends on
    // it is never written)
    const int below = ty > 0 ? th - LX : th, above = ty + 1 < nty ? th + LX : th;
    Cells<T> *rows = smem;               // [buffer][b0, n0, bl, nl][thread]
    Cells<T> *tab = smem + 8 * nth;      // [2][row of the thread][thread], see tile_smem

    Cells<T> b[R], n[R], ub[R], un[R];
    auto load = [&](const T *f, int r) -> Cells<T> {
        if (EDGE && (x0 >= nx || y0 + r >= ny)) return zero_cells<T>();
        T v[kCells];
        Vec<T>::load(f + (long long)(y0 + r) * pitch + x0, v);
        return split4(v);
    };
#pragma unroll
    for (int r = 0; r < R; ++r) {
        b[r] = load(P.b, r);
        n[r] = load(P.n, r);
    }
    if (NOISE == 0) {
        // sigma's face sums, once for all stages: two additions in thirteen
        // operations of a face
        Cells<T> s = load(P.s, 0);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const Cells<T> sA = r + 1 < R || ty + 1 < nty ? load(P.s, r + 1) : s;
            tab[r * nth + th] = x_sums(s, __shfl_up_sync(kFull, s.O.y, 1, LX));
            tab[(R + r) * nth + th] = y_sums(s, sA);
            s = sA;
        }
    }

    const int stages = HEUN ? 2 * steps : steps;
#pragma unroll 1
    for (int st = 0; st < stages; ++st) {
        const bool second = HEUN && (st & 1);
        Cells<T> *pub = rows + (st & 1) * 4 * nth;
        pub[th] = b[0];
        pub[nth + th] = n[0];
        pub[2 * nth + th] = b[R - 1];
        pub[3 * nth + th] = n[R - 1];
        const Cells<T> *sg = tab;
        if (NOISE) {
            // a new sigma for every time step, beside the one still being read
            Cells<T> *w = tab + ((HEUN ? st >> 1 : st) & 1) * R * nth;
            if (!second) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    T v[kCells];
                    nz.four((long long)(y0 + r) * nx + x0, v);
                    w[r * nth + th] = split4_nat(v);
                }
                nz.step += 1;
            }
            sg = w;
        }
        if (HEUN && !second) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                ub[r] = b[r];
                un[r] = n[r];
            }
        }
        __syncthreads();
        Cells<T> s;  // NOISE: sigma of the row at hand
        YFaces<T> yB;
        if (NOISE) {
            s = sg[th];
            yB = row_yfaces<T, LAW, MOB>(sg[(R - 1) * nth + below], pub[3 * nth + below],
                                         pub[2 * nth + below], s, n[0], b[0], k);
        } else {
            yB = row_yfaces_s2<T, LAW, MOB>(tab[(2 * R - 1) * nth + below], pub[3 * nth + below],
                                            pub[2 * nth + below], n[0], b[0], k);
        }
        if (EDGE && y0 == 0) yB = zero_yfaces<T>();
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const Cells<T> nA = r + 1 < R ? n[r + 1 < R ? r + 1 : r] : pub[nth + above];
            const Cells<T> bA = r + 1 < R ? b[r + 1 < R ? r + 1 : r] : pub[above];
            Cells<T> sA, sx;
            YFaces<T> yA;
            if (NOISE) {
                sA = r + 1 < R ? sg[(r + 1) * nth + th] : sg[above];
                yA = row_yfaces<T, LAW, MOB>(s, n[r], b[r], sA, nA, bA, k);
                sx = x_sums(s, __shfl_up_sync(kFull, s.O.y, 1, LX));
            } else {
                yA = row_yfaces_s2<T, LAW, MOB>(tab[(R + r) * nth + th], n[r], b[r], nA, bA, k);
                sx = tab[r * nth + th];
            }
            if (EDGE && y0 + r + 1 >= ny) yA = zero_yfaces<T>();
            const T lb = __shfl_up_sync(kFull, b[r].O.y, 1, LX);
            const T ln = __shfl_up_sync(kFull, n[r].O.y, 1, LX);
            const XFaces<T> xf =
                row_xfaces_s2<T, LAW, MOB, !EDGE, LX>(sx, n[r], b[r], ln, lb, k, x0, nx);
            Cells<T> ob, on;
            row_update<T, +1>(b[r], n[r], xf, yB, yA, k, ob, on);
            if (HEUN && second) {
                ob = heun_mean(ub[r], ob, k);
                on = heun_mean(un[r], on, k);
            }
            b[r] = ob;
            n[r] = on;
            yB = yA;
            if (NOISE) s = sA;
        }
    }

    if (x0 < box.wx0 || x0 >= box.wx1) return;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int j = y0 + r;
        if (j < box.wy0 || j >= box.wy1) continue;
        T vb[kCells], vn[kCells];
        const long long off = (long long)j * pitch + x0;
        if (!EDGE || x0 + kCells <= nx) {
            join4(b[r], vb);
            join4(n[r], vn);
            Vec<T>::store(P.bo + off, vb);
            Vec<T>::store(P.no + off, vn);
        } else {
            // the row's last group: cell x0 + c lives at column x0 + pair_col(c)
            join4_nat(b[r], vb);
            join4_nat(n[r], vn);
#pragma unroll
            for (int c = 0; c < kCells; ++c)
                if (x0 + c < nx) {
                    P.bo[off + pair_col(c)] = vb[c];
                    P.no[off + pair_col(c)] = vn[c];
                }
        }
    }
}

}  // namespace stencil
}  // namespace cx
