// cx_internal.h -- internal declarations shared by the library's translation
// units: the handle layout, kernel argument blocks and launchers.
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include "cx.h"

namespace cx {

// Named range on profiler timelines for the life of a scope (NVTX; a
// no-op unless a profiling tool is attached).
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// Launches a pass kernel as a programmatic dependent of the kernel before it
// in the stream: the launch is set up while that kernel drains, and the
// kernel's blocks wait in pass_wait() for its writes instead of being launched
// after them.  A chain of small passes then costs 1.5 instead of 4.1 us per
// pass on its own (152 empty blocks), and a pass 2.3 us less: 64^2 2.7 -> 1.5,
// 256^2 4.1 -> 2.7, 1024^2 5.1 -> 4.3, 2048^2 11.3 -> 9.9 us per time step.
// The kernels do not release their dependents early
// (cudaTriggerProgrammaticLaunchCompletion): the next pass's blocks would then
// fill the first SMs that drain two deep and leave others empty (256^2 in FP64
// 20.7 -> 30.2 us per step, 2048^2 in FP32 9.9 -> 10.7).
template <typename... P, typename... A>
inline cudaError_t launch_pass(void (*kern)(P...), dim3 grid, int threads, size_t smem,
                               cudaStream_t st, A... args)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kern, P(args)...);
}
#ifdef __CUDACC__
// Every kernel launched by launch_pass calls this before it reads or writes
// what other kernels of the stream write or read.  What comes after is loaded
// coherently (no __ldg, whose loads the compiler may move ahead of this).
__device__ __forceinline__ void pass_wait() { cudaGridDependencySynchronize(); }
#endif

// Per-run coefficients of the face fluxes.  The kernels evaluate unscaled
// face fluxes and apply the constant factors once per cell, so that one
// step reads
//   b' = b + dt theta n b + cA (phiE - phiW + phiN - phiS)
//   n' = n - dt n b       - cG (gE - gW + gN - gS)
// with, on a face between L (left/lower) and R (right/upper),
//   phi = s2 n2 b2 (db + hc b2 dm)          central mobility b_f^2
//   phi = s2 n2 (b2 db + hc b_d^2 dm)       donor-cell mobility b_d^2
//   g   = dm
// where s2 = sL+sR, n2 = nL+nR, b2 = bL+bR, db = bR-bL, dm = nL-nR and b_d
// is b of the lower-n cell.  hc = cChi under the constant law and, under the
// receptor law, cChi / (2+n2)^2 in FP32 and 1 / (cChi (2+n2))^2 in FP64.  Derivation: sigma_f n_f b_f =
// s2 n2 b2 / 8, b_f^2 = b2^2 / 4, so hc = chi(n_f) / 2 (central) or 2 chi(n_f)
// (donor cell), and for the receptor law chi(n_f) = 4 chi0 / (2+n2)^2.
struct Coef {
    double cA;    // dt / (8 dx^2)
    double cChi;  // constant: chi0 / 2; receptor: 2 chi0; donor cell: 4 times
                  // that.  Receptor in FP64: 1 / sqrt of it (kNoChemoF64 at most)
    double cG;    // dt Dn / dx^2
    double cR;    // dt theta
    double cN;    // dt
};

// The FP64 receptor law's largest scale (chi0 = 0, and chi0 below about 1e-39):
// the weight is then at most 2^-128, far below the rounding of any flux, and the
// square of the denominator, 2^128 (2 + n_L + n_R)^2, is finite up to
// n_L + n_R = 2^447.  A larger scale loses that range for nothing (2^500
// overflowed from n_L + n_R = 4094 on, and the reciprocal's correction made
// 0 inf of it).
constexpr double kNoChemoF64 = 0x1p64;

struct Sigma {  // how sigma is obtained
    int per_step;     // 0: read the sigma array; 1: regenerate from Philox every step
    int dist;         // CX_NOISE_*
    double sigma0, amp;
    uint64_t seed;
};

// One launch of the step kernel.  stage 0: u_out = u + dt r(u) (forward
// Euler, or the first Heun stage); stage 1: the second Heun stage,
// u_out = (u0 + u + dt r(u)) / 2 with u0 read pointwise from (bu, nu) and
// written back in place (bo == bu, no == nu).
struct StepArgs {
    const void *b, *n, *s;  // stencil input state (+ sigma array, static noise)
    const void *bu, *nu;    // stage 1: state at the start of the step
    void *bo, *no;          // output state
    int nx, ny;
    long long pitch;        // elements per row
    int law, mob, stage;
    int rows;               // tile height in rows (grid.y = ceil(ny / rows))
    Coef k;
    Sigma sg;
    long long step;         // index of the time step being taken (noise counter)
};

// Launchers (return a cudaError_t from the launch).  recipe 0: FP64 sigma
// recipe, 1: FP32 recipe (per-step noise of an FP32 state).
cudaError_t launch_sigma_init(int prec, void *sigma, int nx, int ny, long long pitch,
                              uint64_t seed, uint64_t step, double sigma0, double amp,
                              int dist, int recipe, cudaStream_t st);
cudaError_t launch_initial_state(int prec, void *b, void *n, int nx, int ny, long long pitch,
                                 double dx, double n0, double bM, double r0sq, cudaStream_t st);
cudaError_t launch_step(int prec, const StepArgs &a, cudaStream_t st);
// Two stages in one pass (cx_fused.cu): heun 0 takes the Euler steps a.step
// and a.step + 1, heun 1 the Heun step a.step; reads (b, n, s), writes
// (bo, no), which must be other buffers.  bu / nu / stage are not used.
cudaError_t launch_fused(int prec, const StepArgs &a, int heun, cudaStream_t st);

// In-row order of the device arrays.  Each aligned group of four cells of a
// row, columns 4g .. 4g+3, is stored as (4g, 4g+2, 4g+1, 4g+3): a 16-byte
// vector load then hands a thread its cells already as the pairs
// (4g, 4g+2) and (4g+1, 4g+3) that the paired FP32 arithmetic works on, with
// no register moves to regroup them (1.05x on the 16384^2 FP32 pass).  The
// order swaps the middle two of each group, so it is its own inverse.  Rows
// therefore need a pitch that is a multiple of 4 elements; a row's last
// group may hold a cell beyond nx in the padding columns.
__host__ __device__ __forceinline__ long long pair_col(long long i)
{
    return (i & ~3LL) | ((i & 1LL) << 1) | ((i >> 1) & 1LL);
}
// Swaps the middle two elements of every group of four of the first
// ceil(nx/4)*4 columns of each row, in place: converts an array between the
// natural in-row order and the pair order (either way).
cudaError_t launch_pair_order(int prec, void *a, int nx, int ny, long long pitch, cudaStream_t st);

// The address under which a kernel may write the `count` elements of `elem`
// bytes at `host`, or nullptr unless all of them are pinned and aligned to
// their size (cx_read.cu).
void *pinned_view(void *host, size_t count, size_t elem);
// A field in pair order -> packed rows of nx elements in natural order and of
// type `dtype` (CX_F64 / CX_F32) at `dst`, device or pinned host memory.
cudaError_t launch_read_field(int prec, const void *field, int nx, int ny, long long pitch, void *dst,
                              int dtype, cudaStream_t st);

struct DiagScratch {
    double *partials;  // [blocks][8]
    double *result;    // [8], device or pinned host memory
    int blocks;
};
int diag_blocks_for(int ny);
// pair_order: the fields are in the library's pair order (else natural).
cudaError_t launch_diagnostics(int prec, const void *b, const void *n, int nx, int ny,
                               long long pitch, double b_threshold, DiagScratch s,
                               cudaStream_t st, bool pair_order = true);

// b on a circle of `radius` about the domain centre, ns samples (cx_labels.cu).
cudaError_t launch_polar(int prec, const void *b, int nx, int ny, long long pitch, double dx,
                         double radius, int ns, double *out, cudaStream_t st);

// Store `msg` as this thread's cx_last_error() text; returns `code`.
int record_error(int code, const char *msg);

// Host helpers shared by the single-grid and batch entry points
// (cx_api.cu): parameter validation, the time step (CX_ERR_DT_UNSTABLE
// above the limit), the scaled flux coefficients and the envelope level.
int validate_params(const cx_grid *g, const cx_params *p);
int resolve_time_step(const cx_grid *g, const cx_params *p, double *dt);
Coef make_coef(const cx_grid &g, const cx_params &p, double dt);
double envelope_level(const cx_params &p);
double march_us(double cells, bool heun, bool per_step);

// Batched stepping and diagnostics (cx_batch.cu).  `inst` is the device
// instance table, `work` the device work list (int4: instance, tile x,
// tile y, unused).
size_t inst_dev_bytes(int prec);
void fill_inst(int prec, void *table, int i, void *b0, void *b1, void *n0, void *n1, void *s,
               int nx, int ny, long long pitch, const Coef &k, double bth, uint64_t seed,
               double sigma0, double amp, int dist);
// Per-step noise of a batch pass: on = 1 redraws sigma every step; the
// pass's first time step is *step_base + step_off (step_base: device int64
// written by launch_set_step before the pass or the graph holding it).
struct BatchNoise {
    int on;
    const long long *step_base;
    int step_off;
};
cudaError_t launch_set_step(long long *step_base, long long step, cudaStream_t st);
cudaError_t launch_batch_step(int prec, int law, int mob, const void *inst, const int4 *work,
                              int nwork, int parity, int rows, int stage, const BatchNoise &nz,
                              cudaStream_t st);
// Two stages per pass over a 480-column work list: reads u(parity), writes
// u(parity^1); heun 0: two Euler steps, 1: one Heun step.
cudaError_t launch_batch_fused(int prec, int law, int mob, const void *inst, const int4 *work,
                               int nwork, int parity, int rows, int heun, const BatchNoise &nz,
                               cudaStream_t st);
cudaError_t launch_batch_diag(int prec, const void *inst, int first, int count, int blocks,
                              int parity, double *part, double *out, cudaStream_t st);
// nsteps steps of the work items [0, nwork) in one cooperative launch with
// a bounded grid barrier between steps; `barrier` is a device block of
// grid_barrier_bytes() whose first 8 bytes must be zero at launch and whose
// int at offset 8 becomes non-zero if a wait ran out.
size_t grid_barrier_bytes();
cudaError_t launch_batch_resident(int prec, int law, int mob, const void *inst, const int4 *work,
                                  int nwork, int parity, int rows, int nsteps, int heun,
                                  void *barrier, long long spin_limit, const BatchNoise &nz,
                                  cudaStream_t st);

// A pass of the register-tile kernel (cx_tile.cu; FP32): `steps` time steps on
// tiles of 4 lx columns and (threads / lx) r rows that overlap by the halo
// that the pass's stages need.
struct TilePlan {
    int steps, lx, r, threads;
    bool heun;
    int stages() const { return heun ? 2 * steps : steps; }
    int width() const { return 4 * lx; }
    int height() const { return threads / lx * r; }
    int halo_x() const { return (stages() + 3) / 4 * 4; }  // whole groups of four cells
    int halo_y() const { return stages(); }
};
// Tiles along a side of n cells; the first and the last lie against the walls
// and need no halo there.  0: tiles of this size keep no cell of such a side.
__host__ __device__ inline int tile_count(int n, int size, int halo)
{
    const int step = size - 2 * halo;
    if (n <= size) return 1;
    return step <= 0 ? 0 : 1 + (n - size + step - 1) / step;
}
inline int tiles_x(int nx, const TilePlan &p) { return tile_count(nx, p.width(), p.halo_x()); }
inline int tiles_y(int ny, const TilePlan &p) { return tile_count(ny, p.height(), p.halo_y()); }
// How many row times of two warps sharing an FP64 unit a round-robin of
// `blocks` one-warp blocks over `units` units takes per row (cx_api.cu,
// auto_tile_rows_f64).
inline double f64_rounds(long long blocks, long long units)
{
    const long long q = (blocks + units - 1) / units;
    return q == 1 ? 1.4 : (double)q;
}
struct TileGrid {
    int nx, ny, count;  // `count` grids of this size
};
double plan_tiles(const TileGrid *grids, int count, int sms, bool heun, bool per_step,
                  long long steps, TilePlan *best);
// The tiles of a pass over a batch, in the kernel's parameters: the instances, in
// the order of their area, lie in n runs, each instance of a run with `tiles`
// blocks, `across` of them side by side; the run's blocks start at `first`
// (run[n].first: all blocks), its instances at `place` of the table.
// Block i << shift belongs to run index[i].  A run is one size (up to 224 of
// them), or a few sizes of similar area (across 0), whose smaller instances
// leave some of their blocks idle.  A list in device memory would have to be
// allocated for every length of a pass, and kept as long as any captured launch
// that reads it.  Lists and runs: 20 strips of 400 cells, 1000 steps and 40
// reads, 1423 and 1406 us; 512 steps of 96 instances of 256^2 6905 and 6925 us, of
// 40 of 300^2 with Heun 10808 and 10921 (other register spills); 256 steps of 129
// different grids of up to 311 x 149 1224 and 1240, of 300 such grids 2629 and
// 2743.  The parameters stay below 4 KB: beyond that a launch takes the host 5-8
// us longer.
constexpr int kTileRuns = 224, kTileIndex = 64;
struct TileRun {
    int first, tiles, place, across;
};
struct TileRuns {
    int n, shift;
    TileRun run[kTileRuns + 1];
    unsigned short index[kTileIndex + 1];
};
// Whether a side of n cells needs tile i: the tile before it ends short of the
// wall.
__host__ __device__ inline bool tile_needed(int i, int n, int size, int halo)
{
    return i == 0 || (i - 1) * (size - 2 * halo) + size < n;
}
// What a pass runs on: one grid (law, mobility and stage of the arguments not
// used), or instances of a batch.
struct TileLaunch {
    const StepArgs *grid;
    const void *inst;  // the instance table in the order of the runs
    const TileRuns *runs;
    int parity;
    BatchNoise nz;
};
cudaError_t launch_tile(int law, int mob, bool per_step, const TileLaunch &a, const TilePlan &p,
                        cudaStream_t st);
// The same for FP64 strips with a static sigma (cx_strip.cu); *march: the
// march's modelled time per step.
double plan_strips(const TileGrid *grids, int count, int sms, int law, bool heun, long long steps,
                   TilePlan *best, double *march);
cudaError_t launch_strip(int law, int mob, const TileLaunch &a, const TilePlan &p, cudaStream_t st);

}  // namespace cx

struct cx_ctx {
    cx_grid g;
    cx_params p;
    uint64_t seed;
    int prec;             // CX_PREC_*
    size_t elem;          // bytes per element
    long long pitch;      // elements per row (rows 128-byte aligned)
    void *b[2], *n[2];    // ping-pong state
    void *sigma;
    int own_fields;       // 1: b, n, sigma allocated (and freed) by the library
    int cur;              // index of the buffer holding the current state
    int64_t step;
    double dt;
    cudaStream_t stream;
    int device;
    int num_sms;          // streaming multiprocessors of that device
    int tile_rows;        // rows per step-kernel tile (0: automatic)
    int time_block;       // explicit stages per pass over the grid (1 or 2)
    int depth_set;        // time_block was chosen by cx_set_time_block
    int64_t plan_for;     // cx_step's n_steps that `plan` was made for (0: none yet)
    int plan_tiles;       // that call runs on register tiles
    cx::TilePlan plan;
    cx::DiagScratch diag;
    double *h_diag;       // pinned [8]
    // staged uploads (cx_stage_state / cx_commit_state), created on first use
    void *stage_b, *stage_n;    // device staging arrays, library-owned, same pitch
    cudaStream_t copy_stream;   // the staged host-to-device copies
    cudaEvent_t staged;         // recorded after the staged copies
    cudaEvent_t stage_free;     // recorded once the compute stream is done with the staging arrays
    int stage_pending;          // a staged upload awaits cx_commit_state
    int stage_free_valid;       // stage_free has been recorded
};
