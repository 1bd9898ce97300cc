// cx_batch_api.cu -- the cx_batch_* entry points (include/cx.h): a set of
// independent simulations (one parameter sweep) stepped together by the
// batched kernels of cx_batch.cu.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <new>
#include <utility>
#include <vector>

#include "cx_internal.h"

namespace {

int bfail(int code, const char *msg) { return cx::record_error(code, msg); }

int bcuda(cudaError_t e, const char *what)
{
    char buf[300];
    snprintf(buf, sizeof buf, "%s: %s", what, cudaGetErrorString(e));
    return cx::record_error(e == cudaErrorMemoryAllocation ? CX_ERR_OOM : CX_ERR_CUDA, buf);
}

#define BX_CUDA(call, what)                                  \
    do {                                                     \
        cudaError_t e_ = (call);                             \
        if (e_ != cudaSuccess) return bcuda(e_, (what));     \
    } while (0)

// columns per tile of the one-stage march: 128 threads (FP32) or 32 (FP64) x 4 cells
int tile_cols(int prec) { return prec == CX_PREC_F64 ? 128 : 512; }
constexpr int kFusedTileCols = 120;  // written columns per (one-warp) tile of the two-stage march
constexpr int kDiagBlocksPerInst = 64;

size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

}  // namespace

struct cx_batch {
    int count = 0, prec = 0, law = 0, mob = 0, scheme = 0;
    int noise = 0;                  // 1: sigma redrawn every step (CX_NOISE_PER_STEP)
    long long *d_step = nullptr;    // time step the next pass starts from (noise == 1)
    std::vector<cx_grid> g;
    std::vector<cx_params> p;
    std::vector<uint64_t> seed;
    std::vector<double> dt;
    std::vector<long long> pitch;
    std::vector<void *> fb[2], fn[2], fs;
    std::vector<long long> footprint;  // device bytes of each instance's fields
    void *arena = nullptr;
    size_t elem = 4;
    void *d_inst = nullptr;
    std::vector<unsigned char> h_inst;
    int4 *d_work = nullptr;       // tile_cols() tiles (one stage per pass)
    std::vector<int> work_begin;  // first work item of each instance (+ total)
    int4 *d_work2 = nullptr;      // 120-column tiles (two stages per pass)
    std::vector<int> work2_begin;
    int rows = 32;                  // tile height set, or reported as the default
    int march_rows = 32;            // tile height in effect
    bool tuned = false;             // a knob of the marches was set: they run as told
    int num_sms = 1;
    std::vector<cx::TileGrid> sizes;  // the instances' distinct sizes
    int64_t plan_for = 0;           // steps that `plan` was made for (0: none yet)
    bool tiles = false;             // passes run on register tiles
    cx::TilePlan plan{};
    void *d_by_size = nullptr;      // the instance table, size by size as in `sizes`
    int graph_steps = 64;
    long long group_bytes = 0;
    int time_block = 1;             // explicit stages per pass (1 or 2)
    std::vector<int> group_first;  // instance index where each group starts (+ count)
    std::vector<cudaGraphExec_t> gexec[2];  // per group, by starting parity
    std::vector<int> gend[2];               // parity after that graph
    int resident_steps = 0;         // > 0: steps per cooperative launch of a group
    void *d_barrier = nullptr;      // grid barrier state of the resident kernel
    long long spin_limit = 1 << 22; // polls before a barrier wait gives up
    int cur = 0;
    int64_t step = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    double *d_part = nullptr, *h_res = nullptr;  // h_res: pinned, written by the diagnostics kernel
};

namespace {

void drop_graphs(cx_batch *B)
{
    for (int p = 0; p < 2; ++p) {
        for (auto &e : B->gexec[p])
            if (e) cudaGraphExecDestroy(e);
        B->gexec[p].clear();
        B->gend[p].clear();
    }
}

void free_batch(cx_batch *B)
{
    if (!B) return;
    if (B->stream) cudaStreamSynchronize(B->stream);
    drop_graphs(B);
    if (B->arena) cudaFree(B->arena);
    if (B->d_inst) cudaFree(B->d_inst);
    if (B->d_work) cudaFree(B->d_work);
    if (B->d_work2) cudaFree(B->d_work2);
    if (B->d_by_size) cudaFree(B->d_by_size);
    if (B->d_part) cudaFree(B->d_part);
    if (B->h_res) cudaFreeHost(B->h_res);
    if (B->d_barrier) cudaFree(B->d_barrier);
    if (B->d_step) cudaFree(B->d_step);
    if (B->own_stream && B->stream) cudaStreamDestroy(B->stream);
    delete B;
}

// A host table to the device, complete when the call returns: the passes, on
// this stream, may read it before they wait for the kernels ahead of them.
cudaError_t upload(cx_batch *B, void *dst, const void *src, size_t bytes)
{
    const cudaError_t e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, B->stream);
    return e == cudaSuccess ? cudaStreamSynchronize(B->stream) : e;
}

// Tile work lists for tiles of `rows` rows, instance by instance: the one-stage
// march's tiles and the two-stage march's 120-column tiles.  If one cannot be
// made, the height and the lists in effect stay.
int build_work(cx_batch *B, int rows)
{
    int4 *d[2] = {nullptr, nullptr};
    std::vector<int> begin[2];
    cudaError_t e = cudaSuccess;
    for (int f = 0; f < 2 && e == cudaSuccess; ++f) {
        const int cols = f ? kFusedTileCols : tile_cols(B->prec);
        std::vector<int4> w;
        begin[f].assign(B->count + 1, 0);
        for (int i = 0; i < B->count; ++i) {
            begin[f][i] = (int)w.size();
            const int tx = (B->g[i].nx + cols - 1) / cols;
            const int ty = (B->g[i].ny + rows - 1) / rows;
            for (int y = 0; y < ty; ++y)
                for (int x = 0; x < tx; ++x) w.push_back(make_int4(i, x, y, 0));
        }
        begin[f][B->count] = (int)w.size();
        e = cudaMalloc((void **)&d[f], w.size() * sizeof(int4));
        if (e == cudaSuccess) e = upload(B, d[f], w.data(), w.size() * sizeof(int4));
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        for (int4 *p : d)
            if (p) cudaFree(p);
        return bcuda(e, "tile work lists");
    }
    if (B->d_work) cudaFree(B->d_work);
    if (B->d_work2) cudaFree(B->d_work2);
    B->d_work = d[0];
    B->d_work2 = d[1];
    B->work_begin.swap(begin[0]);
    B->work2_begin.swap(begin[1]);
    B->march_rows = rows;
    return CX_OK;
}

// Tile height of a batch that has not been tuned, in place of the default
// (B->rows).  FP32 (two-stage march, 16 one-warp tiles per SM at a time): the
// least height at which one round of tiles covers the batch if that is below
// 72, else 64 rows: a round that is barely exceeded costs nearly two (16
// instances of 1024^2: 60 rows, 1.07 rounds, 44.0 us per step; 64 rows, 0.95,
// 36.9), and from there on 64 rows fill the rounds better than 128 (24
// instances of 512^2 .. 2048^2 98.6 -> 87.7 us per step, 128 of them 431 -> 417,
// 64 of 1024^2 133 -> 125).  FP64: the height that a single grid would take.
int auto_rows(const cx_batch *B)
{
    if (B->prec == CX_PREC_F32) {
        const long long slots = 16LL * B->num_sms;
        for (int r = 8; r < 72; ++r) {
            long long tiles = 0;
            for (const cx::TileGrid &s : B->sizes)
                tiles += (long long)s.count * ((s.nx + kFusedTileCols - 1) / kFusedTileCols) *
                         ((s.ny + r - 1) / r);
            if (tiles <= slots) return r;
        }
        return 64;
    }
    const long long cols = tile_cols(B->prec), units = 4LL * B->num_sms;
    long long best = 1;
    double cost = 0.0;
    for (long long r = 1; r <= B->rows; ++r) {
        long long tiles = 0;
        for (const cx::TileGrid &s : B->sizes)
            tiles += (s.nx + cols - 1) / cols * ((s.ny + r - 1) / r) * s.count;
        const double now = cx::f64_rounds(tiles, units) * ((double)r + 0.5);
        if (cost == 0.0 || now <= cost) {
            cost = now;
            best = r;
        }
    }
    return (int)best;
}

void build_groups(cx_batch *B);

int default_rows(int prec) { return prec == CX_PREC_F32 ? 128 : 32; }
int default_time_block(int prec) { return prec == CX_PREC_F32 ? 2 : 1; }  // as a single grid

int even_for_euler(const cx_batch *B, int graph_steps)
{
    return B->scheme == CX_SCHEME_EULER && (graph_steps & 1) ? graph_steps + 1 : graph_steps;
}

// After a knob was set (`tuned`) or all were given back: the height in effect,
// and the marches' work lists.
int apply_tuning(cx_batch *B, bool tuned)
{
    B->tuned = tuned;
    B->plan_for = 0;
    B->tiles = false;
    build_groups(B);
    const int rows = tuned ? B->rows : auto_rows(B);
    return rows == B->march_rows ? CX_OK : build_work(B, rows);
}

// Whether runs of `steps` steps take several steps per pass, as a single grid
// does: an untuned batch on register tiles (FP32) or strips (FP64, every
// instance one row high, static sigma), where they are modelled to be faster.
bool use_tiles(cx_batch *B, int64_t steps)
{
    if (B->tuned) return false;
    if (B->plan_for != steps) {
        const bool heun = B->scheme == CX_SCHEME_HEUN, per_step = B->noise != 0;
        const cx::TileGrid *sizes = B->sizes.data();
        const int ns = (int)B->sizes.size();
        double us = HUGE_VAL, march = 0.0;
        if (B->prec == CX_PREC_F32) {
            us = cx::plan_tiles(sizes, ns, B->num_sms, heun, per_step, steps, &B->plan);
            double cells = 0.0;  // computed by the march, halo rows and idle columns included
            for (const cx::TileGrid &s : B->sizes)
                cells += (double)s.count * ((s.nx + kFusedTileCols - 1) / kFusedTileCols * kFusedTileCols) *
                         s.ny * (B->march_rows + 2) / B->march_rows;
            march = cx::march_us(cells, heun, per_step);
        } else if (!per_step && std::all_of(B->sizes.begin(), B->sizes.end(),
                                            [](const cx::TileGrid &s) { return s.ny == 1; })) {
            us = cx::plan_strips(sizes, ns, B->num_sms, B->law, heun, steps, &B->plan, &march);
        }
        B->tiles = us < march;
        B->plan_for = steps;
    }
    return B->tiles;
}

// The steps that a call of n_steps plans for: a graph's if it replays one (and
// the rest by the same plan).
int64_t run_length(const cx_batch *B, int64_t n_steps)
{
    return B->graph_steps > 0 && n_steps >= B->graph_steps ? B->graph_steps : n_steps;
}

// Steps of the next register-tile pass of `left`: as few passes as the plan
// allows, of equal length.
int tile_pass_steps(const cx_batch *B, int64_t left)
{
    const int64_t passes = (left + B->plan.steps - 1) / B->plan.steps;
    return (int)((left + passes - 1) / passes);
}

// Consecutive groups of instances whose fields fit group_bytes (one group
// with every instance when group_bytes == 0; an instance larger than the
// budget forms a group of its own).
void build_groups(cx_batch *B)
{
    B->group_first.clear();
    long long acc = 0;
    for (int i = 0; i < B->count; ++i) {
        if (i == 0 || (B->group_bytes > 0 && acc + B->footprint[i] > B->group_bytes)) {
            B->group_first.push_back(i);
            acc = 0;
        }
        acc += B->footprint[i];
    }
    B->group_first.push_back(B->count);
}

// The noise argument of a pass whose first time step is step_off after the
// step last written to d_step.
cx::BatchNoise pass_noise(const cx_batch *B, int step_off)
{
    return cx::BatchNoise{B->noise, B->d_step, step_off};
}

// Before the passes (or the graph) that start at time step `step`: where the
// per-step noise reads its step from.
cudaError_t mark_step(cx_batch *B, int64_t step)
{
    return B->noise ? cx::launch_set_step(B->d_step, (long long)step, B->stream) : cudaSuccess;
}

// One time step of instances [i0, i1) at the given parity, step_off steps
// after the marked step.
cudaError_t one_step(cx_batch *B, int i0, int i1, int parity, int step_off)
{
    const int w0 = B->work_begin[i0], w1 = B->work_begin[i1];
    const int4 *work = B->d_work + w0;
    const cx::BatchNoise nz = pass_noise(B, step_off);
    cudaError_t e = cx::launch_batch_step(B->prec, B->law, B->mob, B->d_inst, work, w1 - w0,
                                          parity, B->march_rows, 0, nz, B->stream);
    if (e == cudaSuccess && B->scheme == CX_SCHEME_HEUN)
        e = cx::launch_batch_step(B->prec, B->law, B->mob, B->d_inst, work, w1 - w0, parity,
                                  B->march_rows, 1, nz, B->stream);
    return e;
}

// The runs of the batch's instances for passes of `plan`.
void fill_runs(const cx_batch *B, const cx::TilePlan &plan, cx::TileRuns *z)
{
    const size_t sizes = B->sizes.size();
    z->n = (int)std::min<size_t>(sizes, cx::kTileRuns);
    int place = 0, first = 0;
    for (int k = 0; k < z->n; ++k) {
        const size_t s0 = sizes * k / z->n, s1 = sizes * (k + 1) / z->n;
        cx::TileRun r{first, 0, place, s1 - s0 == 1 ? cx::tiles_x(B->sizes[s0].nx, plan) : 0};
        for (size_t i = s0; i < s1; ++i) {
            const cx::TileGrid &g = B->sizes[i];
            r.tiles = std::max(r.tiles, cx::tiles_x(g.nx, plan) * cx::tiles_y(g.ny, plan));
            place += g.count;
        }
        first += r.tiles * (place - r.place);
        z->run[k] = r;
    }
    z->run[z->n] = cx::TileRun{first, 0, place, 0};
    z->shift = 0;
    while (first > ((long long)cx::kTileIndex << z->shift)) ++z->shift;
    for (int i = 0, k = 0; i <= cx::kTileIndex; ++i) {
        const long long blk = std::min<long long>(first - 1, (long long)i << z->shift);
        while (z->run[k + 1].first <= blk) ++k;
        z->index[i] = (unsigned short)k;
    }
}

// One pass of `steps` steps over every instance on register tiles or strips
// (an untuned batch has one group).
cudaError_t tile_pass(cx_batch *B, int parity, int steps, int step_off)
{
    cx::TilePlan plan = B->plan;
    plan.steps = steps;
    cx::TileRuns runs{};
    fill_runs(B, plan, &runs);
    cx::TileLaunch a{};
    a.inst = B->d_by_size;
    a.runs = &runs;
    a.parity = parity;
    a.nz = pass_noise(B, step_off);
    return B->prec == CX_PREC_F64 ? cx::launch_strip(B->law, B->mob, a, plan, B->stream)
                                  : cx::launch_tile(B->law, B->mob, B->noise != 0, a, plan, B->stream);
}

int next_parity(const cx_batch *B, int parity) { return B->scheme == CX_SCHEME_HEUN ? parity : parity ^ 1; }

// One pass over instances [i0, i1) starting at *parity, step_off steps
// after the marked step: two stages when the depth is 2 (two Euler steps if
// at least two are left, or one Heun step), else one step.  Sets *steps to
// the time steps taken and *parity to the parity after them.
cudaError_t one_pass(cx_batch *B, int i0, int i1, int *parity, int64_t left, int step_off,
                     int *steps)
{
    const bool heun = B->scheme == CX_SCHEME_HEUN;
    if (B->tiles) {
        *steps = tile_pass_steps(B, left);
        const cudaError_t e = tile_pass(B, *parity, *steps, step_off);
        *parity ^= 1;
        return e;
    }
    if (B->time_block == 2 && (heun || left >= 2)) {
        const int w0 = B->work2_begin[i0], w1 = B->work2_begin[i1];
        const cudaError_t e = cx::launch_batch_fused(B->prec, B->law, B->mob, B->d_inst,
                                                     B->d_work2 + w0, w1 - w0, *parity, B->march_rows,
                                                     heun ? 1 : 0, pass_noise(B, step_off),
                                                     B->stream);
        *parity ^= 1;
        *steps = heun ? 1 : 2;
        return e;
    }
    const cudaError_t e = one_step(B, i0, i1, *parity, step_off);
    *parity = next_parity(B, *parity);
    *steps = 1;
    return e;
}

// Capture graph_steps steps of group gi starting at `parity`; *end gets the
// parity after them (a graph is kept per starting parity).
int capture_group(cx_batch *B, int gi, int parity, cudaGraphExec_t *out, int *end)
{
    cudaGraph_t graph = nullptr;
    BX_CUDA(cudaStreamBeginCapture(B->stream, cudaStreamCaptureModeThreadLocal), "graph capture begin");
    cudaError_t e = cudaSuccess;
    int par = parity;
    for (int64_t left = B->graph_steps; left > 0 && e == cudaSuccess;) {
        int taken = 1;
        e = one_pass(B, B->group_first[gi], B->group_first[gi + 1], &par, left,
                     (int)(B->graph_steps - left), &taken);
        left -= taken;
    }
    cudaError_t e2 = cudaStreamEndCapture(B->stream, &graph);
    if (e != cudaSuccess) return bcuda(e, "launch during graph capture");
    if (e2 != cudaSuccess) return bcuda(e2, "graph capture end");
    e = cudaGraphInstantiate(out, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return bcuda(e, "graph instantiate");
    *end = par;
    return CX_OK;
}

int check_batch(const cx_batch *B)
{
    if (!B) return bfail(CX_ERR_INVALID_ARG, "NULL batch");
    return CX_OK;
}

// After the stream has drained: did a resident launch's barrier wait run
// out?  The flag is cleared once reported.
int check_barrier(cx_batch *B)
{
    int err = 0;
    BX_CUDA(cudaMemcpy(&err, (char *)B->d_barrier + 8, sizeof err, cudaMemcpyDeviceToHost),
            "barrier flag read");
    if (err) {
        BX_CUDA(cudaMemsetAsync((char *)B->d_barrier + 8, 0, sizeof err, B->stream), "barrier flag reset");
        return bfail(CX_ERR_TIMEOUT, "a grid barrier wait of the resident batch kernel ran out; "
                                     "the batch state is undefined");
    }
    return CX_OK;
}

// `left` steps of instances [i0, i1), the first of them time step `step`,
// by cooperative launches of resident_steps steps each; returns the parity
// after them.
int run_resident(cx_batch *B, int i0, int i1, int par, int64_t left, int64_t step, int *par_out)
{
    const int w0 = B->work_begin[i0], w1 = B->work_begin[i1];
    while (left > 0) {
        const int chunk = (int)(left < B->resident_steps ? left : B->resident_steps);
        BX_CUDA(cudaMemsetAsync(B->d_barrier, 0, 8, B->stream), "barrier reset");
        BX_CUDA(mark_step(B, step), "step mark");
        BX_CUDA(cx::launch_batch_resident(B->prec, B->law, B->mob, B->d_inst, B->d_work + w0, w1 - w0,
                                          par, B->march_rows, chunk, B->scheme == CX_SCHEME_HEUN,
                                          B->d_barrier, B->spin_limit, pass_noise(B, 0), B->stream),
                "resident batch launch");
        step += chunk;
        if (B->scheme == CX_SCHEME_EULER && (chunk & 1)) par ^= 1;
        left -= chunk;
    }
    *par_out = par;
    return CX_OK;
}

}  // namespace

extern "C" {

int cx_batch_create(int32_t count, const cx_grid *grids, const cx_params *params,
                    const uint64_t *seeds, cx_batch **out)
{
    if (!out) return bfail(CX_ERR_INVALID_ARG, "out must not be NULL");
    *out = nullptr;
    if (count < 1 || count > 65535) return bfail(CX_ERR_INVALID_ARG, "count must lie in 1..65535");
    if (!grids || !params || !seeds) return bfail(CX_ERR_INVALID_ARG, "grids, params and seeds must not be NULL");
    for (int i = 0; i < count; ++i) {
        int rc = cx::validate_params(&grids[i], &params[i]);
        if (rc) return rc;
        const cx_params &a = params[i], &z = params[0];
        if (a.precision != z.precision || a.scheme != z.scheme || a.chemo_law != z.chemo_law ||
            a.mobility != z.mobility || a.noise_mode != z.noise_mode)
            return bfail(CX_ERR_INVALID_ARG, "all instances of a batch must share precision, "
                                             "scheme, chemo_law, mobility and noise_mode");
    }
    cx_batch *B = new (std::nothrow) cx_batch;
    if (!B) return bfail(CX_ERR_OOM, "host allocation of the batch failed");
    B->count = count;
    B->prec = params[0].precision;
    B->law = params[0].chemo_law;
    B->mob = params[0].mobility;
    B->scheme = params[0].scheme;
    B->noise = params[0].noise_mode == CX_NOISE_PER_STEP ? 1 : 0;
    B->time_block = default_time_block(B->prec);
    // Two stages per pass recompute 4 halo rows per tile: 128-row tiles keep
    // that to 3 % (1024 instances of 1024^2: 5.6e11 cell-updates/s against
    // 4.6e11 with 32-row tiles; 64 to 256 rows within 2 % of the best)
    B->rows = default_rows(B->prec);
    B->elem = B->prec == CX_PREC_F64 ? sizeof(double) : sizeof(float);
    B->g.assign(grids, grids + count);
    B->p.assign(params, params + count);
    B->seed.assign(seeds, seeds + count);
    B->dt.resize(count);
    for (int i = 0; i < count; ++i) {
        int rc = cx::resolve_time_step(&grids[i], &params[i], &B->dt[i]);
        if (rc) { free_batch(B); return rc; }
    }
    // arena layout
    const long long align = 128 / (long long)B->elem;
    std::vector<size_t> off(5 * (size_t)count);
    size_t total = 0;
    B->pitch.resize(count);
    B->footprint.resize(count);
    for (int i = 0; i < count; ++i) {
        B->pitch[i] = ((long long)grids[i].nx + align - 1) / align * align;
        const size_t bytes = round_up((size_t)B->pitch[i] * grids[i].ny * B->elem, 256);
        for (int a = 0; a < 5; ++a) {
            off[5 * i + a] = total;
            total += bytes;
        }
        B->footprint[i] = (long long)(5 * bytes);
    }
    cudaError_t e = cudaStreamCreateWithFlags(&B->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) { free_batch(B); return bcuda(e, "stream creation"); }
    B->own_stream = true;
    e = cudaMalloc(&B->arena, total);
    if (e == cudaSuccess) e = cudaMemsetAsync(B->arena, 0, total, B->stream);
    if (e != cudaSuccess) { cudaGetLastError(); free_batch(B); return bcuda(e, "arena allocation"); }
    for (int q = 0; q < 2; ++q) {
        B->fb[q].resize(count);
        B->fn[q].resize(count);
    }
    B->fs.resize(count);
    char *base = (char *)B->arena;
    for (int i = 0; i < count; ++i) {
        B->fb[0][i] = base + off[5 * i + 0];
        B->fb[1][i] = base + off[5 * i + 1];
        B->fn[0][i] = base + off[5 * i + 2];
        B->fn[1][i] = base + off[5 * i + 3];
        B->fs[i] = base + off[5 * i + 4];
    }
    // instance table
    const size_t isz = cx::inst_dev_bytes(B->prec);
    B->h_inst.assign(isz * count, 0);
    for (int i = 0; i < count; ++i)
        cx::fill_inst(B->prec, B->h_inst.data(), i, B->fb[0][i], B->fb[1][i], B->fn[0][i],
                      B->fn[1][i], B->fs[i], grids[i].nx, grids[i].ny, B->pitch[i],
                      cx::make_coef(grids[i], params[i], B->dt[i]), cx::envelope_level(params[i]),
                      seeds[i], params[i].sigma0, params[i].noise_amp, params[i].noise_dist);
    e = cudaMalloc(&B->d_inst, B->h_inst.size());
    if (e == cudaSuccess) e = upload(B, B->d_inst, B->h_inst.data(), B->h_inst.size());
    if (e == cudaSuccess) e = cudaMalloc((void **)&B->d_part, 8 * sizeof(double) * (size_t)count * kDiagBlocksPerInst);
    if (e == cudaSuccess) e = cudaMallocHost((void **)&B->h_res, 8 * sizeof(double) * (size_t)count);
    if (e == cudaSuccess) e = cudaMalloc(&B->d_barrier, cx::grid_barrier_bytes());
    if (e == cudaSuccess) e = cudaMemsetAsync(B->d_barrier, 0, cx::grid_barrier_bytes(), B->stream);
    if (e == cudaSuccess && B->noise) e = cudaMalloc((void **)&B->d_step, sizeof(long long));
    if (e == cudaSuccess && B->noise) e = cudaMemsetAsync(B->d_step, 0, sizeof(long long), B->stream);
    // the instances by area, then by width
    std::map<std::pair<long long, int>, std::vector<int>> sizes;
    for (int i = 0; i < count; ++i)
        sizes[{(long long)grids[i].nx * grids[i].ny, grids[i].nx}].push_back(i);
    std::vector<unsigned char> by_size;
    for (const auto &z : sizes) {
        const cx_grid &g = grids[z.second[0]];
        B->sizes.push_back(cx::TileGrid{g.nx, g.ny, (int)z.second.size()});
        for (int i : z.second)
            by_size.insert(by_size.end(), B->h_inst.begin() + isz * i, B->h_inst.begin() + isz * (i + 1));
    }
    if (e == cudaSuccess) e = cudaMalloc(&B->d_by_size, by_size.size());
    if (e == cudaSuccess) e = upload(B, B->d_by_size, by_size.data(), by_size.size());
    if (e != cudaSuccess) { cudaGetLastError(); free_batch(B); return bcuda(e, "batch tables"); }
    if (const char *s = getenv("CX_BARRIER_SPIN_LIMIT")) B->spin_limit = atoll(s);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&B->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        B->num_sms < 1) {
        cudaGetLastError();
        B->num_sms = 1;  // only the choice of tiles uses it
    }
    int rc = build_work(B, auto_rows(B));
    if (rc) { free_batch(B); return rc; }
    build_groups(B);
    // initial state of every instance
    for (int i = 0; i < count && e == cudaSuccess; ++i) {
        const cx_params &a = params[i];
        e = cx::launch_sigma_init(B->prec, B->fs[i], grids[i].nx, grids[i].ny, B->pitch[i], seeds[i],
                                  0, a.sigma0, a.noise_amp, a.noise_dist, 0, B->stream);
        if (e == cudaSuccess)
            e = cx::launch_initial_state(B->prec, B->fb[0][i], B->fn[0][i], grids[i].nx, grids[i].ny,
                                         B->pitch[i], grids[i].dx, a.n0, a.bM, a.r0sq, B->stream);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(B->stream);
    if (e != cudaSuccess) { free_batch(B); return bcuda(e, "batch initialisation"); }
    *out = B;
    return CX_OK;
}

void cx_batch_destroy(cx_batch *B) { free_batch(B); }

int cx_batch_set_stream(cx_batch *B, void *stream)
{
    int rc = check_batch(B);
    if (rc) return rc;
    if (!stream) return bfail(CX_ERR_INVALID_ARG, "a batch needs a non-default stream (graph capture)");
    BX_CUDA(cudaStreamSynchronize(B->stream), "synchronize old stream");
    if (B->own_stream) cudaStreamDestroy(B->stream);
    B->own_stream = false;
    B->stream = (cudaStream_t)stream;
    return CX_OK;
}

int cx_batch_set_tuning(cx_batch *B, int32_t tile_rows, int32_t graph_steps, int64_t group_bytes,
                        int32_t resident_steps)
{
    int rc = check_batch(B);
    if (rc) return rc;
    if (tile_rows < 1 || tile_rows > 4096 || graph_steps < 0 || graph_steps > 100000 ||
        group_bytes < 0 || resident_steps < 0 || resident_steps > 1000000)
        return bfail(CX_ERR_INVALID_ARG, "tile_rows 1..4096, graph_steps 0..100000, group_bytes >= 0, "
                                         "resident_steps 0..1000000");
    BX_CUDA(cudaStreamSynchronize(B->stream), "synchronize before retuning");
    drop_graphs(B);
    B->rows = tile_rows;
    B->graph_steps = even_for_euler(B, graph_steps);
    B->group_bytes = group_bytes;
    B->resident_steps = resident_steps;
    return apply_tuning(B, true);
}

int cx_batch_reset_tuning(cx_batch *B, int32_t graph_steps)
{
    int rc = check_batch(B);
    if (rc) return rc;
    if (graph_steps < 0 || graph_steps > 100000) return bfail(CX_ERR_INVALID_ARG, "graph_steps 0..100000");
    BX_CUDA(cudaStreamSynchronize(B->stream), "synchronize before retuning");
    drop_graphs(B);
    B->rows = default_rows(B->prec);
    B->time_block = default_time_block(B->prec);
    B->graph_steps = even_for_euler(B, graph_steps);
    B->group_bytes = 0;
    B->resident_steps = 0;
    return apply_tuning(B, false);
}

int cx_batch_get_pass(cx_batch *B, int64_t n_steps, int32_t *rows, int32_t *steps)
{
    int rc = check_batch(B);
    if (rc) return rc;
    if (!rows || !steps || n_steps < 1)
        return bfail(CX_ERR_INVALID_ARG, "need rows, steps and n_steps >= 1");
    const bool tiles = use_tiles(B, run_length(B, n_steps));
    const bool two = B->time_block == 2 && B->scheme == CX_SCHEME_EULER && B->resident_steps == 0 &&
                     n_steps >= 2;
    *rows = tiles ? 0 : B->march_rows;
    *steps = tiles ? B->plan.steps : two ? 2 : 1;
    return CX_OK;
}

int cx_batch_get_tuning(cx_batch *B, int32_t *tile_rows, int32_t *graph_steps, int64_t *group_bytes,
                        int32_t *resident_steps)
{
    int rc = check_batch(B);
    if (rc) return rc;
    if (tile_rows) *tile_rows = B->rows;
    if (graph_steps) *graph_steps = B->graph_steps;
    if (group_bytes) *group_bytes = B->group_bytes;
    if (resident_steps) *resident_steps = B->resident_steps;
    return CX_OK;
}

int cx_batch_set_time_block(cx_batch *B, int32_t stages)
{
    int rc = check_batch(B);
    if (rc) return rc;
    if (stages != 1 && stages != 2)
        return bfail(CX_ERR_INVALID_ARG, "time block: must be 1 or 2 stages per pass");
    BX_CUDA(cudaStreamSynchronize(B->stream), "synchronize before retuning");
    drop_graphs(B);
    B->time_block = stages;
    return apply_tuning(B, true);
}

int cx_batch_get_time_block(cx_batch *B, int32_t *stages)
{
    int rc = check_batch(B);
    if (rc) return rc;
    if (!stages) return bfail(CX_ERR_INVALID_ARG, "stages must not be NULL");
    *stages = B->time_block;
    return CX_OK;
}

int cx_batch_step(cx_batch *B, int64_t n_steps)
{
    cx::NvtxRange range("cx_batch_step");
    int rc = check_batch(B);
    if (rc) return rc;
    if (n_steps < 0) return bfail(CX_ERR_INVALID_ARG, "n_steps < 0");
    if (n_steps == 0) return CX_OK;
    // (the graphs hold the plan for graph_steps, which only a knob changes)
    B->tiles = use_tiles(B, run_length(B, n_steps));
    const int ngroups = (int)B->group_first.size() - 1;
    if (B->graph_steps > 0 && (int)B->gexec[0].size() != ngroups) {
        drop_graphs(B);
        for (int p = 0; p < 2; ++p) {
            B->gexec[p].assign(ngroups, nullptr);
            B->gend[p].assign(ngroups, 0);
        }
    }
    int end_parity = B->cur;
    for (int gi = 0; gi < ngroups; ++gi) {
        const int i0 = B->group_first[gi], i1 = B->group_first[gi + 1];
        int par = B->cur;
        int64_t left = n_steps;
        if (B->resident_steps > 0) {
            rc = run_resident(B, i0, i1, par, left, B->step, &end_parity);
            if (rc) return rc;
            continue;
        }
        if (B->graph_steps > 0) {
            while (left >= B->graph_steps) {
                if (!B->gexec[par][gi]) {
                    rc = capture_group(B, gi, par, &B->gexec[par][gi], &B->gend[par][gi]);
                    if (rc) return rc;
                }
                BX_CUDA(mark_step(B, B->step + (n_steps - left)), "step mark");
                BX_CUDA(cudaGraphLaunch(B->gexec[par][gi], B->stream), "graph launch");
                left -= B->graph_steps;
                par = B->gend[par][gi];
            }
        }
        int64_t marked = -1;  // `left` when the step was last marked
        while (left > 0) {
            if (marked < 0 || marked - left > (1 << 30)) {
                BX_CUDA(mark_step(B, B->step + (n_steps - left)), "step mark");
                marked = left;
            }
            int taken = 1;
            BX_CUDA(one_pass(B, i0, i1, &par, left, (int)(marked - left), &taken), "batch step launch");
            left -= taken;
        }
        end_parity = par;
    }
    B->cur = end_parity;
    B->step += n_steps;
    return CX_OK;
}

int cx_batch_synchronize(cx_batch *B)
{
    int rc = check_batch(B);
    if (rc) return rc;
    BX_CUDA(cudaStreamSynchronize(B->stream), "batch synchronize");
    return check_barrier(B);
}

int cx_batch_diagnostics(cx_batch *B, cx_diag *out)
{
    cx::NvtxRange range("cx_batch_diagnostics");
    int rc = check_batch(B);
    if (rc) return rc;
    if (!out) return bfail(CX_ERR_INVALID_ARG, "out must not be NULL");
    BX_CUDA(cx::launch_batch_diag(B->prec, B->d_inst, 0, B->count, kDiagBlocksPerInst, B->cur,
                                  B->d_part, B->h_res, B->stream),
            "batch diagnostics launch");
    BX_CUDA(cudaStreamSynchronize(B->stream), "batch diagnostics synchronize");
    rc = check_barrier(B);
    if (rc) return rc;
    int worst = CX_OK;
    for (int i = 0; i < B->count; ++i) {
        const double *h = B->h_res + 8LL * i;
        const double area = B->g[i].dx * B->g[i].dx;
        cx_diag &d = out[i];
        memset(&d, 0, sizeof d);
        d.step = B->step;
        d.dt = B->dt[i];
        d.t = (double)B->step * B->dt[i];
        d.mass_b = area * h[0];
        d.mass_n = area * h[1];
        d.invariant = area * (h[0] + B->p[i].theta * h[1]);
        d.min_b = h[2];
        d.min_n = h[3];
        d.max_b = h[4];
        d.r_env = h[5] >= 0.0 ? 0.5 * B->g[i].dx * sqrt(h[5]) : 0.0;
        d.area_env = area * h[7];
        d.finite = h[6] == 0.0 ? 1 : 0;
        d.status = !d.finite ? CX_ERR_NONFINITE
                             : ((d.min_b < 0.0 || d.min_n < 0.0) ? CX_ERR_NEGATIVE : CX_OK);
        if (d.status == CX_ERR_NONFINITE || (d.status != CX_OK && worst == CX_OK)) worst = d.status;
    }
    if (worst != CX_OK) return bfail(worst, "an instance of the batch is unhealthy (see status)");
    return CX_OK;
}

static int batch_io(cx_batch *B, int32_t index, int32_t which, int32_t dtype, size_t count)
{
    int rc = check_batch(B);
    if (rc) return rc;
    if (index < 0 || index >= B->count) return bfail(CX_ERR_INVALID_ARG, "instance index out of range");
    if (which < CX_FIELD_B || which > CX_FIELD_SIGMA) return bfail(CX_ERR_INVALID_ARG, "bad field");
    if (dtype != CX_F64 && dtype != CX_F32) return bfail(CX_ERR_INVALID_ARG, "bad dtype");
    if (count != (size_t)B->g[index].nx * (size_t)B->g[index].ny)
        return bfail(CX_ERR_INVALID_ARG, "count != nx*ny of the instance");
    return CX_OK;
}

static void *batch_field(cx_batch *B, int i, int which)
{
    if (which == CX_FIELD_B) return B->fb[B->cur][i];
    if (which == CX_FIELD_N) return B->fn[B->cur][i];
    return B->fs[i];
}

int cx_batch_get_field(cx_batch *B, int32_t index, int32_t which, void *host, int32_t dtype,
                       size_t count)
{
    int rc = batch_io(B, index, which, dtype, count);
    if (rc) return rc;
    if (!host) return bfail(CX_ERR_INVALID_ARG, "host must not be NULL");
    const int sd = B->prec == CX_PREC_F64 ? CX_F64 : CX_F32;
    const size_t row = (size_t)B->g[index].nx * B->elem;
    if (void *view = cx::pinned_view(host, count, dtype == CX_F64 ? 8 : 4)) {
        BX_CUDA(cx::launch_read_field(B->prec, batch_field(B, index, which), B->g[index].nx,
                                      B->g[index].ny, B->pitch[index], view, dtype, B->stream),
                "field read");
        BX_CUDA(cudaStreamSynchronize(B->stream), "field read synchronize");
        return CX_OK;
    }
    std::vector<unsigned char> tmp;
    void *dst = host;
    if (dtype != sd) {
        try { tmp.resize(count * B->elem); } catch (...) { return bfail(CX_ERR_OOM, "host staging"); }
        dst = tmp.data();
    }
    BX_CUDA(cudaStreamSynchronize(B->stream), "synchronize before field read");
    // the array in natural in-row order for the copy, and back to pair order, also
    // when the copy was refused (an array that is pinned in part)
    void *f = batch_field(B, index, which);
    const cx_grid &g = B->g[index];
    BX_CUDA(cx::launch_pair_order(B->prec, f, g.nx, g.ny, B->pitch[index], B->stream), "reorder");
    const cudaError_t copied =
        cudaMemcpy2DAsync(dst, row, f, (size_t)B->pitch[index] * B->elem, row, B->g[index].ny,
                          cudaMemcpyDeviceToHost, B->stream);
    if (copied != cudaSuccess) cudaGetLastError();  // reported below, not by the launch
    BX_CUDA(cx::launch_pair_order(B->prec, f, g.nx, g.ny, B->pitch[index], B->stream), "reorder");
    BX_CUDA(copied, "field copy to host");
    BX_CUDA(cudaStreamSynchronize(B->stream), "field copy synchronize");
    if (dtype != sd) {
        if (sd == CX_F32)
            for (size_t q = 0; q < count; ++q) ((double *)host)[q] = ((const float *)dst)[q];
        else
            for (size_t q = 0; q < count; ++q) ((float *)host)[q] = (float)((const double *)dst)[q];
    }
    return CX_OK;
}

int cx_batch_set_field(cx_batch *B, int32_t index, int32_t which, const void *host, int32_t dtype,
                       size_t count)
{
    int rc = batch_io(B, index, which, dtype, count);
    if (rc) return rc;
    if (!host) return bfail(CX_ERR_INVALID_ARG, "host must not be NULL");
    const int sd = B->prec == CX_PREC_F64 ? CX_F64 : CX_F32;
    const size_t row = (size_t)B->g[index].nx * B->elem;
    std::vector<unsigned char> tmp;
    const void *src = host;
    if (dtype != sd) {
        try { tmp.resize(count * B->elem); } catch (...) { return bfail(CX_ERR_OOM, "host staging"); }
        if (sd == CX_F32)
            for (size_t q = 0; q < count; ++q) ((float *)tmp.data())[q] = (float)((const double *)host)[q];
        else
            for (size_t q = 0; q < count; ++q) ((double *)tmp.data())[q] = ((const float *)host)[q];
        src = tmp.data();
    }
    BX_CUDA(cudaStreamSynchronize(B->stream), "synchronize before field write");
    BX_CUDA(cudaMemcpy2DAsync(batch_field(B, index, which), (size_t)B->pitch[index] * B->elem, src, row,
                              row, B->g[index].ny, cudaMemcpyHostToDevice, B->stream),
            "field copy to device");
    BX_CUDA(cx::launch_pair_order(B->prec, batch_field(B, index, which), B->g[index].nx,
                                  B->g[index].ny, B->pitch[index], B->stream),
            "reorder");
    BX_CUDA(cudaStreamSynchronize(B->stream), "field copy synchronize");
    return CX_OK;
}

int cx_batch_polar_profile(cx_batch *B, int32_t index, double radius, int32_t nsamples,
                           double *host_out)
{
    int rc = check_batch(B);
    if (rc) return rc;
    if (index < 0 || index >= B->count) return bfail(CX_ERR_INVALID_ARG, "instance index out of range");
    if (!host_out || nsamples < 1 || nsamples > (1 << 24) || !(isfinite(radius) && radius >= 0.0))
        return bfail(CX_ERR_INVALID_ARG, "need host_out, 1 <= nsamples <= 2^24, radius >= 0");
    double *d = nullptr;
    BX_CUDA(cudaMalloc((void **)&d, sizeof(double) * (size_t)nsamples), "profile buffer");
    const cx_grid &g = B->g[index];
    cudaError_t e = cx::launch_polar(B->prec, B->fb[B->cur][index], g.nx, g.ny, B->pitch[index], g.dx,
                                     radius, nsamples, d, B->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(host_out, d, sizeof(double) * (size_t)nsamples, cudaMemcpyDeviceToHost,
                            B->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(B->stream);
    cudaFree(d);
    if (e != cudaSuccess) return bcuda(e, "polar profile");
    return CX_OK;
}

int cx_batch_get_time(cx_batch *B, int32_t *count, int64_t *step)
{
    int rc = check_batch(B);
    if (rc) return rc;
    if (count) *count = B->count;
    if (step) *step = B->step;
    return CX_OK;
}

}  // extern "C"
