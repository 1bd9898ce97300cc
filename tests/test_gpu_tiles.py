"""Several time steps per pass on register tiles (FP32) and strips (FP64, one
row), which untuned handles take where they are faster: the same bits as the
one-stage march, which is checked against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cx():
    from paper_1301_5058_gb300 import _build
    _build.build()
    import paper_1301_5058_gb300 as cx
    return cx


BASE = dict(n0=0.5, chi0=1.0, sigma0=3.0, noise_amp=0.5, bM=0.71, r0sq=64.0)


def fields(cx, nx, ny, calls, kw, march, dtype):
    """b and n after the calls' steps from a rough state that fills the grid."""
    rng = np.random.default_rng(nx * 10007 + ny)
    b, n = (0.5 * (1 + 0.5 * rng.uniform(-1, 1, (ny, nx))) for _ in range(2))
    with cx.Sim(nx, ny, 1.0, seed=3, **dict(BASE, **kw)) as sim:
        if march:
            cx.cx_set_time_block(sim.h, 1)
        sim.set_field(cx.CX_FIELD_B, b)
        sim.set_field(cx.CX_FIELD_N, n)
        for steps in calls:
            sim.step(steps)
        return sim.field(cx.CX_FIELD_B, dtype), sim.field(cx.CX_FIELD_N, dtype)


# one tile, tiles that end exactly at a wall, one cell beyond, ragged; up to
# 2048 wide so that every tile shape is chosen for some size
SIZES = [(1, 1), (200, 1), (1, 200), (63, 5), (64, 64), (65, 66), (112, 48), (130, 97), (257, 131),
         (509, 517), (803, 790), (1027, 1021), (2045, 2051)]
FORMS = [dict(), dict(mobility=1, chemo_law=1), dict(scheme=1), dict(noise_mode=1, noise_dist=1),
         dict(scheme=1, noise_mode=1, mobility=1)]


@pytest.mark.parametrize("form", range(len(FORMS)))
@pytest.mark.parametrize("nx,ny", SIZES)
def test_register_tiles_are_the_march_bitwise(cx, nx, ny, form):
    kw = FORMS[form]
    calls = (1, 23, 8)  # one step, passes of unequal length, whole passes
    got = fields(cx, nx, ny, calls, kw, False, np.float32)
    want = fields(cx, nx, ny, calls, kw, True, np.float32)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


@pytest.mark.parametrize("nx", [1, 2, 31, 32, 33, 47, 48, 49, 400, 517])
@pytest.mark.parametrize("kw", [dict(chemo_law=1), dict(mobility=1), dict(scheme=1)],
                         ids=["constant", "upwind", "heun"])
def test_strips_are_the_march_bitwise(cx, nx, kw):
    kw = dict(kw, precision=0)
    got = fields(cx, nx, 1, (1, 23, 8), kw, False, np.float64)
    want = fields(cx, nx, 1, (1, 23, 8), kw, True, np.float64)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


@pytest.mark.parametrize("kw,sizes", [
    (dict(), [(256, 256), (65, 300), (31, 7), (256, 256)]),
    (dict(scheme=1, noise_mode=1, noise_dist=1), [(100, 90), (257, 64), (1, 1)]),
    (dict(precision=0, chemo_law=1), [(400, 1), (33, 1), (1, 1)]),
    (dict(precision=0), [(130, 70), (64, 48)])], ids=["f32", "paper", "strips", "f64"])
def test_untuned_batch_is_single_marches_bitwise(cx, kw, sizes):
    dtype = np.float64 if kw.get("precision") == 0 else np.float32
    specs = [dict(BASE, nx=nx, ny=ny, dx=1.0, seed=20 + i, **kw) for i, (nx, ny) in enumerate(sizes)]
    with cx.Batch(specs) as bt:
        for steps in (64 + 27, 5, 64):  # a captured chunk and a remainder, a short call, a chunk
            bt.step(steps)
        got = [(bt.field(i, cx.CX_FIELD_B, dtype), bt.field(i, cx.CX_FIELD_N, dtype))
               for i in range(len(specs))]
    for s, (b, n) in zip(specs, got):
        p = {k: v for k, v in s.items() if k not in ("nx", "ny", "dx", "seed")}
        with cx.Sim(s["nx"], s["ny"], s["dx"], seed=s["seed"], **p) as sim:
            cx.cx_set_time_block(sim.h, 1)
            sim.step(64 + 27 + 5 + 64)
            assert np.array_equal(b, sim.field(cx.CX_FIELD_B, dtype))
            assert np.array_equal(n, sim.field(cx.CX_FIELD_N, dtype))


@pytest.mark.parametrize("nx,ny,prec", [(200, 130, 1), (300, 1, 0), (96, 80, 0)])
def test_steps_captured_in_a_graph(cx, nx, ny, prec):
    # the passes of a step call are launched as dependents of one another;
    # captured and replayed they give what the call itself gives
    torch = pytest.importorskip("torch")
    dtype = np.float32 if prec else np.float64
    kw = dict(BASE, precision=prec)
    with cx.Sim(nx, ny, 1.0, seed=5, **kw) as sim, cx.Sim(nx, ny, 1.0, seed=5, **kw) as ref:
        stream = torch.cuda.Stream()
        cx.cx_set_stream(sim.h, stream.cuda_stream)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            sim.step(23)
        graph.replay()
        torch.cuda.synchronize()
        ref.step(23)
        for which in (cx.CX_FIELD_B, cx.CX_FIELD_N):
            assert np.array_equal(sim.field(which, dtype), ref.field(which, dtype))


def test_tall_grids_stay_within_the_launch(cx):
    # as many tile rows as a launch may have: the choice of tiles respects it
    with cx.Sim(1, 2_000_000, 1.0, seed=1, **BASE) as sim, \
            cx.Sim(1, 2_000_000, 1.0, seed=1, **BASE) as ref:
        cx.cx_set_time_block(ref.h, 2)
        cx.cx_set_tile_rows(ref.h, 64)
        sim.step(6)
        ref.step(6)
        assert np.array_equal(sim.field(cx.CX_FIELD_B, np.float32), ref.field(cx.CX_FIELD_B, np.float32))
