"""What runs under which knobs: handles left alone choose for themselves, a
knob pins the marches, a reset gives the choice back; never another bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BASE = dict(n0=0.5, chi0=1.0, sigma0=3.0, noise_amp=0.5, bM=0.71, r0sq=64.0)


@pytest.fixture(scope="module")
def cx():
    from paper_1301_5058_gb300 import _build
    _build.build()
    import paper_1301_5058_gb300 as cx
    return cx


@pytest.mark.parametrize("nx,ny,prec,default", [(256, 256, 1, 2), (400, 1, 0, 1)])
def test_reset_gives_a_single_grid_its_choice_back(cx, nx, ny, prec, default):
    kw = dict(BASE, precision=prec, chemo_law=1 - prec)
    dtype = np.float32 if prec else np.float64
    with cx.Sim(nx, ny, 1.0, seed=1, **kw) as sim, cx.Sim(nx, ny, 1.0, seed=1, **kw) as ref:
        rows = cx.cx_get_tile_rows(sim.h)
        assert cx.cx_get_pass(sim.h, 64)[0] == 0 and cx.cx_get_pass(sim.h, 64)[1] > 2
        for knob in (lambda: cx.cx_set_time_block(sim.h, default),  # a default one pins as well
                     lambda: cx.cx_set_tile_rows(sim.h, 17)):
            knob()
            assert cx.cx_get_pass(sim.h, 64) == (cx.cx_get_tile_rows(sim.h), default)
            assert cx.cx_get_pass(sim.h, 1)[1] == 1
            sim.step(9)
            cx.cx_reset_tuning(sim.h)
            assert (cx.cx_get_time_block(sim.h), cx.cx_get_tile_rows(sim.h)) == (default, rows)
            assert cx.cx_get_pass(sim.h, 64)[0] == 0
            sim.step(9)
        ref.step(36)
        for which in (cx.CX_FIELD_B, cx.CX_FIELD_N):
            assert np.array_equal(sim.field(which, dtype), ref.field(which, dtype))


def test_a_tuned_small_grid_still_runs_on_tiles(cx, tmp_path, monkeypatch):
    monkeypatch.setenv("CX_TUNE_CACHE", str(tmp_path / "tune.json"))
    from paper_1301_5058_gb300 import autotune
    with cx.Sim(256, 256, 1.0, seed=1, **BASE) as sim:  # 0.7 us per step; the marches 2.7
        for _ in range(2):  # timed, then from the cache
            autotune.tune_single(sim, steps=32, reps=3)
            assert cx.cx_get_pass(sim.h, 64)[0] == 0


@pytest.mark.parametrize("size,prec,rows,depth", [((256, 256), 1, 128, 2), ((400, 1), 0, 32, 1)])
def test_batch_knobs_pin_the_marches_at_their_defaults_too(cx, size, prec, rows, depth):
    kw = dict(BASE, precision=prec, chemo_law=1 - prec)
    dtype = np.float32 if prec else np.float64
    specs = [dict(nx=size[0], ny=size[1], dx=1.0, seed=i, **kw) for i in range(4)]
    with cx.Batch(specs) as bt, cx.Batch(specs) as ref:
        assert cx.cx_batch_get_pass(bt.h, 64)[0] == 0 and cx.cx_batch_get_pass(bt.h, 64)[1] > 2
        for pin in (lambda: bt.tune(rows, 64, 0, 0, depth), lambda: bt.tune(rows, 32, 0),
                    lambda: cx.cx_batch_set_time_block(bt.h, depth)):
            pin()
            assert cx.cx_batch_get_tuning(bt.h)[0] == rows
            assert cx.cx_batch_get_pass(bt.h, 64) == (rows, depth)
            bt.step(70)
            bt.tune(0, 64, 0, 0, 0)
            assert cx.cx_batch_get_tuning(bt.h) == (rows, 64, 0, 0)
            assert cx.cx_batch_get_time_block(bt.h) == depth
            assert cx.cx_batch_get_pass(bt.h, 64)[0] == 0
            bt.step(70)
        bt.tune(7, 0, 0, 5)  # the resident mode: one stage per pass
        assert cx.cx_batch_get_pass(bt.h, 64) == (7, 1)
        bt.step(9)
        ref.step(6 * 70 + 9)
        for i in range(4):
            assert np.array_equal(bt.field(i, cx.CX_FIELD_B, dtype), ref.field(i, cx.CX_FIELD_B, dtype))
        for bad in (-1, 100001):
            with pytest.raises(cx.CxError):
                cx.cx_batch_reset_tuning(bt.h, bad)


def test_height_in_effect_of_an_untouched_batch(cx):
    # the sweep's mix of sizes stays on the marches: 64 rows, whatever the
    # reported default
    from paper_1301_5058_gb300 import workloads as W
    with cx.Batch(W.sweep_specs(24, seed=0, steps=100)) as bt:
        assert cx.cx_batch_get_tuning(bt.h)[0] == 128
        assert cx.cx_batch_get_pass(bt.h, 64) == (64, 2)
        bt.tune(128, 64, 0, 0, 2)
        assert cx.cx_batch_get_pass(bt.h, 64) == (128, 2)
