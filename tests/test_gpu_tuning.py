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
