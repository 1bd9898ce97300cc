"""What the autotuner picks, applies and keeps, with the handles and the clock
replaced by fakes."""
import json
import types

import pytest

from paper_1301_5058_gb300 import autotune


class FakeLib:
    """The calls of the tuners on one handle; `timings` maps what is in force
    (None: the library's own choice) to seconds per step."""

    def __init__(self, timings, default):
        self.timings, self.default, self.force = timings, default, None
        self.depth, self.rows = default

    def cx_set_stream(self, h, stream):
        pass

    def cx_set_time_block(self, h, depth):
        self.depth = depth
        self.force = (self.depth, self.rows)

    def cx_set_tile_rows(self, h, rows):
        self.rows = rows
        self.force = (self.depth, self.rows)

    def cx_get_time_block(self, h):
        return self.depth

    def cx_get_tile_rows(self, h):
        return self.rows

    def cx_reset_tuning(self, h):
        self.depth, self.rows = self.default
        self.force = None


@pytest.fixture
def tuner(monkeypatch, tmp_path):
    import torch
    monkeypatch.setenv("CX_TUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: types.SimpleNamespace(cuda_stream=0))

    def use(lib):
        monkeypatch.setattr(autotune, "cx", lib)
        monkeypatch.setattr(autotune, "_time_steps",
                            lambda *a: lib.timings.get(lib.force, 1.0))
        return lib
    use.cache = tmp_path / "tune.json"
    return use


def sim_of(side):
    return types.SimpleNamespace(
        h=1, step=lambda n: None, grid=types.SimpleNamespace(nx=side, ny=side),
        params=types.SimpleNamespace(precision=1, scheme=0, noise_mode=0))


@pytest.mark.parametrize("pinned,force,choice", [
    ({}, None, (2, 4)),                    # register tiles fastest
    ({(2, 64): 0.3}, (2, 64), (2, 64)),    # a march fastest
    ({(2, 4): 0.3}, (2, 4), (2, 4)),       # the march that a new handle reports
    ({(2, 4): 0.5}, None, (2, 4))])        # no faster than the library's choice
def test_single_grid_is_left_alone_where_that_is_fastest(tuner, pinned, force, choice):
    lib = tuner(FakeLib({None: 0.5, **pinned}, (2, 4)))
    got, results = autotune.tune_single(sim_of(1024), use_cache=True)
    assert got == choice and lib.force == force
    assert results[choice] == min(results.values())
    # the same from the cache, on a handle that was tuned to something else
    lib = tuner(FakeLib({}, (2, 4)))
    lib.cx_set_tile_rows(1, 256)
    assert autotune.tune_single(sim_of(1024), use_cache=True) == (choice, {})
    assert lib.force == force


def test_single_entries_without_the_librarys_choice_are_not_used(tuner):
    tuner.cache.write_text(json.dumps({"single/p1/s0/n0/1024x1024": {"choice": [1, 32]}}))
    lib = tuner(FakeLib({None: 0.5}, (2, 4)))
    assert autotune.tune_single(sim_of(1024), use_cache=True)[0] == (2, 4)
    assert lib.force is None


class FakeBatch:
    def __init__(self, timings):
        self.timings, self.force, self._stream, self.h = timings, None, object(), 1
        self.grids = [types.SimpleNamespace(nx=256, ny=256)] * 3
        self.params = [types.SimpleNamespace(precision=1, scheme=0)] * 3

    def tune(self, *knobs):
        self.force = knobs

    def step(self, n):
        pass


@pytest.mark.parametrize("timings,choice", [
    ({autotune.AUTOMATIC: 0.5}, autotune.AUTOMATIC),
    ({autotune.AUTOMATIC: 0.5, (128, 64, 0, 0, 2): 0.4}, (128, 64, 0, 0, 2))])
def test_batch_candidates_include_the_librarys_choice(tuner, monkeypatch, timings, choice):
    bt = FakeBatch(timings)
    monkeypatch.setattr(autotune, "_time_steps", lambda *a: bt.timings.get(bt.force, 1.0))
    got, results = autotune.tune_batch(bt)
    assert got == choice == bt.force and set(results) == set(autotune.BATCH_CANDIDATES)
    bt.force = None
    assert autotune.tune_batch(bt) == (choice, {}) and bt.force == choice
    # an entry that never compared with the library's choice is not used
    tuner.cache.write_text(json.dumps({autotune.batch_key(bt.grids, bt.params):
                                       {"choice": [16, 0, 0, 0, 1]}}))
    assert autotune.tune_batch(bt)[0] == choice
    # of a caller's own candidates the fastest, the library's choice or not
    assert autotune.tune_batch(bt, candidates=[(16, 0, 0, 0, 1)], use_cache=False)[0] == (16, 0, 0, 0, 1)
