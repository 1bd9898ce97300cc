"""The oracle check of a benchmark record runs the kernels of that record."""
import pytest

import bench

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [64, 128])
def test_sweep_check_runs_the_sweeps_march(monkeypatch, rows):
    from paper_1301_5058_gb300 import _build
    _build.build()
    import paper_1301_5058_gb300 as cx
    ran = []
    step = cx.Batch.step

    def spy(self, n):
        ran.append(cx.cx_batch_get_pass(self.h, n))
        step(self, n)
    monkeypatch.setattr(cx.Batch, "step", spy)
    tuning = {"tile_rows": rows, "graph_steps": 64, "group_bytes": 0, "resident_steps": 0,
              "time_block": 2}
    r = bench.oracle_error_sweep(tuning, steps=40)
    assert r["pass"] and ran == [(rows, 2)]
