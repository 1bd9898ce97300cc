"""Batch steps captured by the caller: they need no call of the same length
before them, and other lengths run in between do not disturb them.  Batches
of more distinct sizes than a launch of the register tiles has runs."""
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


def single_march(cx, spec, steps, dtype):
    kw = {k: v for k, v in spec.items() if k not in ("nx", "ny", "dx", "seed")}
    with cx.Sim(spec["nx"], spec["ny"], spec["dx"], seed=spec["seed"], **kw) as sim:
        cx.cx_set_time_block(sim.h, 1)
        sim.step(steps)
        return sim.field(cx.CX_FIELD_B, dtype), sim.field(cx.CX_FIELD_N, dtype)


@pytest.mark.parametrize("kw,sizes", [
    (dict(), [(200, 130), (64, 48), (31, 7)]),
    (dict(precision=0, chemo_law=1), [(400, 1), (33, 1)]),
    (dict(precision=0), [(96, 80)])], ids=["tiles", "strips", "f64"])
def test_captured_steps_of_a_new_length(cx, kw, sizes):
    torch = pytest.importorskip("torch")
    dtype = np.float64 if kw.get("precision") == 0 else np.float32
    specs = [dict(BASE, nx=nx, ny=ny, dx=1.0, seed=20 + i, **kw) for i, (nx, ny) in enumerate(sizes)]
    with cx.Batch(specs) as bt:
        stream = torch.cuda.Stream()
        cx.cx_batch_set_stream(bt.h, stream.cuda_stream)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):  # the batch's first steps
            bt.step(23)
            bt.step(23)  # twice: the state is back in the buffers it started from
        graph.replay()
        torch.cuda.synchronize()
        lengths = [n for n in range(1, 44) if n != 23]
        for n in lengths:
            bt.step(n)
            bt.step(n)
        cx.cx_batch_synchronize(bt.h)
        graph.replay()
        torch.cuda.synchronize()
        got = [(bt.field(i, cx.CX_FIELD_B, dtype), bt.field(i, cx.CX_FIELD_N, dtype))
               for i in range(len(specs))]
    for spec, (b, n) in zip(specs, got):
        want = single_march(cx, spec, 4 * 23 + 2 * sum(lengths), dtype)
        assert np.array_equal(b, want[0]) and np.array_equal(n, want[1])


@pytest.mark.parametrize("count", [8, 9, 20, 223, 224, 225, 600])
@pytest.mark.parametrize("kw", [dict(), dict(noise_mode=1, noise_dist=1), dict(precision=0)],
                         ids=["tiles", "per-step", "strips"])
def test_more_sizes_than_runs_of_a_launch(cx, kw, count):
    f64 = kw.get("precision") == 0
    dtype = np.float64 if f64 else np.float32
    specs = [dict(BASE, nx=(7 + 5 * i) % (701 if f64 else 311) + 1, ny=1 if f64 else i % 149 + 1, dx=1.0, seed=i, **kw)
             for i in range(count)]
    assert len({(s["nx"], s["ny"]) for s in specs}) == count
    specs.append(dict(specs[5], seed=1000))  # a size of two instances
    with cx.Batch(specs) as bt:
        bt.step(64 + 9)
        for i in [*range(0, count, max(1, count // 18)), count - 1, 5, count]:
            want = single_march(cx, specs[i], 64 + 9, dtype)
            assert np.array_equal(bt.field(i, cx.CX_FIELD_B, dtype), want[0]), i
            assert np.array_equal(bt.field(i, cx.CX_FIELD_N, dtype), want[1]), i
