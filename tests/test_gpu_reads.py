"""Field reads into pinned host arrays (one kernel that writes them) against
reads into pageable ones (reorder, copy, reorder back): the same values, the
state untouched, nothing written beyond the array."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cx():
    from paper_1301_5058_gb300 import _build
    _build.build()
    import paper_1301_5058_gb300 as cx
    return cx


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("nx,ny", [(1, 1), (4, 3), (7, 5), (64, 2), (130, 97), (513, 33)])
def test_pinned_reads_equal_pageable_reads(cx, nx, ny, dtype, prec):
    torch = pytest.importorskip("torch")
    tdt = torch.float32 if dtype == np.float32 else torch.float64
    rng = np.random.default_rng(nx)
    kw = dict(n0=0.5, chi0=1.0, sigma0=3.0, noise_amp=0.5, r0sq=64.0, precision=prec)
    b = rng.uniform(0, 1, (ny, nx))
    with cx.Sim(nx, ny, 1.0, seed=3, **kw) as sim, \
            cx.Batch([dict(nx=nx, ny=ny, dx=1.0, seed=3, **kw)] * 2) as bt:
        sim.set_field(cx.CX_FIELD_B, b)
        bt.set_field(1, cx.CX_FIELD_B, b)
        for first in (0, 1, 4):  # the array's offset in its pinned allocation
            host = torch.full((nx * ny + 8,), -1.0, dtype=tdt, pin_memory=True).numpy()
            out = host[first:first + nx * ny].reshape(ny, nx)
            for which in (cx.CX_FIELD_B, cx.CX_FIELD_N, cx.CX_FIELD_SIGMA):
                want = sim.field(which, dtype)
                assert np.array_equal(cx.cx_get_field(sim.h, which, out), want)
                out[:] = -1.0
                assert np.array_equal(cx.cx_batch_get_field(bt.h, 1, which, out),
                                      bt.field(1, which, dtype))
            assert np.all(host[:first] == -1.0) and np.all(host[first + nx * ny:] == -1.0)
