"""Field reads into host arrays that the reading kernel cannot write: they go
through the copies, with the same values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KW = dict(n0=0.5, chi0=1.0, sigma0=3.0, noise_amp=0.5, r0sq=64.0)


@pytest.fixture(scope="module")
def cx():
    from paper_1301_5058_gb300 import _build
    _build.build()
    import paper_1301_5058_gb300 as cx
    return cx


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("offset", [1, 2, 4])
def test_pinned_array_not_aligned_to_its_elements(cx, prec, dtype, offset):
    # records behind a header of `offset` bytes in one pinned allocation
    torch = pytest.importorskip("torch")
    nx, ny = 64, 5
    size = nx * ny * np.dtype(dtype).itemsize
    with cx.Sim(nx, ny, 1.0, seed=3, precision=prec, **KW) as sim, \
            cx.Batch([dict(nx=nx, ny=ny, dx=1.0, seed=3, precision=prec, **KW)]) as bt:
        host = torch.full((size + 16,), 7, dtype=torch.uint8, pin_memory=True).numpy()
        out = np.frombuffer(host, dtype, nx * ny, offset).reshape(ny, nx)
        for get, ref in ((lambda w: cx.cx_get_field(sim.h, w, out), sim.field),
                         (lambda w: cx.cx_batch_get_field(bt.h, 0, w, out),
                          lambda w, d: bt.field(0, w, d))):
            for which in (cx.CX_FIELD_B, cx.CX_FIELD_N, cx.CX_FIELD_SIGMA):
                host[offset:offset + size] = 0
                assert np.array_equal(get(which), ref(which, dtype))
        assert np.all(host[:offset] == 7) and np.all(host[offset + size:] == 7)


@pytest.mark.parametrize("prec", [0, 1])
def test_refused_copy_leaves_the_state_as_it_was(cx, prec):
    # the runtime refuses a copy into an array that is pinned only in part; the
    # field has to be back in the library's order all the same
    torch = pytest.importorskip("torch")
    dtype = np.float32 if prec else np.float64
    nx, ny = 128, 256
    kw = dict(KW, precision=prec)
    page = 65536  # a whole number of pages on any host
    with cx.Sim(nx, ny, 1.0, seed=3, **kw) as sim, \
            cx.Batch([dict(nx=nx, ny=ny, dx=1.0, seed=3, **kw)]) as bt:
        whole = np.zeros(8 * page, np.uint8)
        first = -whole.ctypes.data % page
        out = whole[first:first + nx * ny * np.dtype(dtype).itemsize].view(dtype).reshape(ny, nx)
        assert out.nbytes > page
        rt = torch.cuda.cudart()
        for get, read, step in (
                (lambda: cx.cx_get_field(sim.h, cx.CX_FIELD_B, out),
                 lambda: sim.field(cx.CX_FIELD_B, dtype), sim.step),
                (lambda: cx.cx_batch_get_field(bt.h, 0, cx.CX_FIELD_B, out),
                 lambda: bt.field(0, cx.CX_FIELD_B, dtype), bt.step)):
            want = read()
            assert int(rt.cudaHostRegister(out.ctypes.data, page, 0)) == 0
            try:
                try:
                    get()
                    refused = False
                except cx.CxError:
                    refused = True
            finally:
                assert int(rt.cudaHostUnregister(out.ctypes.data)) == 0
            assert refused or np.array_equal(out, want)
            assert np.array_equal(read(), want)
            step(1)
        assert refused  # on this runtime
        for which in (cx.CX_FIELD_B, cx.CX_FIELD_N):
            assert np.array_equal(sim.field(which, dtype), bt.field(0, which, dtype))
