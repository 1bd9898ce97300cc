"""The FP64 receptor law without chemotaxis (chi0 = 0, the default, or next to
nothing) at every nutrient density: the weight's strength is folded into its
denominator's scale, whose square has to stay finite."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

TOL64 = 1e-12  # relative L2, as for every FP64 state
CASES = [(chi0, n0) for chi0 in (0.0, 1e-300) for n0 in (1.0, 4095.0, 1e5, 1e10)]
STEPS = 9


@pytest.fixture(scope="module")
def cx():
    from paper_1301_5058_gb300 import _build
    _build.build()
    import paper_1301_5058_gb300 as cx
    return cx


def params(chi0, n0, mobility):
    return dict(chi0=chi0, n0=n0, sigma0=3.0, noise_amp=0.5, bM=0.71, r0sq=64.0, precision=0,
                mobility=mobility)


def state_and_result(nx, ny, chi0, n0, mobility, seed):
    """A rough state of densities up to n0, and the oracle's after STEPS steps."""
    rng = np.random.default_rng(nx + ny)
    b, n = (n0 * (0.5 + 0.5 * rng.uniform(0, 1, (ny, nx))) for _ in range(2))
    dt = 0.2 * oracle.dt_limit(dx=1.0, Dn=1.0, theta=1.0, chi0=chi0, n0=n0, bM=0.71, sigma0=3.0,
                               amp=0.5)
    s = oracle.sigma_field(nx, ny, seed, 3.0, 0.5)
    ob, on, _ = oracle.run(s, b, n, STEPS, dx=1.0, dt=dt, Dn=1.0, theta=1.0, chi0=chi0,
                           mobility=mobility)
    return b, n, ob, on


def close(got, want):
    return np.linalg.norm(got - want) <= TOL64 * np.linalg.norm(want)


@pytest.mark.parametrize("mobility", [0, 1])
@pytest.mark.parametrize("chi0,n0", CASES)
@pytest.mark.parametrize("nx,ny,depth", [(70, 45, 1), (70, 45, 2), (150, 1, None)],
                         ids=["grid", "two-stage", "strip"])
def test_no_chemotaxis_at_any_density(cx, nx, ny, depth, chi0, n0, mobility):
    b, n, ob, on = state_and_result(nx, ny, chi0, n0, mobility, 3)
    with cx.Sim(nx, ny, 1.0, seed=3, **params(chi0, n0, mobility)) as sim:
        if depth:
            cx.cx_set_time_block(sim.h, depth)
        sim.set_field(cx.CX_FIELD_B, b)
        sim.set_field(cx.CX_FIELD_N, n)
        sim.step(STEPS)
        assert close(sim.field(cx.CX_FIELD_B), ob) and close(sim.field(cx.CX_FIELD_N), on)


@pytest.mark.parametrize("mobility", [0, 1])
@pytest.mark.parametrize("nx,ny", [(70, 45), (150, 1)], ids=["grids", "strips"])
def test_no_chemotaxis_in_a_batch(cx, nx, ny, mobility):
    specs = [dict(nx=nx, ny=ny, dx=1.0, seed=i, **params(chi0, n0, mobility))
             for i, (chi0, n0) in enumerate(CASES)]
    refs = []
    with cx.Batch(specs) as bt:
        for i, (chi0, n0) in enumerate(CASES):
            b, n, ob, on = state_and_result(nx, ny, chi0, n0, mobility, i)
            bt.set_field(i, cx.CX_FIELD_B, b)
            bt.set_field(i, cx.CX_FIELD_N, n)
            refs.append((ob, on))
        bt.step(STEPS)
        for i, (ob, on) in enumerate(refs):
            assert close(bt.field(i, cx.CX_FIELD_B), ob), CASES[i]
            assert close(bt.field(i, cx.CX_FIELD_N), on), CASES[i]
