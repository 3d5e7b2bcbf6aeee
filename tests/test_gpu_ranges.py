"""Runs at the ends of the parameters that rsst_init accepts: grids that are
narrow and very tall, reduction rates and C_max laws whose squares leave the
range of a float."""
import numpy as np
import pytest
import torch

from paper_1812_04135_gb300 import rsst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import os
    if not os.path.exists(rsst.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    rsst.lib()


def workload(n, **more):
    w = {"ndim": len(n), "n": n, "dx": (1.0,) * len(n), "gamma": 5.0 / 3.0, "xi": 4.0, "variant": "pvs",
         "bc": ("periodic",) * len(n), "grav": (0.0, 0.0, 0.0), "vertical": -1, "bg_rho": None, "bg_p": None, "cmax": 0.0,
         "cfl_rule": 0, "covolume": 0.0, "cfl": 0.4}
    w.update(more)
    return w


def uniform(n, rho, v, e):
    U = torch.zeros((len(n) + 2,) + tuple(reversed(n)), dtype=torch.float64)
    U[0], U[1], U[-1] = rho, rho * v, e + 0.5 * rho * v * v
    return U.cuda()


def advance(w, U, steps, dt=0.0, precision="fp64"):
    s = rsst.Solver(w, precision)
    try:
        s.set_state(U)
        s.step(steps, dt)
        return s.get_state("cuda"), s.dt()
    finally:
        s.close()


@pytest.mark.parametrize("precision", ["fp64", "fp64_df"])
def test_narrow_and_very_tall_grid(precision):
    """More rows than 65535 tiles of 8: the run equals that of one of its 40-row periods, bit for bit."""
    nx, period, periods = 8, 40, 15000
    rng = np.random.default_rng(1)
    one = uniform((nx, period), 1.0, 0.0, 1.5)
    one += 0.1 * torch.from_numpy(rng.uniform(-1.0, 1.0, tuple(one.shape))).cuda()
    ref, _ = advance(workload((nx, period)), one, 2, 0.05, precision)
    got, _ = advance(workload((nx, period * periods)), one.repeat(1, periods, 1), 2, 0.05, precision)
    assert torch.equal(got, ref.repeat(1, periods, 1))


@pytest.mark.parametrize("n", [(40,), (20, 12), (10, 9, 8)])
def test_reduction_rate_whose_square_overflows(n):
    """a/xi vanishes beside |V|: dt is that of the flow."""
    U = uniform(n, 1.3, 0.7, 2.0)
    got, dt = advance(workload(n, xi=1e160), U, 2)
    assert dt == pytest.approx(0.4 / (0.7 * len(n)), rel=1e-12)
    assert float((got - U).abs().max()) <= 1e-13


@pytest.mark.parametrize("xi", [1e16, 1e20, 1e30])
def test_double_float_large_reduction_rate(xi):
    """Gas at rest: dt is that of a/xi, also where 1/xi^2 is below the floats."""
    n = (24, 16)
    got, dt = advance(workload(n, xi=xi), uniform(n, 1.3, 0.0, 2.0), 0, precision="fp64_df")
    a = np.sqrt(5.0 / 3.0 * (2.0 / 3.0) * 2.0 / 1.3)
    assert dt == pytest.approx(0.4 / (2.0 * a / xi), rel=1e-12)


@pytest.mark.parametrize("n", [(40,), (20, 12), (10, 9, 8)])
@pytest.mark.parametrize("scale", [-200, 150])
def test_cmax_law_at_speeds_beyond_floats(n, scale):
    """Speeds and C_max times 2^scale: dt times 2^-scale (gas at rest and in motion)."""
    for v in (0.0, 0.7):
        _, dt = advance(workload(n, cmax=0.6), uniform(n, 1.3, v, 2.0), 0)
        f = 2.0 ** scale
        _, dt2 = advance(workload(n, cmax=0.6 * f), uniform(n, 1.3, v * f, 2.0 * f * f), 0)
        assert dt2 * f == pytest.approx(dt, rel=1e-14)


@pytest.mark.parametrize("n", [(40,), (20, 12), (10, 9, 8)])
def test_cmax_law_with_an_unbounded_reduction(n):
    """(a/C_max)^4 overflows: xi is infinite, a/xi = 0 and f = 1."""
    U = uniform(n, 1.3, 0.7, 2.0)
    got, dt = advance(workload(n, cmax=1e-78), U, 2)
    assert dt == pytest.approx(0.4 / (0.7 * len(n)), rel=1e-12)
    assert float((got - U).abs().max()) <= 1e-13


def test_limiter_in_the_far_tail_of_a_profile():
    """A velocity profile whose tail passes through the subnormal numbers stays finite."""
    x = torch.arange(400, dtype=torch.float64) / 10.0
    v = 0.1 * torch.exp(-x * x).cuda()
    U = uniform((400,), 1.0, 0.0, 2.0)
    U[1] = v
    U[2] += 0.5 * v * v
    got, dt = advance(workload((400,), bc=("reflect",)), U, 3)
    assert bool(torch.isfinite(got).all()) and dt > 0.0
