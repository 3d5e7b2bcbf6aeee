"""Loading and reading back a state: rows shorter and longer than a warp, every
boundary, the conversions of each storage over the whole float range, and the
CFL step taken while loading."""
import numpy as np
import pytest
import torch

from oracle import rsst_oracle as ro
from oracle.workload import problem_from
from paper_1812_04135_gb300 import inputs, rsst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import os
    if not os.path.exists(rsst.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    rsst.lib()


@pytest.mark.parametrize("n", [(2,), (31,), (1027,), (33, 5), (2, 67), (260, 9), (7, 9, 34), (65, 3, 2)])
@pytest.mark.parametrize("bc", ["periodic", "reflect"])
@pytest.mark.parametrize("precision", ["fp64", "fp64_df", "fp32_pert"])
def test_round_trip_and_cfl_step(n, bc, precision):
    w = inputs.random_smooth_state(len(n), n, xi=3.0, variant="pvs", bc=(bc,) * len(n))
    v = len(n) - 1
    k = np.arange(n[v] + 4)
    w.update(vertical=v, bg_rho=1.0 + 0.01 * k, bg_p=2.0 - 0.001 * k)
    prob, U = problem_from(w)
    s = rsst.Solver(w, precision)
    s.set_state(U.cuda())
    got, dt = s.get_state("cpu"), s.dt()
    s.close()
    if precision == "fp64":
        want = U
    elif precision == "fp64_df":
        hi = U.float()
        want = hi.double() + (U - hi.double()).float().double()
    else:
        shape = [1] * (len(n) + 1)
        shape[1] = n[v]  # the vertical axis is the last dimension: the slowest in memory
        r0 = torch.as_tensor(w["bg_rho"][2:-2]).reshape(shape[1:])
        e0 = torch.as_tensor(w["bg_p"][2:-2] / (w["gamma"] - 1.0)).reshape(shape[1:])
        U0 = torch.zeros_like(U)
        U0[0] += r0
        U0[-1] += e0
        want = (U - U0).float().double() + U0
    assert torch.equal(got, want)
    assert dt == pytest.approx(ro.cfl_dt(U, prob), rel=1e-12 if precision != "fp32_pert" else 1e-6)


@pytest.mark.parametrize("precision", ["fp64_df", "fp32_pert"])
def test_conversions_over_the_float_range(precision):
    """Zeros, subnormal and largest floats, halfway cases: the bits of the plain conversions."""
    rng = np.random.default_rng(3)
    n = 4096
    x = np.ldexp(1.0 + rng.random(3 * n), rng.integers(-160, 140, 3 * n)) * rng.choice([-1.0, 1.0], 3 * n)
    x[:8] = [0.0, -0.0, 1e-45, -7e-46, 3.4028235677973366e38, 1.1754943157898259e-38, 1.0 + 2.0 ** -24, 1.0 + 3 * 2.0 ** -24]
    x[8:2000] = np.ldexp(np.round(np.ldexp(rng.random(1992), 25)), rng.integers(-60, 60, 1992))  # ties
    U = torch.from_numpy(x.reshape(3, n))
    w = inputs.random_smooth_state(1, (n,), xi=1.0, variant="euler")
    s = rsst.Solver(w, precision)
    s.set_state(U.cuda())
    out = torch.empty_like(U, device="cuda")
    with pytest.raises(rsst.RsstError) as e:  # written all the same
        rsst.rsst_get_state(s.h, out)
    assert e.value.code == rsst.RSST_ENONPHYSICAL
    s.close()
    hi = U.float()
    want = hi.double()
    if precision == "fp64_df":
        want = want + (U - want).float().double()
    got = out.cpu()
    same = (got == want) | (torch.isnan(got) & torch.isnan(want))
    assert bool(same.all()), (U[~same][:5], got[~same][:5], want[~same][:5])
