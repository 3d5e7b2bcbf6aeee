"""The adjoint's gather of ghost contributions on the smallest grids (a cell may
be the image of ghosts at both ends), with the C_max law's derivatives of the
wave speed, and recordings that reuse the memory of the one before."""
import pytest
import torch

from oracle import adjoint as adj
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


def reverse(s, U, dt, nsteps, every, lam):
    s.set_state(U.cuda())
    rsst.rsst_adjoint_record(s.h, dt, nsteps, every)
    lam = lam.clone().cuda()
    dxi = sum(rsst.rsst_adjoint_step(s.h, seg, lam) for seg in reversed(range(rsst.rsst_adjoint_segments(s.h))))
    return lam.cpu(), dxi


@pytest.mark.parametrize("n", [(2,), (3,), (4,), (2, 5), (129, 3), (3, 2, 4)])
@pytest.mark.parametrize("bc", ["periodic", "reflect"])
@pytest.mark.parametrize("cmax", [0.0, 0.6])
def test_small_grids_match_the_oracle(n, bc, cmax):
    w = inputs.random_smooth_state(len(n), n, xi=4.0, variant="pvs", bc=(bc,) * len(n), grav=(0.2, -0.1, 0.3)[:len(n)])
    w["cmax"] = cmax
    prob, U = problem_from(w)
    dt = 0.5 * ro.cfl_dt(U, prob)
    lam = torch.tensor(inputs.uniform_pm1(7, U.numel()).reshape(U.shape))
    want, wxi = adj.step_vjp(U, lam, dt, prob)
    s = rsst.Solver(w, "fp64")
    got, dxi = reverse(s, U, dt, 1, 1, lam)
    s.close()
    scale = float(want.abs().max())
    assert float((got - want).abs().max()) <= 1e-10 * scale
    assert dxi == pytest.approx(wxi, rel=1e-9, abs=1e-12 * scale)


def test_recordings_that_reuse_memory():
    w = inputs.random_smooth_state(2, (20, 13), xi=5.0, variant="pms", bc=("periodic", "reflect"))
    prob, U = problem_from(w)
    dt = 0.5 * ro.cfl_dt(U, prob)
    lam = torch.tensor(inputs.uniform_pm1(8, U.numel()).reshape(U.shape))
    s = rsst.Solver(w, "fp64")
    for nsteps, every in ((6, 3), (5, 3), (6, 3), (4, 2), (1, 1)):  # the same shape with a full and a ragged last segment
        _, _, want, wxi = adj.adjoint_run(U, prob, nsteps, dt, every, lam_final=lambda X: lam)
        got, dxi = reverse(s, U, dt, nsteps, every, lam)
        assert float((got - want).abs().max()) <= 1e-9 * float(want.abs().max()), (nsteps, every)
        assert dxi == pytest.approx(wxi, rel=1e-8), (nsteps, every)
    s.close()
