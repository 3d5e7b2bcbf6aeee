"""The float64 stage kernel's tile shapes and its integer-pipe arithmetic: grids
around every tile choice and ragged on both axes against the oracle, and exact
scaling of a run by powers of two (the wave speeds and reciprocals split
exponents from significands, so any magnitude gives the same bits)."""
import pytest
import torch

from oracle import rsst_oracle as ro
from oracle.workload import problem_from
from paper_1812_04135_gb300 import inputs, rsst
from tests.parity import check_precision

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import os
    if not os.path.exists(rsst.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    rsst.lib()


def gpu_run(w, U, nsteps):
    s = rsst.Solver(w, "fp64")
    try:
        s.set_state(U.cuda())
        s.step(nsteps)
        return s.get_state("cpu"), s.dt()
    finally:
        s.close()


# one and two tiles a SM of each shape (8 x 8, 16 x 8, 16 x 16), remainders of 1 and 15 cells
@pytest.mark.parametrize("n", [(8, 8), (9, 7), (63, 65), (128, 96), (223, 225), (241, 17), (17, 500), (250, 250), (305, 303)])
@pytest.mark.parametrize("bc,cmax", [(("periodic", "periodic"), 0.0), (("reflect", "reflect"), 0.7)])
def test_tile_shapes_match_the_oracle(n, bc, cmax):
    w = inputs.random_smooth_state(2, n, xi=6.0, variant="pvs", bc=bc, grav=(0.1, -0.3))
    w["cmax"] = cmax
    prob, U = problem_from(w)
    ref = ro.run(U, prob, 2)
    got, _ = gpu_run(w, U, 2)
    check_precision(got, ref, w, U, prob, 2, "fp64", 1e-10, what=(n, bc, cmax))


@pytest.mark.parametrize("n", [(40,), (37, 21), (11, 9, 10)])
@pytest.mark.parametrize("variant", ["euler", "pvs", "dms", "pd"])
@pytest.mark.parametrize("power", [-300, 200])
def test_scaling_by_powers_of_two_is_exact(n, variant, power):
    """rho, m and E times 2^k: the same speeds, so the same dt and 2^k times the state, bit for bit."""
    w = inputs.random_smooth_state(len(n), n, xi=5.0, variant=variant)
    _, U = problem_from(w)
    ref, dt = gpu_run(w, U, 3)
    got, dt2 = gpu_run(w, U * 2.0 ** power, 3)
    assert dt2 == dt
    assert torch.equal(got, ref * 2.0 ** power)
