"""The double-float stage kernel's tile shapes: grids around the choice of the
2D tile and ragged on every axis, with walls and the C_max law, against the
oracle."""
import pytest

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


@pytest.mark.parametrize("n", [(8, 8), (9, 7), (63, 65), (17, 241), (130, 97), (209, 207), (305, 303), (9, 8, 5), (17, 23, 11)])
@pytest.mark.parametrize("bc,cmax", [("periodic", 0.0), ("reflect", 0.7)])
def test_tile_shapes_match_the_oracle(n, bc, cmax):
    w = inputs.random_smooth_state(len(n), n, xi=6.0, variant="pvs", bc=(bc,) * len(n), grav=(0.1, -0.3, 0.2)[:len(n)])
    w["cmax"] = cmax
    prob, U = problem_from(w)
    ref = ro.run(U, prob, 2)
    s = rsst.Solver(w, "fp64_df")
    s.set_state(U.cuda())
    s.step(2)
    got = s.get_state("cpu")
    s.close()
    check_precision(got, ref, w, U, prob, 2, "fp64_df", 1e-10, what=(n, bc, cmax))
