"""Loading and reading back narrow grids and lines, whose blocks are shaped by
the row: the round trip, and a step of a narrow periodic grid against the same
state repeated along x (loaded in other blocks), bit for bit."""
import numpy as np
import pytest
import torch

from paper_1812_04135_gb300 import inputs, rsst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import os
    if not os.path.exists(rsst.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    rsst.lib()


def one_step(w, U, precision):
    s = rsst.Solver(w, precision)
    try:
        s.set_state(U)
        back = s.get_state("cuda")
        s.step(1, 1e-3)
        return back, s.get_state("cuda")
    finally:
        s.close()


# rows of 6 to 64 stored cells, 2 to 200 rows: every block width, remainders on both axes
@pytest.mark.parametrize("n", [(2, 2), (3, 200), (4, 9), (5, 33), (8, 3), (11, 65), (12, 7), (13, 5), (28, 6), (60, 2),
                               (2, 3, 50), (4, 4, 31), (9, 2, 3)])
@pytest.mark.parametrize("precision", ["fp64", "fp64_df", "fp32_pert"])
def test_narrow_grid_equals_its_repetition(n, precision):
    w = inputs.random_smooth_state(len(n), n, xi=3.0, variant="pvs")
    U = torch.as_tensor(w["U"]).cuda()
    back, new = one_step(w, U, precision)
    wide = dict(w, n=(n[0] * 40,) + tuple(n[1:]))
    rep = (1,) * len(n) + (40,)
    back2, new2 = one_step(wide, U.repeat(*rep), precision)
    if precision == "fp64":
        assert torch.equal(back, U)
    assert torch.equal(back2, back.repeat(*rep)) and torch.equal(new2, new.repeat(*rep))


@pytest.mark.parametrize("n", [255, 256, 257, 100003])
@pytest.mark.parametrize("precision", ["fp64", "fp64_df", "fp32_pert"])
def test_line_round_trip(n, precision):
    rng = np.random.default_rng(n)
    U = torch.from_numpy(1.0 + rng.random((3, n))).cuda()
    w = inputs.random_smooth_state(1, (n,), xi=3.0, variant="pvs")
    s = rsst.Solver(w, precision)
    try:
        s.set_state(U)
        got = torch.empty_like(U)
        with pytest.raises(rsst.RsstError) as e:  # these energies are below the kinetic one; written all the same
            rsst.rsst_get_state(s.h, got)
        assert e.value.code == rsst.RSST_ENONPHYSICAL
    finally:
        s.close()
    hi = U.float().double()
    want = {"fp64": U, "fp32_pert": hi, "fp64_df": hi + (U - hi).float().double()}[precision]
    assert torch.equal(got, want)
