"""The double-float stage kernel's bounded wait for its tile copy: a test wait
that nothing completes runs out, the run is flagged, and a fresh state steps to
the oracle's result."""
import pytest
import torch

from oracle import rsst_oracle as ro
from oracle.workload import problem_from
from paper_1812_04135_gb300 import inputs, rsst
from tests.parity import rel_linf

pytestmark = pytest.mark.gpu

LIMIT_NS = 2_000_000


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import os
    if not os.path.exists(rsst.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    rsst.lib()


@pytest.mark.parametrize("case", ["shear2d", "polytrope3d"])
@pytest.mark.parametrize("steps", [1, 40])  # plain launches, and blocks that replay a graph
def test_wait_runs_out_drains_and_is_reported(case, steps):
    if case == "shear2d":
        w = inputs.shear_layer_2d(72, 40, xi=30.0, variant="pvs")
    else:
        w = inputs.polytrope_3d(24, 16, 20, xi=50.0, amp=1e-3, contrast=20.0)
    U = torch.from_numpy(w["U"]).cuda()
    s = rsst.Solver(w, "fp64_df")
    try:
        s.set_state(U)
        rsst.rsst_debug_stall_wait_df(s.h, LIMIT_NS)
        s.step(steps)
        with pytest.raises(rsst.RsstError) as e:
            s.sync()
        assert e.value.code == rsst.RSST_ETIMEOUT, str(e.value)
        rsst.rsst_debug_stall_wait_df(s.h, 0)
        s.set_state(U)
        s.step(2)
        prob, U0 = problem_from(w)
        err = rel_linf(s.get_state("cpu"), ro.run(U0, prob, 2), w["gamma"])
        assert max(err) < 1e-10, err
    finally:
        s.close()


def test_hook_is_for_double_float_tiles_only():
    shear, line = inputs.shear_layer_2d(64, 32, xi=30.0, variant="pvs"), inputs.sound_wave_1d(256, xi=10.0)
    for w, precision, limit, code in ((shear, "fp64_df", -1, rsst.RSST_EINVAL), (shear, "fp64_df", 2_000_000_000, rsst.RSST_EINVAL),
                                      (shear, "fp64", LIMIT_NS, rsst.RSST_EUNSUPPORTED),
                                      (shear, "fp32_pert", LIMIT_NS, rsst.RSST_EUNSUPPORTED),
                                      (line, "fp64_df", LIMIT_NS, rsst.RSST_EUNSUPPORTED)):
        s = rsst.Solver(w, precision)
        try:
            with pytest.raises(rsst.RsstError) as e:
                rsst.rsst_debug_stall_wait_df(s.h, limit)
            assert e.value.code == code
        finally:
            s.close()
