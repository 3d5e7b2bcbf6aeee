"""Short 1D float64 lines run many steps in one launch on a thread-block
cluster: sizes around the cells a CTA takes (one CTA, a last CTA with a single
cell, the largest line and the first one beyond it), both boundaries, a wall
background, the C_max law and the covolume gas against the oracle; and the same
bits however the steps are split over calls and launches."""
import numpy as np
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


def gpu_run(w, U, plan, dt=0.0):
    s = rsst.Solver(w, "fp64")
    try:
        s.set_state(U.cuda())
        for k in plan:
            s.step(k, dt)
        return s.get_state("cpu"), s.dt(), s.time()
    finally:
        s.close()


@pytest.mark.parametrize("n", [2, 3, 15, 16, 17, 33, 255, 256, 257, 500, 2033, 2048, 2049])
@pytest.mark.parametrize("case", ["periodic", "reflect", "background", "cmax", "covolume"])
def test_line_matches_the_oracle(n, case):
    w = inputs.random_smooth_state(1, (n,), xi=4.0, variant="pms" if case == "reflect" else "pvs",
                                   bc=("reflect",) if case in ("reflect", "background") else ("periodic",),
                                   grav=(-0.2,) if case == "background" else (0.0,))
    if case == "background":
        z = (np.arange(-2, n + 2) + 0.5) / n
        w.update(vertical=0, bg_rho=2.0 - 0.3 * z, bg_p=1.5 - 0.2 * z)
    if case == "cmax":
        w["cmax"] = 0.5
    if case == "covolume":
        w["covolume"] = 0.1
    prob, U = problem_from(w)
    ref = ro.run(U, prob, 4)
    got, _, _ = gpu_run(w, U, [4])
    check_precision(got, ref, w, U, prob, 4, "fp64", 1e-10, what=(n, case))


@pytest.mark.parametrize("dt", [0.0, 2e-5])
def test_steps_split_over_calls_and_launches_give_the_same_bits(dt):
    w = inputs.sound_wave_1d(256, xi=10.0, eps=1e-3)
    _, U = problem_from(w)
    ref = gpu_run(w, U, [1300], dt)  # more than one launch takes
    for plan in ([1] * 20 + [1280], [1023, 1, 276], [37, 1263]):
        got = gpu_run(w, U, plan, dt)
        assert torch.equal(got[0], ref[0]) and got[1:] == ref[1:], plan


def test_line_flags_a_non_physical_state():
    w = inputs.random_smooth_state(1, (300,), xi=4.0, variant="pvs")
    _, U = problem_from(w)
    s = rsst.Solver(w, "fp64")
    s.set_state(U.cuda())
    s.step(3, 50.0)  # far beyond the stability limit
    with pytest.raises(rsst.RsstError) as e:
        s.sync()
    assert e.value.code == rsst.RSST_ENONPHYSICAL
    s.set_state(U.cuda())
    s.step(3)
    s.sync()
    s.close()
