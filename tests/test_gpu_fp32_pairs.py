"""The 2D float32 tile routine's pairs of columns: grids around the tile, odd
widths (the last column stands alone) and heights that end inside a segment,
with and without a background, walls and the C_max law, against the oracle; and
the conserved sums, which only hold if both warps and tiles that share a face
form it with equal bits."""
import numpy as np
import pytest
import torch

from oracle import rsst_oracle as ro
from oracle.workload import problem_from
from paper_1812_04135_gb300 import inputs, rsst
from tests.parity import rel_linf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import os
    if not os.path.exists(rsst.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    rsst.lib()


def gpu_run(w, U, nsteps):
    s = rsst.Solver(w, "fp32_pert")
    try:
        s.set_state(U.cuda())
        s.step(nsteps)
        return s.get_state("cpu")
    finally:
        s.close()


@pytest.mark.parametrize("n", [(2, 3), (3, 2), (63, 9), (64, 8), (65, 7), (127, 4), (128, 12), (129, 5), (191, 17), (257, 33)])
@pytest.mark.parametrize("case", ["plain", "walls", "background", "background_cmax"])
def test_pairs_match_the_oracle(n, case):
    w = inputs.random_smooth_state(2, n, xi=4.0, variant="pvs", bc=("reflect", "reflect") if case == "walls" else None,
                                   grav=(0.2, -0.1, 0.0) if case == "walls" else (0.0, 0.0, 0.0))
    if case.startswith("background"):
        y = (np.arange(-2, n[1] + 2) + 0.5) / n[1]
        w.update(vertical=1, bg_rho=1.2 + 0.3 * np.sin(2 * np.pi * y), bg_p=1.1 + 0.1 * np.cos(2 * np.pi * y))
    if case.endswith("cmax"):
        w["cmax"] = 0.5
    prob, U = problem_from(w)
    ref = ro.run(U, prob, 3)
    assert max(rel_linf(gpu_run(w, U, 3), ref, w["gamma"])) < 1e-5


def test_shared_faces_conserve():
    w = inputs.random_smooth_state(2, (200, 40), xi=1.0, variant="euler")
    _, U = problem_from(w)
    got = gpu_run(w, U, 50)
    for v in range(4):  # 50 steps of float32 rounding, 8000 cells, random signs
        assert abs(float((got[v] - U[v]).sum())) < 50 * 8000 ** 0.5 * 2.0 ** -23 * float(U[v].abs().max())
