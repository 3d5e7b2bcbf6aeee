"""Faces of the 2D float32 kernel are formed by whichever lane, warp or tile
comes to own them: a periodic run from a shifted state equals the shifted run
bit for bit."""
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


# not multiples of the pair (2), the warp's columns (64), the tile (128 x 8) or the segment (4)
SHIFTS = [(1, 0), (0, 1), (63, 3), (64, 5), (129, 6), (130, 4)]


@pytest.mark.parametrize("background", [False, True])
@pytest.mark.parametrize("cmax", [0.0, 0.5])
def test_shifted_state_gives_the_shifted_run(background, cmax):
    n = (321, 41)
    w = inputs.random_smooth_state(2, n, xi=20.0, variant="pvs")
    w["cmax"] = cmax
    if background:
        y = (np.arange(-2, n[1] + 2) + 0.5) / n[1]
        w.update(vertical=1, bg_rho=1.2 + 0.3 * np.sin(2 * np.pi * y), bg_p=1.1 + 0.1 * np.cos(2 * np.pi * y))
    U = torch.as_tensor(w["U"]).cuda()
    s = rsst.Solver(w, "fp32_pert")
    try:
        def run(V):
            s.set_state(V)
            s.step(6, 1e-3)
            return s.get_state("cuda")

        ref = run(U)
        for sx, sy in SHIFTS:
            sy = 0 if background else sy
            got = run(torch.roll(U, (sy, sx), (1, 2)))
            assert torch.equal(got, torch.roll(ref, (sy, sx), (1, 2))), (sx, sy)
    finally:
        s.close()
