"""Graph blocks on 1D float64 lines: a line above 2048 cells replays them; a
shorter one runs on the cluster kernel and takes no notice of the setting."""
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


@pytest.mark.parametrize("n,launches", [(2100, 2 * 58), (256, 3)])
def test_graph_steps_on_a_line(n, launches):
    w = inputs.sound_wave_1d(n, xi=10.0, variant="pvs")
    got = []
    for k in (0, 2, 16):
        s = rsst.Solver(w, "fp64")
        s.set_graph_steps(k)
        s.set_state(torch.from_numpy(w["U"]).cuda())
        before = s.launches()
        for m in (37, 1, 20):
            s.step(m)
        got.append((s.launches() - before, s.dt(), s.time(), s.get_state("cpu")))
        s.close()
    for g in got:
        assert g[0] == launches and g[1:3] == got[0][1:3] and torch.equal(g[3], got[0][3])
