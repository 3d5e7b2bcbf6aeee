"""dt under the C_max law against a float64 evaluation: gas at rest, so that
c_tot is a/xi alone.  Each of the kernel's roundings counted (P 1, a^2 4, w 3,
1/sqrt 3, the root 2, rates and dt 4; the squares' errors halve at each root)
gives 14 roundings of 2^-53, the evaluation here 10: 3e-15."""
import math

import pytest
import torch

from paper_1812_04135_gb300 import rsst

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(40,), (2100,), (19, 33), (9, 10, 11)])
def test_cmax_dt_has_float64_accuracy(n):
    nd, gamma, cmax, cfl = len(n), 5.0 / 3.0, 1.3, 0.4
    dx = tuple(1.0 / v for v in n)
    w = {"ndim": nd, "n": n, "dx": dx, "gamma": gamma, "xi": 1.0, "variant": "pvs", "bc": ("periodic",) * nd,
         "grav": (0.0, 0.0, 0.0), "vertical": -1, "bg_rho": None, "bg_p": None, "cmax": cmax, "cfl_rule": 0,
         "covolume": 0.0, "cfl": cfl}
    s = rsst.Solver(w, "fp64")
    try:
        for i in range(12):
            rho, e = 0.3 + 0.37 * i, 10.0 ** (i / 3.0 - 1.5) * 1.1
            U = torch.zeros((nd + 2,) + tuple(reversed(n)), dtype=torch.float64)
            U[0], U[-1] = rho, e
            a2 = gamma * ((gamma - 1.0) * e) / rho
            c = math.sqrt(a2 / math.sqrt(1.0 + a2 * a2 / cmax ** 4))
            want = cfl / (c * sum(1.0 / h for h in dx))
            s.set_state(U.cuda())
            assert abs(s.dt() / want - 1.0) <= 3e-15
            s.step(3)
            assert abs(s.dt() / want - 1.0) <= 3e-15
    finally:
        s.close()
