"""Single device helpers (rsst_math_eval) at the values where their bit
arithmetic is tight, against numpy in float64."""
import numpy as np
import pytest

from paper_1812_04135_gb300 import rsst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import os
    if not os.path.exists(rsst.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    rsst.lib()


def significands(low, exponent=0):
    """Every leading 24-bit significand with the given 29 low bits, times 2^exponent."""
    return np.ldexp(1.0 + (np.arange(1 << 23) * 2.0 ** 29 + low) * 2.0 ** -52, exponent)


LOWS = [0, 1, (1 << 28) - 1, 1 << 28, (1 << 29) - 1]


@pytest.mark.parametrize("low", LOWS)
@pytest.mark.parametrize("exponent", [0, -700])
def test_reciprocal_at_every_leading_significand(low, exponent):
    x = significands(low, exponent)
    got, want = rsst.rsst_math_eval("rcp", x), 1.0 / x
    assert np.abs(got.view(np.int64) - want.view(np.int64)).max() <= 1


def test_pair_to_double_rounds_the_sum():
    """The nearest double of h + l, powers of two (the unit below them is half) among the h."""
    rng = np.random.default_rng(5)
    e = rng.integers(-70, 120, 1 << 20)
    h = np.ldexp(1.0 + rng.integers(0, 1 << 23, e.size) * 2.0 ** -23 * (rng.random(e.size) < 0.5), e).astype(np.float32)
    below = np.where(np.frexp(h)[0] == 0.5, 0.25, 0.5)
    l = (rng.uniform(-1.0, 1.0, e.size) * 2.0 ** -rng.integers(0, 30, e.size) * below * np.spacing(h)).astype(np.float32)
    got = rsst.rsst_math_eval("pair_to_double", h, l)
    assert np.array_equal(got, h.astype(np.float64) + l.astype(np.float64))


@pytest.mark.parametrize("low", LOWS)
@pytest.mark.parametrize("exponent", [0, 1, -2])
def test_adjoint_speeds_at_every_leading_significand(low, exponent):
    x = significands(low, exponent)
    s = np.sqrt(x)
    # the root's pair 2^-42; its reciprocal's seed error 2^-22 squared and its roundings 2^-45 on top
    assert np.abs(rsst.rsst_math_eval("speed", x) / s - 1.0).max() <= 2.0 ** -42
    assert np.abs(rsst.rsst_math_eval("inv_speed", x) * s - 1.0).max() <= 2.0 ** -41


def test_adjoint_speeds_at_any_magnitude():
    """The derivative of |V| is V/|V| however small the speed."""
    x = np.ldexp(1.0 + np.random.default_rng(6).random(1 << 16), np.linspace(-1021, 1022, 1 << 16).astype(int))
    s = np.sqrt(x)
    assert np.abs(rsst.rsst_math_eval("speed", x) / s - 1.0).max() <= 2.0 ** -42
    assert np.abs(rsst.rsst_math_eval("inv_speed", x) * s - 1.0).max() <= 2.0 ** -41
    assert np.array_equal(rsst.rsst_math_eval("speed", [0.0, 5e-324]), [0.0, 0.0])
    assert np.array_equal(rsst.rsst_math_eval("inv_speed", [0.0, 5e-324]), [0.0, 0.0])


def mc(a, b):
    s = np.where((np.abs(a) <= np.abs(b)) & (4 * np.abs(a) <= np.abs(a + b)), 2 * a,
                 np.where(4 * np.abs(b) <= np.abs(a + b), 2 * b, 0.5 * (a + b)))
    return np.where((np.sign(a) * np.sign(b)) > 0, s, 0.0)


@pytest.mark.parametrize("fn,factor", [("mc_slope", 1.0), ("half_mc", 0.5)])
def test_limiter_next_to_the_subnormal_range(fn, factor):
    """Differences in the far tail of a profile: no sign or exponent wraps (the values are exact up to the smallest
    normal number)."""
    rng = np.random.default_rng(7)
    e = rng.integers(-1074, -1000, (2, 1 << 16))
    a, b = np.ldexp(rng.uniform(0.5, 1.0, e.shape), e) * rng.choice([-1.0, 1.0], e.shape)
    got = rsst.rsst_math_eval(fn, a, b)
    assert np.abs(got - factor * mc(a, b)).max() <= 2.0 ** -1022


def test_wave_speed_pair_accuracy():
    """|V| + a/xi from rho |V|^2, P and 1/rho.  Each square is a product of float pairs (2^-45: the two low parts'
    product 2^-46 and two roundings 2^-47), halved by the root; a root's correction of 2^-22.4 has three
    roundings (2^-44.8); the pairs' sum one (2^-46).  Together below 2^-43.7."""
    rng = np.random.default_rng(8)
    worst = 0.0
    for _ in range(8):
        n = 1 << 22
        rho, P = np.exp(rng.uniform(-7, 7, n)), np.exp(rng.uniform(-7, 7, n))
        ir = 1.0 / rho
        k = P * np.exp(rng.uniform(-25, 5, n)) * (rng.random(n) < 0.9)
        gx = 5.0 / 3.0 / 900.0
        want = np.sqrt(k * ir) + np.sqrt(gx * (P * ir))
        worst = max(worst, np.abs(rsst.rsst_math_eval("ctot", k, P, ir) / want - 1.0).max())
    assert worst <= 2.0 ** -43.7, np.log2(worst)


def test_cmax_wave_speed_at_any_magnitude():
    """The C_max law's c_tot: float64-accurate in its sound term, |V| to 2^-42, over the range of float64."""
    rng = np.random.default_rng(9)
    n = 1 << 16
    x = np.ldexp(1.0 + rng.random(n), np.linspace(-1000, 1000, n).astype(int))
    zero = np.zeros(n)
    assert np.abs(rsst.rsst_math_eval("ctot_cmax", zero, x) / np.sqrt(x) - 1.0).max() <= 2.0 ** -52
    assert np.abs(rsst.rsst_math_eval("ctot_cmax", x, zero) / np.sqrt(x) - 1.0).max() <= 2.0 ** -42
    assert rsst.rsst_math_eval("rsqrt", [np.inf])[0] == 0.0


def test_double_float_flux_of_a_small_difference():
    """States that agree in their leading floats: the dissipation alpha (rho_L - rho_R) keeps its relative accuracy
    (the speed 2^-44, the product 2^-46)."""
    rng = np.random.default_rng(10)
    n = 1 << 18
    hi = (1.0 + rng.random(n)).astype(np.float32).astype(np.float64)
    low = rng.integers(-(1 << 22), 1 << 22, (2, n)) * 2.0 ** -47
    rl, rr, E = hi + low[0], hi + low[1], 1.0 + rng.random(n).astype(np.float32)
    got = rsst.rsst_math_eval("df_flux", rl, rr, E)
    want = np.sqrt(E / np.minimum(rl, rr)) * (rl - rr)
    assert (np.abs(got - want) <= 2.0 ** -43 * np.abs(want)).all()


def test_float32_pair_pressure_tendency_rounds_once_at_the_energy_tendency():
    """dP/(gamma - 1) = |V|^2/2 drho - V.dm + dE with small first terms: their roundings (2^-22 of at most 2^-5 dE
    together) and one of dE's size."""
    rng = np.random.default_rng(11)
    n = 1 << 20
    f = np.float32
    mx, my, dr, dx, dy = (rng.uniform(-0.125, 0.125, n).astype(f) for _ in range(5))
    dE = (rng.choice([-1.0, 1.0], n) * (1.0 + rng.random(n))).astype(f)
    got = rsst.rsst_math_eval("pair_tendency", np.ones(n), mx, my, dr, dx, dy, dE)
    mx, my, dr, dx, dy, dE = (v.astype(np.float64) for v in (mx, my, dr, dx, dy, dE))
    want = 0.5 * (mx * mx + my * my) * dr - (mx * dx + my * dy) + dE
    half_ulp = 0.5 * np.spacing(np.abs(want).astype(f)).astype(np.float64)
    assert (np.abs(got - want) <= half_ulp + 2.0 ** -22 * 2.0 ** -5).all()


def test_float32_pair_speed_difference_rounds_one_product():
    """c_tot - c_tot0 of a state whose P1 rho0 and P0 rho1 nearly cancel: one of the products is rounded (2^-24 of
    it), the other goes into the sum exactly; 2^-20 of the result for everything after."""
    rng = np.random.default_rng(12)
    n = 1 << 20
    f = np.float32
    r0, P0, r1 = ((1.0 + rng.random(n)).astype(f) for _ in range(3))
    r1 = (r1 * f(0.25)).astype(f)
    P1 = (P0 * r1 / r0 * (1.0 + rng.uniform(-1.0, 1.0, n) * 2.0 ** -10)).astype(f)
    got = rsst.rsst_math_eval("pair_dc", r1, P1, r0, P0)
    r0, P0, r1, P1 = (v.astype(np.float64) for v in (r0, P0, r1, P1))
    rho, P = r0 + r1, P0 + P1
    a, a0 = np.sqrt(P / rho), np.sqrt(P0 / r0)
    diff = P1 * r0 - P0 * r1
    want = diff / (rho * r0) / (a + a0)
    bound = 2.0 ** -24 * np.maximum(P1 * r0, P0 * r1) * 1.01 / (rho * r0) / (a + a0) + 2.0 ** -20 * np.abs(want)
    assert (np.abs(got - want) <= bound).all()
