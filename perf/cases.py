"""Performance cases of the RSST step: what users of the library run, from the
1D validation line to the 16.8 M-cell shear layer, in every precision, with
the batch and the discrete adjoint.

A pass is one run segment as a program drives it: load a state, advance it,
read the new state back (``Solver``, ``BatchSolver``, ``rsst_run``).  Float64
and double-float runs keep float64 snapshots.  A float32-perturbation run's
snapshot is what such a run holds: the perturbation about the background (the
full state without one), in float32.

``exact`` is the same scheme in plain torch float64 (arXiv:1812.04135,
Sec. 4.2: MUSCL with the monotonized-central limiter, local Lax-Friedrichs
with c_tot = |V| + a/xi, SSP-RK2; reduced tendencies of Sec. 3.2 and App. A,
force of App. B).
"""
import math

import numpy as np
import torch

from paper_1812_04135_gb300 import rsst

GAMMA = 5.0 / 3.0
CFL = 0.4


def _case(kind, n, precision, steps, variant="pvs", xi=30.0, **more):
    """kind: which initial state; n: cells (nx, ny, nz), 0 on unused axes."""
    n = tuple(n) + (0,) * (3 - len(n))
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "precision": precision, "steps": steps, "variant": variant,
         "xi": xi, "contrast": 10.0, "cmax": 0.0, "covolume": 0.0, "cfl_rule": 0, "fixed_dt": False, "runs": 0, "every": 0}
    c.update(more)
    return c


def listed():
    def named(name, *a, **k):
        return dict(_case(*a, **k), name=name)

    return [
        # the smallest run: the 1D sound wave that validates a form's wave speed (launches and latency only)
        named("sound1d_256_fp64", "sound", (256,), "fp64", 128, xi=10.0),
        # a small grid of the convergence study (oblique wave, fixed dt): a few tiles, latency again
        named("wave2d_64_fp64", "wave", (64, 64), "fp64", 64, xi=5.0, fixed_dt=True),
        # the headline configuration: float64 shear layer, density ratio 10
        named("shear2d_512_fp64", "shear", (512, 512), "fp64", 32),
        # Rayleigh-Taylor under gravity between walls, the C_max law, a size that no tile divides
        named("rt2d_250_fp64_cmax", "rt", (250, 250), "fp64", 32, variant="pms", xi=1.0, cmax=4.0),
        # stratified convection box in 3D, contrast 100, float64
        named("box3d_256x128x128_fp64", "box", (256, 128, 128), "fp64", 4, xi=50.0, contrast=100.0),
        # double-float: float64-grade results at a fraction of the float64 step's cost
        named("shear2d_512_df", "shear", (512, 512), "fp64_df", 32),
        # the same in 3D, ragged on every axis
        named("box3d_90x70x50_df", "box", (90, 70, 50), "fp64_df", 16, variant="pms", xi=20.0, contrast=20.0),
        # the largest single run: float32 perturbation, state far beyond L2
        named("shear2d_4096_fp32", "shear", (4096, 4096), "fp32_pert", 16),
        # Rayleigh-Taylor production grid of medium size in float32, ragged
        named("rt2d_1000_fp32", "rt", (1000, 1000), "fp32_pert", 32, variant="pms", xi=10.0),
        # stratified convection box in float32, at a moderate reduction: the step divides dP/dt by xi^2 by subtraction, so a
        # float32 run's own round-off grows as xi^2
        named("box3d_256x128x128_fp32", "box", (256, 128, 128), "fp32_pert", 16, xi=20.0, contrast=100.0),
        # a parameter study: 64 shear layers of uneven size, xi and density ratio, advanced together
        named("batch_64_fp32", "batch", (), "fp32_pert", 32, runs=64),
        # sensitivities: forward run and reverse sweep of the discrete adjoint with checkpoints
        named("adjoint2d_256", "adjoint", (256, 256), "fp64", 40, xi=20.0, contrast=20.0, every=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sound", "wave", "shear", "shear", "rt", "rt", "box2", "box", "box", "batch", "adjoint"])
    pform = rng.choice(["pvs", "pvs", "pms", "pd"])  # the density-reduced forms blow up on large density ratios
    precision = rng.choice(["fp64", "fp64", "fp64_df", "fp32_pert", "fp32_pert"])
    law = {"cmax": rng.choice([0.0, 0.0, 0.0, 1.0]), "cfl_rule": rng.choice([0, 0, 0, 1])}
    # cells x steps that a pass may advance, per precision
    cap = {"fp64": 12e6, "fp64_df": 30e6, "fp32_pert": 200e6}[precision]
    if kind == "sound":
        return _case(kind, (_log(rng, 16, 16384),), precision, rng.randrange(17, 129),
                     variant=rng.choice(["euler", "dvs", "pvs", "dms", "pms", "pd"]), xi=rng.choice([1.0, 3.0, 10.0]))
    if kind == "wave":
        n = _log(rng, 16, 256)
        return _case(kind, (n, n), "fp64", rng.randrange(8, 65), variant=rng.choice(["dvs", "pvs", "dms", "pms", "pd"]),
                     xi=5.0, fixed_dt=True)
    if kind == "shear":
        most = {"fp64": 1024, "fp64_df": 1536, "fp32_pert": 4096}[precision]
        nx, ny = _log(rng, 48, most), _log(rng, 48, most)
        steps = max(2, min(rng.randrange(8, 40), int(cap / (nx * ny))))
        gas = {"covolume": 0.02} if precision == "fp64" and rng.random() < 0.25 else {}
        return _case(kind, (nx, ny), precision, steps, variant=pform, xi=rng.choice([1.0, 3.0, 10.0, 30.0]),
                     contrast=rng.choice([1.0, 3.0, 10.0]), **law, **gas)
    if kind in ("rt", "box2"):
        most = {"fp64": 768, "fp64_df": 1024, "fp32_pert": 2048}[precision]
        n = _log(rng, 40, most)
        m = n if kind == "rt" else _log(rng, 40, most)
        steps = max(2, min(rng.randrange(8, 40), int(cap / (n * m))))
        if law["cmax"] and kind == "rt":
            law["cmax"] = 4.0
        return _case(kind, (n, m), precision, steps, variant=pform, xi=rng.choice([3.0, 10.0, 20.0]), contrast=20.0, **law)
    if kind == "box":
        nx, ny, nz = _log(rng, 16, 200), _log(rng, 16, 200), _log(rng, 40, 160)
        steps = max(1, min(rng.randrange(4, 24), int(cap / (nx * ny * nz))))
        return _case(kind, (nx, ny, nz), precision, steps, variant=pform,
                     xi=rng.choice([5.0, 10.0, 20.0] if precision == "fp32_pert" else [10.0, 20.0, 50.0]),
                     contrast=rng.choice([20.0, 100.0]), **law)
    if kind == "batch":
        return _case(kind, (), "fp32_pert", rng.randrange(4, 25), variant=pform, runs=rng.randrange(3, 49))
    return _case(kind, (_log(rng, 40, 256), _log(rng, 40, 256)), "fp64", rng.randrange(6, 33), variant=pform,
                 xi=rng.choice([5.0, 20.0]), contrast=20.0, every=rng.randrange(3, 17))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _rand(gen, *shape):
    return torch.rand(shape, generator=gen, dtype=torch.float64, device="cuda") * 2.0 - 1.0


def _centres(n, length=1.0, ghosts=0):
    return (np.arange(-ghosts, n + ghosts) + 0.5) * (length / n)


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _pack(rho, vel, p, covolume=0.0):
    v2 = sum(v * v for v in vel)
    e = p * (1.0 - covolume * rho) / (GAMMA - 1.0)
    return torch.stack([rho] + [rho * v for v in vel] + [e + 0.5 * rho * v2])


def _polytrope(z, contrast):
    top = 0.4 / (contrast ** (2.0 / 3.0) - 1.0)
    theta = top + 0.4 * (1.0 - z)
    rho = (theta / top) ** 1.5
    return rho, rho * theta


def _problem(c, seed):
    """(run description as ``rsst.Solver`` takes it, initial state)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n = [v for v in (c["nx"], c["ny"], c["nz"]) if v]
    w = {"ndim": len(n), "n": tuple(n), "dx": tuple(1.0 / v for v in n), "gamma": GAMMA, "xi": c["xi"],
         "variant": c["variant"], "bc": ("periodic",) * len(n), "grav": (0.0, 0.0, 0.0), "vertical": -1, "bg_rho": None,
         "bg_p": None, "cmax": c["cmax"], "cfl_rule": c["cfl_rule"], "covolume": c["covolume"], "cfl": CFL}
    kind = "box2" if c["kind"] == "adjoint" else c["kind"]
    if kind == "sound":
        # the right-going sound eigenmode of the reduced system on a gas at rest (a = 1), any phase
        eps = 1e-6 if c["precision"] != "fp32_pert" else 1e-2
        phase = 2.0 * math.pi * float(_rand(gen, 1)[0])
        s = eps * torch.sin(2.0 * math.pi * _cuda(_centres(n[0])) + phase)
        return w, _pack(1.0 + s, [c["xi"] * s], (1.0 + GAMMA * s) / GAMMA)
    if kind == "wave":
        # oblique entropy and shear wave at 30 degrees over P = 1000
        th = math.radians(30.0)
        lx, ly = 1.0 / math.cos(th), 1.0 / math.sin(th)
        w["dx"] = (lx / n[0], ly / n[1])
        x, y = _cuda(_centres(n[0], lx))[None, :], _cuda(_centres(n[1], ly))[:, None]
        s = 1e-5 * torch.sin(2.0 * math.pi * (x * math.cos(th) + y * math.sin(th)) + 2.0 * math.pi * float(_rand(gen, 1)[0]))
        vx, vy = math.cos(th) - s * math.sin(th), math.sin(th) + s * math.cos(th)
        return w, _pack(1.0 + s, [vx, vy], torch.full_like(s, 1000.0))
    if kind == "shear":
        # dense band moving through light gas, tanh edges, velocity noise, P = 1; the profile at rest is the background
        def band(y):
            return np.tanh((y - 0.25) / 0.02) - np.tanh((y - 0.75) / 0.02)

        ratio, c_dense = c["contrast"], math.sqrt(GAMMA / c["contrast"])
        y, yg = _centres(n[1]), _centres(n[1], ghosts=2)
        w.update(vertical=1, bg_rho=1.0 + 0.5 * (ratio - 1.0) * band(yg), bg_p=np.ones(n[1] + 4))
        noise = 1e-4 * c_dense * _rand(gen, 2, n[1], n[0])
        rho = _cuda(1.0 + 0.5 * (ratio - 1.0) * band(y))[:, None].expand(n[1], n[0])
        vx = _cuda(0.01 * c_dense * (band(y) - 1.0))[:, None] + noise[0]
        return w, _pack(rho, [vx, noise[1]], torch.ones_like(rho), c["covolume"])
    if kind == "rt":
        # heavy gas over light gas between free-slip walls, P = 1000 at the top
        def rho_of(y):
            return 1.0 + 4.5 * (1.0 + np.tanh((y - 0.5) / 0.025))

        def p_of(y):
            def lncosh2(z):
                return np.abs(z) + np.log1p(np.exp(-2.0 * np.abs(z)))

            return 1000.0 + 5.5 * (1.0 - y) + 0.5 * 0.025 * 9.0 * (lncosh2(20.0) - lncosh2((y - 0.5) / 0.025))

        y, yg = _centres(n[1]), _centres(n[1], ghosts=2)
        w.update(bc=("periodic", "reflect"), grav=(0.0, -1.0, 0.0), vertical=1, bg_rho=rho_of(yg), bg_p=p_of(yg))
        amp = 0.01 * torch.sin(4.0 * math.pi * _cuda(_centres(n[0])) + math.pi * float(_rand(gen, 1)[0]))
        rho = _cuda(rho_of(y))[:, None] * (1.0 + amp[None, :] + 1e-4 * _rand(gen, n[1], n[0]))
        zero = torch.zeros_like(rho)
        return w, _pack(rho, [zero, zero], _cuda(p_of(y))[:, None].expand_as(rho))
    # hydrostatic polytrope with walls across gravity, as a convection run holds it: entropy and velocity disturbances
    # (density 1e-2 at fixed pressure, Mach 1e-2)
    nd = len(n)
    h = 1.0 / n[-1]
    z, zg = _centres(n[-1]), _centres(n[-1], ghosts=2)
    bg_rho, bg_p = _polytrope(zg, c["contrast"])
    w.update(dx=(h, h, h) if nd == 3 else (1.0 / n[0], h), bc=("periodic",) * (nd - 1) + ("reflect",),
             grav=(0.0,) * (nd - 1) + (-1.0,) + (0.0,) * (3 - nd), vertical=nd - 1, bg_rho=bg_rho, bg_p=bg_p)
    rz, pz = (_cuda(v).reshape((-1,) + (1,) * (nd - 1)) for v in _polytrope(z, c["contrast"]))
    rho = rz * (1.0 + 1e-2 * _rand(gen, *reversed(n)))
    vel = [1e-2 * torch.sqrt(GAMMA * pz / rz) * _rand(gen, *reversed(n)) for _ in n]
    return w, _pack(rho, vel, pz.expand_as(rho))


def _batch_problems(c, seed):
    """The runs of a parameter study: sizes, xi and density ratios belong to the case, the noise to the seed."""
    r = np.random.RandomState(c["runs"])
    got = []
    for i in range(c["runs"]):
        n = int(r.choice([128, 192, 256, 384, 512, 768, 1024]))
        one = _case("shear", (n, n), "fp32_pert", c["steps"], variant=c["variant"], xi=float(r.choice([1.0, 3.0, 10.0, 30.0])),
                    contrast=float(r.choice([1.0, 3.0, 10.0, 100.0])))
        got.append(_problem(one, seed * 1000 + i))
    return got


def _background(w):
    """U0 = (rho0, 0, P0 / (gamma - 1)) along the vertical axis, shaped to broadcast; None without a background."""
    if w["bg_rho"] is None:
        return None
    zero = np.zeros(w["n"][w["vertical"]])
    rows = np.stack([w["bg_rho"][2:-2]] + [zero] * w["ndim"] + [w["bg_p"][2:-2] / (GAMMA - 1.0)])
    shape = [rows.shape[0]] + [1] * w["ndim"]
    shape[w["ndim"] - w["vertical"]] = rows.shape[1]
    return _cuda(rows).reshape(shape)


def _dt_of(w, U):
    """A fixed step for a run that is compared at one time: the initial state's Courant step, rounded down."""
    return 0.9 * float(_cfl_dt(w, U))


def prepare(case, seed):
    if case["kind"] == "batch":
        probs = _batch_problems(case, seed)
        b = rsst.BatchSolver([w for w, _ in probs])
        torch.cuda.current_stream().synchronize()  # the batch runs on a stream of its own
        for i, (_, U) in enumerate(probs):
            b.set_state(i, U)
        b.autotune(3)
        return {"case": case, "batch": b, "U": [U for _, U in probs], "U0": [_background(w) for w, _ in probs]}
    w, U = _problem(case, seed)
    dt = _dt_of(w, U) if case["fixed_dt"] or case["kind"] == "adjoint" else 0.0
    st = {"case": case, "solver": rsst.Solver(w, case["precision"]), "U": U, "U0": _background(w), "dt": dt}
    if case["kind"] == "adjoint":
        st["xi"] = torch.tensor(w["xi"], dtype=torch.float64, requires_grad=True)
        st["weight"] = _weight(U)
    return st


def _weight(U):
    """Cotangent of the final state: a smooth observable, the same for every run."""
    x = torch.linspace(0.0, 2.0 * math.pi, U.shape[-1], dtype=torch.float64, device="cuda")
    y = torch.linspace(0.0, math.pi, U.shape[-2], dtype=torch.float64, device="cuda")
    k = torch.arange(1, U.shape[0] + 1, dtype=torch.float64, device="cuda").reshape(-1, 1, 1)
    return torch.cos(k * x) * torch.sin(y)[None, :, None] / (U.shape[-1] * U.shape[-2])


def _snapshot(U, U0):
    """A float32 run's snapshot: its perturbation in float32."""
    if U0 is None:
        return U.to(torch.float32)
    out = torch.empty(U.shape, dtype=torch.float32, device=U.device)
    return torch.sub(U, U0, out=out)


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        for i, U in enumerate(state["U"]):
            b.set_state(i, U)
        b.step(case["steps"])
        # get_state returns when the run's state is complete
        return [_snapshot(b.get_state(i), U0) for i, U0 in enumerate(state["U0"])]
    s = state["solver"]
    if case["kind"] == "adjoint":
        U = state["U"].requires_grad_(True)
        UN = rsst.rsst_run(U, state["xi"], s, state["dt"], case["steps"], case["every"])
        gU, gxi = torch.autograd.grad(UN, [U, state["xi"]], grad_outputs=state["weight"])
        return {"state": UN.detach(), "dJ_dU": gU, "dJ_dxi": gxi}
    s.set_state(state["U"])
    s.step(case["steps"], state["dt"])
    U = s.get_state()
    return _snapshot(U, state["U0"]) if case["precision"] == "fp32_pert" else U


def work(case):
    """Bytes: the caller's float64 state in, the snapshot out, and the run's state read and written once a step
    (the next step's dt needs the whole state).  Operations: the scheme's float count per cell and stage (2D: two faces
    of 128 and 53 for the cell), the adjoint's forward, recompute and reverse together."""
    if case["kind"] == "batch":
        r = np.random.RandomState(case["runs"])
        cells = 0
        for _ in range(case["runs"]):
            cells += int(r.choice([128, 192, 256, 384, 512, 768, 1024])) ** 2
            r.choice([1.0, 3.0, 10.0, 30.0]), r.choice([1.0, 3.0, 10.0, 100.0])
        nd = 2
    else:
        n = [v for v in (case["nx"], case["ny"], case["nz"]) if v]
        cells, nd = math.prod(n), len(n)
    nv = nd + 2
    per = {1: 143, 2: 309, 3: 530}[nd]
    size = 4 if case["precision"] == "fp32_pert" else 8
    if case["kind"] == "adjoint":
        # in, out, cotangent, gradient; every step's state written and read again by the reverse sweep
        return {"bytes": float(cells * nv * 8 * (4 + 4 * case["steps"])), "flops": float(1471 * cells * 2 * case["steps"])}
    return {"bytes": float(cells * nv * (8 + size + 2 * size * case["steps"])), "flops": float(per * cells * 2 * case["steps"])}


# ---------------------------------------------------------------------------
# The same scheme in plain torch float64
# ---------------------------------------------------------------------------

def _prims(w, q):
    b = w["covolume"]
    rho = q[0]
    v = [m / rho for m in q[1:-1]]
    v2 = sum(x * x for x in v)
    p = (GAMMA - 1.0) * (q[-1] - 0.5 * rho * v2)
    if b:
        p = p / (1.0 - b * rho)
    a2 = GAMMA * p / rho
    if b:
        a2 = a2 / (1.0 - b * rho)
    return rho, v, v2, p, a2


def _xi_of(w, a2):
    return (1.0 + (a2 / w["cmax"] ** 2) ** 2) ** 0.25 if w["cmax"] else w["xi"]


def _ctot(w, v2, a2):
    moving = v2 > 0.0
    return torch.sqrt(torch.where(moving, v2, torch.ones_like(v2))) * moving + torch.sqrt(a2) / _xi_of(w, a2)


def _cfl_dt(w, q):
    rho, v, v2, p, a2 = _prims(w, list(q))
    c = _ctot(w, v2, a2).max()
    rates = [1.0 / h for h in w["dx"][:w["ndim"]]]
    return CFL / (c * (max(rates) if w["cfl_rule"] else sum(rates)))


def _mc(a, b):
    """Zero for opposite signs, else the smallest of 2a, 2b, (a+b)/2."""
    s = torch.where(a.abs() <= b.abs(), a, b) * 2.0
    m = 0.5 * (a + b)
    s = torch.where(s.abs() <= m.abs(), s, m)
    return torch.where(a * b > 0.0, s, torch.zeros_like(s))


def _with_ghosts(w, q, d):
    ax = w["ndim"] - d  # axis of dimension d in [nvar, ...]
    n = q.shape[ax]
    first, last = q.narrow(ax, 0, 2), q.narrow(ax, n - 2, 2)
    if w["bc"][d] == "periodic":
        return torch.cat([last, q, first], ax), ax
    sign = torch.ones([q.shape[0]] + [1] * w["ndim"], dtype=q.dtype, device=q.device)
    sign[1 + d] = -1.0
    lo, hi = first.flip(ax) * sign, last.flip(ax) * sign
    if w["vertical"] == d:
        r, p = _cuda(w["bg_rho"]), _cuda(w["bg_p"])
        e = p * (1.0 - w["covolume"] * r) / (GAMMA - 1.0)
        u0 = torch.stack([r] + [torch.zeros_like(r)] * w["ndim"] + [e])
        view = [q.shape[0]] + [1] * w["ndim"]
        view[ax] = 2
        lo = lo + (u0[:, 0:2] - u0[:, 2:4].flip(1)).reshape(view)
        hi = hi + (u0[:, n + 2:n + 4] - u0[:, n:n + 2].flip(1)).reshape(view)
    return torch.cat([lo, q, hi], ax), ax


def _flux(w, q, d):
    q = list(q)
    rho, v, v2, p, a2 = _prims(w, q)
    f = [q[1 + d]] + [m * v[d] + p if e == d else m * v[d] for e, m in enumerate(q[1:-1])] + [(q[-1] + p) * v[d]]
    return torch.stack(f), _ctot(w, v2, a2)


def _rhs(w, q, xi=None):
    """L(q); ``xi``: a tensor in place of the run's rate (for its derivative)."""
    w = w if xi is None else dict(w, xi=xi)
    dU = torch.zeros_like(q)
    for d in range(w["ndim"]):
        g, ax = _with_ghosts(w, q, d)
        n = q.shape[ax]
        diff = g.narrow(ax, 1, n + 3) - g.narrow(ax, 0, n + 3)
        s = 0.5 * _mc(diff.narrow(ax, 0, n + 2), diff.narrow(ax, 1, n + 2))
        mid = g.narrow(ax, 1, n + 2)
        left, right = (mid + s).narrow(ax, 0, n + 1), (mid - s).narrow(ax, 1, n + 1)
        fl, cl = _flux(w, left, d)
        fr, cr = _flux(w, right, d)
        f = 0.5 * (fl + fr) - 0.5 * torch.where(cl >= cr, cl, cr) * (right - left)
        dU = dU - (f.narrow(ax, 1, n) - f.narrow(ax, 0, n)) / w["dx"][d]
    rows = list(dU)
    var = w["variant"]
    if var != "euler":
        b = w["covolume"]
        rho, v, v2, p, a2 = _prims(w, list(q))
        e = p * (1.0 - b * rho) / (GAMMA - 1.0)
        xi2 = _xi_of(w, a2) ** 2
        f = 1.0 - 1.0 / xi2
        if var in ("pvs", "pms", "pd"):
            vdm = sum(x * m for x, m in zip(v, rows[1:-1]))
            s = ((0.5 * v2 + b * p / (GAMMA - 1.0)) * rows[0] - vdm + rows[-1]) * (GAMMA - 1.0) / (1.0 - b * rho)
            k = 1.0 / a2
        else:
            s, k = rows[0], torch.ones_like(rho)
        if var == "pd":
            rows[-1] = rows[-1] - f * s * (1.0 - b * rho) / (GAMMA - 1.0)
        else:
            moves = var in ("pvs", "dvs")
            h = (e + p + (0.5 if moves else -0.5) * rho * v2) / rho
            rows[0] = rows[0] - f * s * k
            if moves:
                rows[1:-1] = [m - f * s * k * x for m, x in zip(rows[1:-1], v)]
            rows[-1] = rows[-1] - f * s * k * h
    for d in range(w["ndim"]):
        if w["grav"][d]:
            rows[1 + d] = rows[1 + d] + q[0] * w["grav"][d]
            rows[-1] = rows[-1] + q[1 + d] * w["grav"][d]
    return torch.stack(rows)


def _step(w, q, dt, xi=None):
    star = q + dt * _rhs(w, q, xi)
    return 0.5 * q + 0.5 * (star + dt * _rhs(w, star, xi))


def _advance(w, q, steps, dt):
    with torch.no_grad():
        for _ in range(steps):
            q = _step(w, q, dt if dt > 0.0 else _cfl_dt(w, q))
    return q


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for w, U in _batch_problems(case, seed):
            out.append(_advance(w, U, case["steps"], 0.0) - _background(w))
        return out
    w, U = _problem(case, seed)
    if case["kind"] == "adjoint":
        dt, every, steps = _dt_of(w, U), case["every"], case["steps"]
        marks = [U]
        for s in range(0, steps, every):
            marks.append(_advance(w, marks[-1], min(every, steps - s), dt))
        lam, gxi = _weight(U), 0.0
        for i in reversed(range(len(marks) - 1)):
            xi = torch.tensor(w["xi"], dtype=torch.float64, device="cuda", requires_grad=True)
            q0 = marks[i].detach().requires_grad_(True)
            q = q0
            for _ in range(min(every, steps - i * every)):
                q = _step(w, q, dt, xi)
            lam, g = torch.autograd.grad(q, [q0, xi], grad_outputs=lam)
            gxi = gxi + g
        return {"state": marks[-1], "dJ_dU": lam, "dJ_dxi": gxi.cpu()}
    q = _advance(w, U, case["steps"], _dt_of(w, U) if case["fixed_dt"] else 0.0)
    if case["precision"] == "fp32_pert":
        U0 = _background(w)
        return q if U0 is None else q - U0
    return q
