"""Workloads of the library's public entry points, with their inputs, their unavoidable
work and their results in plain 64-bit arithmetic.

A case names one call sequence of a user's program: advancing one lattice
(`Simulation`), a batch of lattices (`Batch`), a differentiable rollout
(`adjoint.rollout`) or the finite-difference solver (`FDSolver`). Sizes and parameters
are those of the package's sweeps, tests and benchmark. `exact` restates the method
(equation of state, step, gradient, finite-difference scheme) in float64 torch.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2107_06355_gb300 as P
from paper_2107_06355_gb300 import adjoint as A

MODES = {"cs": P.EOS_CS, "smooth": P.EOS_SMOOTH, "peng": P.EOS_PENG}
BETA = 4.6  # tanh factor of the paper's interface profiles
DEV = "cuda"


# ---- the cases ---------------------------------------------------------------------


def listed():
    return [
        # The smallest use: one 256 x 4 planar interface relaxed in a single context (the
        # coexistence configuration, T_r = 0.8). 1,024 nodes: launches and latency count.
        dict(name="planar_256x4", kind="single", shape="planar", nx=256, ny=4, walls=False, eos="smooth", Tr=0.8,
             a_l=0.5, a_v=0.5, alpha=0.342, relax="unit", forcing="li", kappa=0.0, W=8.0, steps=100),
        # The paper's coexistence sweep: (2, 200) planar interfaces over T_r, equations of
        # state and forcing schemes, stepped 100 at a time between convergence checks.
        dict(name="coexistence_sweep", kind="planar_sweep", n=24, nx=2, ny=200, steps=100),
        # Six independent relaxation times on an odd-sized droplet (general MRT collision).
        dict(name="mrt_droplet_257x131", kind="single", shape="droplet", nx=257, ny=131, walls=False, eos="smooth",
             Tr=0.6, a_l=0.387, a_v=2.0, alpha=0.834, relax="mrt", forcing="li", kappa=0.0, W=8.0, steps=50),
        # A static droplet as users run them for Laplace or spurious-current checks.
        dict(name="droplet_512", kind="single", shape="droplet", nx=512, ny=512, walls=False, eos="smooth", Tr=0.6,
             a_l=0.387, a_v=2.0, alpha=0.834, relax="unit", forcing="li", kappa=0.0, W=8.0, steps=50),
        # The paper's droplet impact on a film (600 x 250, walls, tau(rho), Sec. IV).
        dict(name="impact_600x250", kind="single", shape="impact", nx=600, ny=250, walls=True, eos="smooth", Tr=0.5,
             a_l=0.363, a_v=2.0, alpha=0.775, relax="two_phase", forcing="li", kappa=0.0, W=7.0, steps=50),
        # The large droplet impact (2048 x 1024, T_r = 0.35, density ratio 7.9e4).
        dict(name="impact_2048x1024", kind="single", shape="impact", nx=2048, ny=1024, walls=True, eos="smooth",
             Tr=0.35, a_l=0.363, a_v=2.0, alpha=0.838, relax="two_phase", forcing="li", kappa=0.0, W=6.0, steps=20),
        # Laplace-law droplets with and without the surface-tension control, one batch.
        dict(name="laplace_kappa", kind="batch", shape="droplet", n=6, lmin=192, lmax=192, eos="smooth", Tr=0.6,
             a_l=0.387, a_v=2.0, alpha=0.834, relax="unit", kappa=0.5, W=8.0, steps=50, plan="auto", size_seed=0),
        # The stability study: droplet impacts over T_r and viscosity ratio, one isolated
        # batch on the graph plan with a guard per check.
        dict(name="stability_study", kind="impact_sweep", n=35, nx=600, ny=250, steps=20),
        # The 64-lattice sweep of uneven sizes from host densities to host densities.
        dict(name="sweep_64", kind="host_sweep", n=64, lmin=64, lmax=1024, steps=50, size_seed=210706355),
        # Gradients in the initial density and alpha through a stored 256^2 rollout.
        dict(name="adjoint_256", kind="adjoint", shape="droplet", nx=256, ny=256, walls=False, eos="smooth", Tr=0.5,
             a_l=0.363, a_v=2.0, alpha=0.775, relax="unit", kappa=0.0, W=8.0, steps=400, interval=0, param="alpha"),
        # Gradients in the initial density and kappa through a checkpointed walled
        # two-phase rollout with the surface-tension source.
        dict(name="adjoint_walls_kappa", kind="adjoint", shape="impact", nx=300, ny=125, walls=True, eos="smooth",
             Tr=0.5, a_l=0.363, a_v=2.0, alpha=0.775, relax="two_phase", kappa=0.2, W=7.0, steps=100, interval=10,
             param="kappa"),
        # The paper's finite-difference reference of the impact (dx = 1/2, dt = 0.8 dx^2).
        dict(name="fd_impact_1200x500", kind="fd", nx=1200, ny=500, walls=True, eos="smooth", Tr=0.5, a_l=0.363,
             a_v=2.0, alpha=0.775, tau_nu=0.7, tau_e=1.0, dx=0.5, dt=0.2, vary=False, kappa=0.0, W=7.0, steps=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single"] * 4 + ["batch"] * 2 + ["adjoint", "fd", "planar_sweep", "host_sweep"])
    eos = rng.choice([dict(eos="smooth", Tr=0.6, a_l=0.387, a_v=2.0, alpha=0.834),
                      dict(eos="smooth", Tr=0.5, a_l=0.363, a_v=2.0, alpha=0.775),
                      dict(eos="cs", Tr=round(rng.uniform(0.6, 0.8), 3), a_l=0.387, a_v=0.387, alpha=0.5)])
    if kind == "single":
        shape = rng.choice(["planar", "droplet", "droplet", "impact"])
        ny = rng.choice([2, 4, 5]) if shape == "planar" else _log_int(rng, 40, 1400)
        nx = _log_int(rng, 64, 1024) if shape == "planar" else max(40, min(2048, int(ny * rng.uniform(0.7, 2.5))))
        relax = rng.choice(["unit", "unit", "two_phase", "two_phase", "mrt"])
        return dict(kind="single", shape=shape, nx=nx, ny=ny, walls=shape == "impact", relax=relax,
                    forcing="li", kappa=rng.choice([0.0, 0.0, 0.3, -0.5]), W=8.0, steps=rng.randint(10, 60), **eos)
    if kind == "batch":
        return dict(kind="batch", shape="droplet", n=rng.randint(2, 20), lmin=48, lmax=rng.randint(96, 700),
                    relax=rng.choice(["unit", "unit", "two_phase"]), kappa=rng.choice([0.0, 0.0, 0.4]), W=8.0,
                    steps=rng.randint(10, 60), plan=rng.choice(["auto", "graph"]), size_seed=rng.randint(0, 1 << 30),
                    **eos)
    if kind == "planar_sweep":
        return dict(kind="planar_sweep", n=rng.randint(4, 33), nx=rng.choice([1, 2, 4]), ny=2 * rng.randint(80, 150),
                    steps=rng.randint(20, 150))
    if kind == "host_sweep":
        return dict(kind="host_sweep", n=rng.randint(3, 40), lmin=64, lmax=rng.randint(100, 1024),
                    steps=rng.randint(10, 50), size_seed=rng.randint(0, 1 << 30))
    if kind == "adjoint":
        two = rng.random() < 0.5
        return dict(kind="adjoint", shape="impact" if two else "droplet", nx=_log_int(rng, 60, 512),
                    ny=_log_int(rng, 60, 256), walls=two, relax="two_phase" if two else "unit",
                    kappa=rng.choice([0.0, 0.3]), W=8.0, steps=rng.randint(20, 120), interval=rng.choice([0, 0, 8]),
                    param=rng.choice(["alpha", "kappa"]), eos="smooth", Tr=0.6, a_l=0.387, a_v=2.0, alpha=0.834)
    walls = rng.random() < 0.5
    return dict(kind="fd", nx=_log_int(rng, 64, 2048), ny=_log_int(rng, 64, 1024), walls=walls, tau_nu=0.8, tau_e=1.0,
                dx=0.5, dt=0.1, vary=rng.random() < 0.4, kappa=rng.choice([0.0, 0.3]), W=8.0, steps=rng.randint(4, 12),
                eos="smooth", Tr=0.6, a_l=0.387, a_v=2.0, alpha=0.834)


# ---- what a case consists of ---------------------------------------------------------


def _instances(case):
    """The lattices of a case: one dict per lattice with the keys of a "single" case."""
    k = case["kind"]
    if k in ("single", "adjoint"):
        return [case]
    if k == "batch":
        rs = np.random.RandomState(case["size_seed"] % (1 << 31))
        out = []
        for i in range(case["n"]):
            nx = int(rs.randint(case["lmin"], case["lmax"] + 1))
            ny = nx if i % 2 == 0 else int(rs.randint(case["lmin"], case["lmax"] + 1))
            kappa = case["kappa"] * (1.0, 0.0, -0.6)[i % 3]
            out.append(dict(case, nx=nx, ny=ny, walls=False, kappa=kappa, forcing="li",
                            R=min(nx, ny) / (8.0, 6.0, 4.0)[i % 3]))
        return out
    if k == "planar_sweep":
        out = []
        for i in range(case["n"]):
            v = i % 4
            e = (dict(eos="cs", Tr=0.7 + 0.2 * i / max(1, case["n"] - 1), a_l=0.5, a_v=0.5, alpha=0.5, forcing="li"),
                 dict(eos="smooth", Tr=0.5, a_l=0.5, a_v=0.5, alpha=(0.610, 0.342, 0.216)[i % 3], forcing="li"),
                 dict(eos="smooth", Tr=0.5, a_l=0.5, a_v=2.0, alpha=(0.554, 0.322, 0.207)[i % 3], forcing="li"),
                 dict(eos="peng", Tr=0.7, a_l=0.387, a_v=0.387, alpha=0.5, forcing="guo"))[v]
            out.append(dict(kind="single", shape="planar_y", nx=case["nx"], ny=case["ny"], walls=False, relax="unit",
                            kappa=0.0, W=18.0 if v == 3 else 10.0, steps=case["steps"], **e))
        return out
    if k == "impact_sweep":
        return [dict(kind="single", shape="impact", nx=case["nx"], ny=case["ny"], walls=True, eos="cs",
                     Tr=(0.45, 0.5, 0.55, 0.6, 0.65)[i % 5], a_l=0.363, a_v=0.363, alpha=0.5, relax="two_phase",
                     forcing="li", visc_ratio=float(2 + 2 * (i // 5)), kappa=0.0, W=7.0, steps=case["steps"])
                for i in range(case["n"])]
    if k == "host_sweep":
        L = np.random.default_rng(case["size_seed"]).integers(case["lmin"], case["lmax"] + 1, size=case["n"])
        return [dict(kind="single", shape="droplet" if i % 2 else "planar_y", nx=int(L[i]) if i % 2 else 4,
                     ny=int(L[i]), R=L[i] / 4.0, walls=False, eos="smooth", Tr=0.35 + 0.6 * i / max(1, case["n"] - 1),
                     a_l=0.363, a_v=2.0, alpha=0.775, relax="unit", forcing="li", kappa=0.0, W=8.0,
                     steps=case["steps"]) for i in range(case["n"])]
    raise ValueError(k)


def _eos_params(c):
    return P.EOSParams(MODES[c["eos"]], c["Tr"], c["a_l"], c["a_v"], c["alpha"], r_theta=0.45 if c["eos"] == "peng" else 0.0)


MRT = dict(tau_rho=1.0, tau_e=1.1, tau_zeta=0.9, tau_j=1.0, tau_q=1.2, tau_nu=0.8)


def _relax(c):
    forcing = P.FORCING_GUO if c.get("forcing") == "guo" else P.FORCING_LI
    if c["relax"] == "two_phase":
        return P.Relax(kind=P.RELAX_TWO_PHASE, forcing=forcing, tau_l=0.6, visc_ratio=c.get("visc_ratio", 1.5),
                       kappa=c["kappa"])
    return P.Relax(forcing=forcing, kappa=c["kappa"], **(MRT if c["relax"] == "mrt" else {}))


def _bc(c):
    return P.BC_WALLS_Y if c["walls"] else P.BC_PERIODIC


def _fields(c, seed, dx=1.0):
    """Seeded initial density and velocity of one lattice: an interface, a droplet or a
    droplet above a film between the coexistence densities, jittered in place, with a
    small relative density noise and small random velocities."""
    rv, rl = _coexistence(c["a_l"], c["Tr"])
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    u = lambda *s: torch.rand(*s, generator=g, device=DEV, dtype=torch.float64) * 2.0 - 1.0  # noqa: E731
    nx, ny, W = c["nx"], c["ny"], c["W"]
    jx, jy = u(2).tolist()
    x = torch.arange(nx, device=DEV, dtype=torch.float64)[None, :] * dx
    y = torch.arange(ny, device=DEV, dtype=torch.float64)[:, None] * dx
    zero = torch.zeros((ny, nx), device=DEV, dtype=torch.float64)
    lx, ly = nx * dx, ny * dx
    if c["shape"].startswith("planar"):
        s, n = (y, ly) if c["shape"] == "planar_y" else (x, lx)
        phi = 0.5 * (torch.tanh(BETA * (s - 0.25 * n - 0.2 * jx) / W) - torch.tanh(BETA * (s - 0.75 * n - 0.2 * jy) / W))
        along, across = 1e-3 * (2.0 + jx) + zero, 1e-4 * (2.0 + jy) + zero  # a slow uniform drift
        vx, vy = (along, across) if c["shape"] == "planar_y" else (across, along)
        return (rv + (rl - rv) * phi + zero) * (1.0 + 1e-5 * u(ny, nx)), vx, vy
    if c["shape"] == "droplet":
        R = c.get("R") or min(lx, ly) / 4.0
        r = torch.sqrt((x - 0.5 * lx - jx) ** 2 + (y - 0.5 * ly - jy) ** 2)
        phi = 0.5 * (1.0 - torch.tanh(BETA * (r - R) / W))
        vx, vy = 1e-3 * phi * jx + zero, 1e-3 * phi * jy + zero
    else:
        R, film = 0.2 * ly, 0.1 * ly
        r = torch.sqrt((x - 0.5 * lx - jx) ** 2 + (y - film - R - W) ** 2)
        drop = 0.5 * (1.0 - torch.tanh(BETA * (r - R) / W))
        phi = torch.maximum(drop, 0.5 * (1.0 - torch.tanh(BETA * (y - film) / W)))
        vx, vy = zero, -(0.05 + 0.002 * jy) * drop
    return (rv + (rl - rv) * phi) * (1.0 + 1e-5 * u(ny, nx)), vx + 0.0, vy + 0.0


# ---- prepare and run -------------------------------------------------------------------


def prepare(case, seed):
    k, inst = case["kind"], None
    if k == "fd":
        init = _fields(dict(case, shape="impact" if case["walls"] else "droplet"), seed, dx=case["dx"])
        two = dict(tau_l=case["tau_nu"], visc_ratio=2.0) if case["vary"] else {}
        fd = P.FDSolver(case["nx"], case["ny"], _eos_params(case), tau_nu=case["tau_nu"], tau_e=case["tau_e"],
                        dx=case["dx"], bc=_bc(case), kappa=case["kappa"], **two)
        return dict(case=case, init=init, sim=fd)
    inst = _instances(case)
    if k == "adjoint":
        rho0, _, _ = _fields(case, seed)
        value = case["kappa"] if case["param"] == "kappa" else case["alpha"]
        spec = A.RolloutSpec(case["nx"], case["ny"], _bc(case), _eos_params(case), _relax(case), case["steps"],
                             interval=case["interval"], param=case["param"])
        weight = torch.randn(rho0.shape, device=DEV, dtype=torch.float64,
                             generator=torch.Generator(device=DEV).manual_seed(int(seed) + 1))
        return dict(case=case, rho0=rho0, value=value, spec=spec, weight=weight)
    init = [_fields(c, int(seed) * 1009 + i) for i, c in enumerate(inst)]
    if k == "single":
        sim = P.Simulation(case["nx"], case["ny"], _bc(case), _eos_params(case), _relax(case))
        return dict(case=case, init=init[0], sim=sim)
    b = P.Batch([(c["nx"], c["ny"], _bc(c)) for c in inst], [_eos_params(c) for c in inst], [_relax(c) for c in inst])
    if k in ("planar_sweep", "impact_sweep"):
        b.set_isolation(True)
    for i, f in enumerate(init):
        b.init_equilibrium(i, *f)
    if k == "host_sweep" or case.get("plan") == "auto":
        b.autotune(10)
        if k != "host_sweep":
            for i, f in enumerate(init):
                b.init_equilibrium(i, *f)
    else:
        b.set_plan(P.PLAN_GRAPH, 0)
    st = dict(case=case, init=init, batch=b)
    if k == "host_sweep":
        st["src"] = [f[0].cpu().pin_memory() for f in init]
        st["dst"] = [torch.empty_like(t).pin_memory() for t in st["src"]]
        st["init"] = None
    elif k == "planar_sweep":
        b.guard()
    return st


def run(st):
    c = st["case"]
    k = c["kind"]
    if k == "single":
        sim = st["sim"]
        sim.init_equilibrium(*st["init"])
        sim.step(c["steps"])
        return [sim.get_f(), *sim.fields()]
    if k == "batch":  # the droplets restart from their initial fields
        b = st["batch"]
        for i, f in enumerate(st["init"]):
            b.init_equilibrium(i, *f)
        b.step(c["steps"])
        return [b.get_f(i) for i in range(b.n)]
    if k == "planar_sweep":  # the sweep's loop: the interfaces keep relaxing from pass to pass
        b = st["batch"]
        b.step(c["steps"])
        return dict(guard=b.guard(), f=[b.get_f(i) for i in range(b.n)])
    if k == "impact_sweep":
        b = st["batch"]
        for i, f in enumerate(st["init"]):
            b.init_equilibrium(i, *f)
        b.step(c["steps"])
        return dict(guard=b.guard(), f=[b.get_f(i) for i in range(b.n)])
    if k == "host_sweep":
        st["batch"].run_host(st["src"], c["steps"], st["dst"])
        return list(st["dst"])
    if k == "adjoint":
        rho0 = st["rho0"].detach().requires_grad_(True)
        theta = torch.tensor(st["value"], dtype=torch.float64, requires_grad=True)
        rho = A.rollout(rho0, theta, st["spec"])
        (rho * st["weight"]).sum().backward()
        return [rho.detach(), rho0.grad, theta.grad]
    fd = st["sim"]
    fd.set_state(*st["init"])
    fd.step(c["steps"], c["dt"])
    return list(fd.get_state())


def work(case):
    """Per node and step the nine populations are read and written once (144 bytes); the
    adjoint also reads lambda and what its state needs and writes lambda; the
    finite-difference step reads and writes rho, u twice (predictor and corrector).
    flops: the additions, products, reciprocals and square roots of the equations."""
    n = case["steps"]
    if case["kind"] == "fd":
        nodes = case["nx"] * case["ny"]
        return dict(bytes=nodes * (96.0 * n + 48.0), flops=nodes * 430.0 * n)
    nodes = sum(c["nx"] * c["ny"] for c in _instances(case))
    if case["kind"] == "adjoint":
        return dict(bytes=nodes * n * (144.0 + 32.0 + 144.0 + 32.0), flops=nodes * n * 450.0)
    return dict(bytes=nodes * (144.0 * n + 80.0), flops=nodes * n * 140.0)


# ---- the same results in plain float64 ---------------------------------------------------


def _cs(r, a, RT):
    return r * RT * (1.0 + r + r * r - r**3) / (1.0 - r) ** 3 - a * r * r  # b = 4: eta = rho


def _cs_slope(r, a, RT):
    return RT * (1.0 + 4.0 * r + 4.0 * r**2 - 4.0 * r**3 + r**4) / (1.0 - r) ** 4 - 2.0 * a * r


def _cs_mu(r, a, RT):
    return RT * (math.log(r) + (4 * r - 3 * r * r) / (1 - r) ** 2 + (4 * r - 2 * r * r) / (1 - r) ** 3) - 2 * a * r


def _root(f, lo, hi):
    flo = f(lo)
    for _ in range(200):
        m = 0.5 * (lo + hi)
        if m in (lo, hi):
            break
        fm = f(m)
        if (fm > 0) == (flo > 0):
            lo = m
        else:
            hi = m
    return 0.5 * (lo + hi)


@functools.lru_cache(None)
def _critical_t(a):
    e = _root(lambda e: 1 - 5 * e - 20 * e**2 - 4 * e**3 + 5 * e**4 - e**5, 0.01, 0.5)
    return 2 * a / (2 * (4 + 4 * e - 2 * e * e) / (1 - e) ** 4 + e * (20 + 8 * e - 4 * e * e) / (1 - e) ** 5), e


@functools.lru_cache(None)
def _maxwell(a, Tr):
    """(rho_v, rho_l, p_sat, rho_max, rho_min, R T) of Carnahan-Starling with b = 4, R = 1."""
    Tc, rc = _critical_t(a)
    RT = Tr * Tc
    r_max = _root(lambda r: _cs_slope(r, a, RT), 1e-9, rc)
    r_min = _root(lambda r: _cs_slope(r, a, RT), rc, 0.9)
    rv = lambda p: _root(lambda r: _cs(r, a, RT) - p, 1e-14, r_max)  # noqa: E731
    rl = lambda p: _root(lambda r: _cs(r, a, RT) - p, r_min, 0.95)  # noqa: E731
    lo = max(_cs(r_min, a, RT), 1e-13)
    p = _root(lambda p: _cs_mu(rl(p), a, RT) - _cs_mu(rv(p), a, RT), lo, _cs(r_max, a, RT))
    v, li = rv(p), rl(p)
    for _ in range(4):  # Newton on equal pressure and chemical potential
        F1, F2 = _cs(v, a, RT) - _cs(li, a, RT), _cs_mu(v, a, RT) - _cs_mu(li, a, RT)
        dv, dl = _cs_slope(v, a, RT), _cs_slope(li, a, RT)
        det = -dv * dl / li + dl * dv / v
        v -= (-F1 * dl / li + F2 * dl) / det
        li -= (dv * F2 - dv / v * F1) / det
    return v, li, _cs(v, a, RT), r_max, r_min, RT


def _coexistence(a, Tr):
    return _maxwell(a, Tr)[:2]


_GX, _GW = np.polynomial.legendre.leggauss(32)


def _log_nodes(lo, hi, panels=48):
    s = np.linspace(math.log(lo), math.log(hi), panels + 1)
    h = 0.5 * (s[1] - s[0])
    r = np.exp((s[:-1, None] + h * (_GX[None, :] + 1.0)).ravel())
    return r, np.tile(_GW * h, panels) * r


def _shape(c, alpha=None):
    """Constants of the equation of state of a case (numbers), and eps of Eq. VaporLiqEq."""
    rv, rl, p_cs, rmax, rmin, RT = _maxwell(c["a_l"], c["Tr"])
    e = dict(mode=c["eos"], rv=rv, rl=rl, rmax=rmax, rmin=rmin, a_l=c["a_l"], RT_l=RT, a_v=c["a_l"], RT_v=RT, dP=0.0)
    if c["eos"] == "smooth":
        e.update(a_v=c["a_v"], RT_v=_maxwell(c["a_v"], c["Tr"])[5])
        ps = _maxwell(c["a_v"], c["Tr"])[2]
        e.update(ps=ps, dP=ps - p_cs)
        p_min = ps - (c["alpha"] if alpha is None else alpha) * (p_cs - _cs(rmin, c["a_l"], RT))
        r3 = (ps - p_min) / (_cs_slope(rl, c["a_l"], RT) * (rl - rmin))
        e.update(pmin=p_min, ia3=(1 - 2 * r3) / ((rl - rmin) * (1 - r3)) ** 2, b3=(ps - p_min) * (1 - r3) / (1 - 2 * r3))
        slope = _cs_slope(rv, e["a_v"], e["RT_v"]) * (rmax - rv)
        nodes = [_log_nodes(*x) for x in ((rv, rmax), (rmax, rmin), (rmin, rl))]

        def with_rise(q):  # q = (p_max - p_sat) / (p'(rho_v) (rho_max - rho_v)), in (0, 1/2)
            e.update(pmax=ps + q * slope, ia1=(1 - 2 * q) / ((rmax - rv) * (1 - q)) ** 2,
                     b1=q * slope * (1 - q) / (1 - 2 * q))
            return sum(float(np.sum(w * (ps - _pressure(e, r, np)) / r**2)) for r, w in nodes)

        with_rise(_root(with_rise, 1e-9, 0.5 * (1 - 1e-12)))
    else:
        e.update(ps=p_cs)
    parts = [(rv, rmax), (rmax, rmin), (rmin, rl)]
    r = np.concatenate([_log_nodes(*x)[0] for x in parts])
    w = np.concatenate([_log_nodes(*x)[1] for x in parts])
    p = _pressure(e, r, np)
    psi2 = -2.0 * (p - r / 3.0)
    base = w * (e["ps"] - p) * (_slope(e, r) - 1.0 / 3.0) / -psi2
    eps = 2.0
    for _ in range(60):
        t = base * psi2 ** (-0.5 * eps)
        step = t.sum() / (t * (-0.5 * np.log(psi2))).sum()
        eps -= step
        if abs(step) < 1e-15 * abs(eps):
            break
    e["eps"] = eps
    return e


def _slope(e, r):
    if e["mode"] == "cs":
        return _cs_slope(r, e["a_l"], e["RT_l"])
    d1, d3, span = r - e["rmax"], r - e["rmin"], e["rmin"] - e["rmax"]
    t = d1 / span
    q1 = -e["b1"] * d1 * e["ia1"] / np.sqrt(np.maximum(1e-300, 1 - d1 * d1 * e["ia1"]))
    q2 = 6.0 * (e["pmin"] - e["pmax"]) * t * (1.0 - t) / span
    q3 = e["b3"] * d3 * e["ia3"] / np.sqrt(np.maximum(1e-300, 1 - d3 * d3 * e["ia3"]))
    return np.where(r <= e["rmax"], q1, np.where(r < e["rmin"], q2, q3))


def _pressure(e, r, lib=torch):
    """p(rho) (Eq. CS; Smooth C-S of Sec. III.D); each piece is evaluated inside its own range."""
    one = lib.ones_like(r)
    liquid = _cs(r, e["a_l"], e["RT_l"]) + e["dP"]
    if e["mode"] == "cs":
        return liquid
    in1, in3 = (r > e["rv"]) & (r <= e["rmax"]), (r >= e["rmin"]) & (r < e["rl"])
    d1 = lib.where(in1, r - e["rmax"], 0.0 * one)
    d3 = lib.where(in3, r - e["rmin"], 0.0 * one)
    t = (r - e["rmax"]) / (e["rmin"] - e["rmax"])
    p1 = e["pmax"] - e["b1"] + e["b1"] * lib.sqrt(1.0 - d1 * d1 * e["ia1"])
    p2 = e["pmax"] + (e["pmin"] - e["pmax"]) * t * t * (3.0 - 2.0 * t)
    p3 = e["pmin"] + e["b3"] - e["b3"] * lib.sqrt(1.0 - d3 * d3 * e["ia3"])
    out = lib.where(in1, p1, lib.where(in3, p3, p2))
    out = lib.where(r >= e["rl"], liquid, out)
    return lib.where(r <= e["rv"], _cs(r, e["a_v"], e["RT_v"]), out)


CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
WF = (0.0,) + (1 / 3,) * 4 + (1 / 12,) * 4
MOM = ((1,) * 9, (-4, -1, -1, -1, -1, 2, 2, 2, 2), (4, -2, -2, -2, -2, 1, 1, 1, 1), CX, (0, -2, 0, 2, 0, 1, -1, -1, 1),
       CY, (0, 0, -2, 0, 2, 1, 1, -1, -1), (0, 1, -1, 1, -1, 0, 0, 0, 0), (0, 0, 0, 0, 0, 1, -1, 1, -1))


def _equilibrium(rho, ux, uy):
    return torch.stack([WT[i] * rho * (1 + 3 * (CX[i] * ux + CY[i] * uy) + 4.5 * (CX[i] * ux + CY[i] * uy) ** 2
                                       - 1.5 * (ux * ux + uy * uy)) for i in range(9)])


def _state(f, e, c, kappa):
    """rho, u, psi, F and the source tensor Q of a state."""
    psi_of = lambda r: torch.sqrt(-2.0 * (_pressure(e, r) - r / 3.0))  # noqa: E731
    rho = f.sum(0)
    psi = psi_of(rho)
    ghost = [float(psi_of(torch.tensor([e[k]], dtype=torch.float64).to(f.device)).detach()) for k in ("rl", "rv")]

    def at(i):
        p = torch.roll(psi, (-CY[i], -CX[i]), (0, 1))
        if c["walls"] and CY[i]:
            p = p.clone()
            p[-1 if CY[i] > 0 else 0] = ghost[1 if CY[i] > 0 else 0]
        return p

    n = [None] + [at(i) for i in range(1, 9)]
    Fx, Fy = (psi * sum(WF[i] * C[i] * n[i] for i in range(1, 9)) for C in (CX, CY))
    ux, uy = ((sum(C[i] * f[i] for i in range(1, 9)) + 0.5 * F) / rho for C, F in ((CX, Fx), (CY, Fy)))
    Q = None
    if c["kappa"] != 0.0 or isinstance(kappa, torch.Tensor):
        Q = [-0.5 * kappa * psi * sum(WF[i] * X[i] * Y[i] * (n[i] - psi) for i in range(1, 9))
             for X, Y in ((CX, CX), (CY, CY), (CX, CY))]
    return rho, ux, uy, psi, Fx, Fy, Q


def _lbm_step(f, e, c, kappa):
    rho, ux, uy, psi, Fx, Fy, Q = _state(f, e, c, kappa)
    M = torch.tensor(MOM, dtype=torch.float64, device=f.device)
    mv = lambda B, v: torch.einsum("ki,iyx->kyx", B, v)  # noqa: E731
    m, meq = mv(M, f), mv(M, _equilibrium(rho, ux, uy))
    te = tz = 1.0
    lam = torch.ones_like(f)
    if c["relax"] == "two_phase":
        tl, tv = 0.6, 0.5 + c.get("visc_ratio", 1.5) * 0.1
        tau = tl * (rho - e["rv"]) / (e["rl"] - e["rv"]) + tv * (rho - e["rl"]) / (e["rv"] - e["rl"])
        lam = torch.cat([lam[:7], (1.0 / tau)[None], (1.0 / tau)[None]])
    elif c["relax"] == "mrt":
        te, tz = MRT["tau_e"], MRT["tau_zeta"]
        t = [MRT["tau_" + s] for s in ("rho", "e", "zeta", "j", "q", "j", "q", "nu", "nu")]
        lam = lam / torch.tensor(t, dtype=torch.float64, device=f.device)[:, None, None]
    sigma = 0.0 if c.get("forcing") == "guo" else e["eps"] / 16.0
    uF, F2 = ux * Fx + uy * Fy, 12.0 * sigma * (Fx * Fx + Fy * Fy) / psi**2
    S = torch.stack([0 * rho, 6 * uF + F2 / (te - 0.5), -6 * uF - F2 / (tz - 0.5), Fx, -Fx, Fy, -Fy,
                     2 * (ux * Fx - uy * Fy), ux * Fy + uy * Fx])
    ms = m - lam * (m - meq) + (1 - 0.5 * lam) * S
    if Q is not None:
        z = 0 * rho
        ms = ms + lam * torch.stack([z, 1.5 * (Q[0] + Q[1]), -1.5 * (Q[0] + Q[1]), z, z, z, z, -(Q[0] - Q[1]), -Q[2]])
    g = mv(M.T / (M * M).sum(1), ms)
    out = [torch.roll(g[i], (CY[i], CX[i]), (0, 1)) for i in range(9)]
    if c["walls"]:
        for i in range(9):
            if CY[i]:
                row = 0 if CY[i] > 0 else -1
                out[i] = out[i].clone()
                out[i][row] = g[OPP[i]][row]
    return torch.stack(out)


def _exact_lbm(c, fields):
    e = _shape(c)
    f = _equilibrium(*fields)
    for _ in range(c["steps"]):
        f = _lbm_step(f, e, c, c["kappa"])
    return f, _state(f, e, c, c["kappa"])[:4]


def _exact_adjoint(c, seed):
    rho0 = _fields(c, seed)[0].requires_grad_(True)
    names = ("pmax", "ia1", "b1", "pmin", "ia3", "b3", "eps")
    base = _shape(c)
    leaf = {k: torch.tensor(base[k], dtype=torch.float64, device=DEV, requires_grad=True) for k in names}
    e = dict(base, **leaf)
    kappa = torch.tensor(c["kappa"], dtype=torch.float64, device=DEV, requires_grad=True)
    zero = torch.zeros_like(rho0)
    f = _equilibrium(rho0, zero, zero)
    for _ in range(c["steps"]):
        f = _lbm_step(f, e, c, kappa)
    rho = f.sum(0)
    weight = torch.randn(rho0.shape, device=DEV, dtype=torch.float64,
                         generator=torch.Generator(device=DEV).manual_seed(int(seed) + 1))
    (rho * weight).sum().backward()
    if c["param"] == "kappa":
        g = kappa.grad
    else:  # the shape's constants by central differences at h and h/2 (Richardson)
        at = lambda x: np.array([_shape(c, c["alpha"] + x)[k] for k in names])  # noqa: E731
        h = 1e-3
        d = [(at(s) - at(-s)) / (2 * s) for s in (h, h / 2, h / 4)]
        r1, r2 = (4 * d[1] - d[0]) / 3, (4 * d[2] - d[1]) / 3
        dc = (16 * r2 - r1) / 15
        g = sum(leaf[k].grad * float(v) for k, v in zip(names, dc))
    return [rho.detach(), rho0.grad, g.detach()]


def _exact_fd(c, seed):
    e = _shape(c)
    e0 = e["eps"]
    rho, ux, uy = _fields(dict(c, shape="impact" if c["walls"] else "droplet"), seed, dx=c["dx"])
    psi_of = lambda r: torch.sqrt(-2.0 * (_pressure(e, r) - r / 3.0))  # noqa: E731
    psi_l = psi_of(torch.tensor([e["rl"]], dtype=torch.float64, device=DEV))
    h, G = c["dx"], -1.0
    sh = lambda a, i, j: torch.roll(a, (-j, -i), (0, 1))  # noqa: E731
    ex = ((1, 0), (0, 1))
    cen = lambda a, d: (sh(a, *ex[d]) - sh(a, -ex[d][0], -ex[d][1])) / (2 * h)  # noqa: E731

    def second(a, d, k):
        if d == k:
            return (sh(a, *ex[d]) - 2 * a + sh(a, -ex[d][0], -ex[d][1])) / h**2
        return (sh(a, 1, 1) - sh(a, 1, -1) - sh(a, -1, 1) + sh(a, -1, -1)) / (4 * h * h)

    def rhs(r, u, forward):
        s = psi_of(r)
        if c["walls"]:  # two ghost rows below and above
            low_r, low_s = 2 * r[:1] - r[1:2], 2 * s[:1] - s[1:2]
            z = torch.zeros_like(low_r)
            s = torch.cat([low_s + 2 * h * (psi_l - low_s), low_s, s, s[-1:], s[-2:-1]])
            r = torch.cat([low_r, low_r, r, r[-1:], r[-2:-1]])
            u = [torch.cat([z, z, v, -v[-1:], z]) for v in u]
        p = _pressure(e, r)
        one = lambda a, d: (sh(a, *ex[d]) - a) / h if forward else (a - sh(a, -ex[d][0], -ex[d][1])) / h  # noqa: E731
        tau, dtau = c["tau_nu"], 0.0
        if c["vary"]:
            tv = 0.5 + 2.0 * (c["tau_nu"] - 0.5)
            dtau = (c["tau_nu"] - tv) / (e["rl"] - e["rv"])
            tau = c["tau_nu"] + dtau * (r - e["rl"])
        mu, mub = r * (tau - 0.5) / 3, r * (c["tau_e"] - tau) / 3
        dmu, dmub = (tau - 0.5 + r * dtau) / 3, (c["tau_e"] - tau - r * dtau) / 3
        dr = [one(r, d) for d in range(2)]
        du = [[one(u[b], d) for b in range(2)] for d in range(2)]
        ps = [cen(s, d) for d in range(2)]
        dd = [[second(s, d, b) for b in range(2)] for d in range(2)]
        lap = dd[0][0] + dd[1][1]
        div = du[0][0] + du[1][1]
        out = [-(r * div + u[0] * dr[0] + u[1] * dr[1])]
        for a in range(2):
            S = ps[0] * dd[a][0] + ps[1] * dd[a][1]
            pp = G * ((1 / 6 - e0 / 4) * S + ps[a] * lap / 12 + 0.25 * s * cen(lap, a) + c["kappa"] / 6 * (ps[a] * lap - S))
            v = sum(dmu * dr[b] * (du[a][b] + du[b][a]) for b in range(2)) + dmub * dr[a] * div
            v = v + sum(mu * (second(u[b], a, b) + second(u[a], b, b)) + mub * second(u[b], a, b) for b in range(2))
            out.append(-sum(u[b] * du[b][a] for b in range(2)) + (v - pp - one(p, a)) / r)
        return [q[2:-2] for q in out] if c["walls"] else out

    U = [rho, ux, uy]
    for _ in range(c["steps"]):
        k = rhs(U[0], U[1:], True)
        V = [a + c["dt"] * b for a, b in zip(U, k)]
        k = rhs(V[0], V[1:], False)
        U = [0.5 * (a + b + c["dt"] * d) for a, b, d in zip(U, V, k)]
    return U


def exact(case, seed):
    k = case["kind"]
    if k == "fd":
        with torch.no_grad():
            return _exact_fd(case, seed)
    if k == "adjoint":
        return _exact_adjoint(case, seed)
    out = []
    with torch.no_grad():
        for i, c in enumerate(_instances(case)):
            if c["eos"] == "peng":  # its cubic's root has no closed form here
                out.append(None)
                continue
            init = _fields(c, int(seed) * 1009 + i)
            if k == "host_sweep":  # run_host takes densities alone: at rest
                init = [init[0], 0.0 * init[0], 0.0 * init[0]]
            f, (rho, ux, uy, psi) = _exact_lbm(c, init)
            if k == "single":
                return [f, rho, ux, uy, psi]
            out.append(rho.cpu() if k == "host_sweep" else f)
    if k in ("planar_sweep", "impact_sweep"):
        return dict(guard=None, f=out)
    return out
