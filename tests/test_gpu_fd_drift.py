"""The finite-difference update adds no mean acceleration: over some hundred steps the mean
velocities stay with the CPU oracle's."""
import numpy as np
import pytest

from oracle import eos as E
from oracle import fd as F

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FORMS = {"constant": dict(tau_nu=0.8, tau_e=1.0), "kappa": dict(tau_nu=0.7, tau_e=1.0, kappa=0.3),
         "vary": dict(tau_e=1.0, tau_l=0.7, visc_ratio=4.0), "vary large": dict(tau_e=1.2, tau_l=0.55, visc_ratio=20.0)}


def solvers(form, dx):
    import paper_2107_06355_gb300 as P

    eosp = P.EOSParams(P.EOS_SMOOTH, 0.6, 0.387, 2.0, 0.834)
    oe = E.make_eos(E.MODE_SMOOTH, 0.6, 0.387, 2.0, 0.834)
    cpu = F.FDSolver(oe, P.eos_setup(eosp)["eps"], dx=dx, **FORMS[form])
    return oe, cpu, P.FDSolver(44, 40, eosp, dx=dx, **FORMS[form])


@pytest.mark.parametrize("form", FORMS)
def test_droplet(form):
    """200 steps: a velocity's error is that of its stages' roundings, about 30 of 2^-53 of terms
    up to 0.05 (dt times pressure gradients over rho at the interface), 3e-17 rms a step without a
    direction: a mean over 1,760 points of 3e-17 sqrt(200 / 1760) = 1e-17 in each solver. 1e-16 is
    asked for; a mean rounding of one unit, 2e-18 to 5e-17 a step, gave 3.5e-16 to 1e-14."""
    dx, dt = 0.5, 0.05
    oe, cpu, gpu = solvers(form, dx)
    y, x = np.mgrid[0:40, 0:44]
    phi = 0.5 * (1.0 - np.tanh(4.6 * (np.hypot(x - 21.3, y - 19.6) * dx - 5.0) / 6.0))
    rho = oe.rho_v + (oe.rho_l - oe.rho_v) * phi
    rng = np.random.default_rng(1)
    u = [1e-3 * rng.uniform(-1, 1, rho.shape) for _ in range(2)]
    gpu.set_state(rho, *u)
    gpu.step(200, dt)
    _, ref = cpu.run(rho.copy(), [v.copy() for v in u], 200 * dt, dt)
    got = [t.cpu().numpy().astype(np.longdouble) for t in gpu.get_state()[1:]]
    gpu.close()
    for g, r in zip(got, ref):
        assert np.isfinite(r).all() and abs(float((g - r).mean())) < 1e-16


@pytest.mark.parametrize("form", ["constant", "vary"])
def test_shear_flow(form):
    """A uniform liquid with u_x = 1e-3 sin(2 pi y / 40): no force acts, u_y stays zero, the mean of
    u_x keeps within the roundings of the stored u_x (2^-54 1e-3 in 400 steps of two, at random:
    1.6e-18 a point, 4e-20 in the mean; 1e-18 is asked for), and u_x with the oracle's to 1e-17."""
    dx, dt = 0.5, 0.05
    oe, cpu, gpu = solvers(form, dx)
    y = np.mgrid[0:40, 0:44][0]
    rho, ux = np.full((40, 44), 1.01 * oe.rho_l), 1e-3 * np.sin(2.0 * np.pi * y / 40)
    gpu.set_state(rho, ux, np.zeros_like(ux))
    gpu.step(400, dt)
    _, ref = cpu.run(rho.copy(), [ux.copy(), np.zeros_like(ux)], 400 * dt, dt)
    gr, gx, gy = [t.cpu().numpy() for t in gpu.get_state()]
    gpu.close()
    assert np.array_equal(gr, rho) and not gy.any()
    assert abs(float(gx.astype(np.longdouble).mean() - ux.astype(np.longdouble).mean())) < 1e-18
    assert np.abs(gx - ref[0]).max() < 1e-17


@pytest.mark.parametrize("form", ["constant", "vary"])
@pytest.mark.parametrize("swap", [False, True])
@pytest.mark.parametrize("small", [1e-8, 1e-3, 1e-60, 1e-250])
def test_small_component_beside_a_large_one(form, swap, small):
    """A uniform liquid drifting at 0.1 across a shear of amplitude `small`: the small component
    keeps the accuracy of its own size. Its right-hand side has about 20 roundings of 2^-53 of its
    own terms, of order 0.1 of it a step: 4e-17 of it, 400 steps of two at worst in one direction
    4e-14, in each solver. 1e-13 is asked for."""
    dx, dt = 0.5, 0.05
    oe, cpu, gpu = solvers(form, dx)
    y, x = np.mgrid[0:40, 0:44]
    ux, uy = small * np.sin(2.0 * np.pi * y / 40), np.full(x.shape, 0.1)
    rho = np.full((40, 44), 1.01 * oe.rho_l)
    if swap:
        ux, uy = np.full(x.shape, 0.1), small * np.sin(2.0 * np.pi * x / 44)
    gpu.set_state(rho, ux, uy)
    gpu.step(400, dt)
    _, ref = cpu.run(rho.copy(), [ux.copy(), uy.copy()], 400 * dt, dt)
    got = [t.cpu().numpy() for t in gpu.get_state()[1:]]
    gpu.close()
    k = 1 if swap else 0
    assert np.abs(got[k] - ref[k]).max() < 1e-13 * small
    assert np.abs(got[1 - k] - ref[1 - k]).max() < 1e-14
