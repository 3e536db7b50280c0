"""The finite-difference update in fixed point against the CPU oracle, 3 steps at sizes
around the blocks' and the stencil's edges, and on points that take the general form.

Tolerances: the oracle's equation of state and force terms carry about 30 roundings of
psi^2 <= 0.12, 4e-16 in all, divided by rho_v = 3e-3 and multiplied by dt h^3 <= 1.6: 2e-13
per right-hand side, 1.3e-12 in the velocities after three steps of two; 1e-11 is asked for,
and the density (scale 0.4, changes of dt h rho du) agrees to the same relative to its
largest value."""
import numpy as np
import pytest

import lbm_inputs as I
from gpu_helpers import normwise
from oracle import eos as E
from oracle import fd as F

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(1, 33, False), (2, 64, False), (3, 40, False), (33, 5, False), (129, 3, False), (34, 66, False),
         (1, 40, True), (2, 33, True), (65, 42, True), (32, 36, True)]
FORMS = {"constant": dict(tau_nu=0.8, tau_e=1.1), "kappa": dict(tau_nu=0.7, tau_e=1.0, kappa=0.3),
         "vary": dict(tau_e=1.0, tau_l=0.7, visc_ratio=5.0), "equal": dict(tau_nu=0.9, tau_e=0.9)}


def pair(nx, ny, walls, form, dx):
    import paper_2107_06355_gb300 as P

    eosp = P.EOSParams(P.EOS_SMOOTH, 0.6, 0.387, 2.0, 0.834)
    oe = E.make_eos(E.MODE_SMOOTH, 0.6, 0.387, 2.0, 0.834)
    cpu = F.FDSolver(oe, P.eos_setup(eosp)["eps"], dx=dx, walls=walls, **FORMS[form])
    gpu = P.FDSolver(nx, ny, eosp, dx=dx, bc=P.BC_WALLS_Y if walls else P.BC_PERIODIC, **FORMS[form])
    return oe, cpu, gpu


def fields(oe, nx, ny, walls, amp):
    if walls:
        rho = I.impact(nx, ny, 0.15 * ny, 0.25 * ny, oe.rho_v, oe.rho_l, 0.0, W=8.0)[0]
    else:
        rho = I.planar(nx, ny, oe.rho_v, oe.rho_l, W=8.0, axis="y" if ny > nx else "x")
    return (I.perturbed(rho, 1e-3, 11), *I.random_velocity((ny, nx), amp, 12))


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("nx, ny, walls", SIZES)
@pytest.mark.parametrize("amp", [0.004, 0.0, 1e-200])
def test_three_steps(form, nx, ny, walls, amp):
    dx = 0.5
    dt = 0.2 * dx * dx
    oe, cpu, gpu = pair(nx, ny, walls, form, dx)
    rho, ux, uy = fields(oe, nx, ny, walls, amp)
    r, u = cpu.run(rho.copy(), [ux.copy(), uy.copy()], 3 * dt, dt)
    gpu.set_state(rho, ux, uy)
    gpu.step(3, dt)
    gr, gx, gy = [t.cpu().numpy() for t in gpu.get_state()]
    assert np.isfinite(r).all() and normwise(gr, r) < 1e-11
    assert np.abs(gx - u[0]).max() < 1e-11 and np.abs(gy - u[1]).max() < 1e-11
    gpu.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e40])
def test_points_outside_the_frames(bad):
    """One velocity that the frames do not hold: its neighbourhood takes the general form, not
    finite wherever the oracle is not (both velocity components share the frames there, so a
    point of the stencil may be more), and beyond the stencils' reach nothing changes."""
    dx, dt = 0.5, 0.05
    oe, cpu, gpu = pair(40, 48, False, "constant", dx)
    rho, ux, uy = fields(oe, 40, 48, False, 0.004)
    ux[20, 13] = bad
    with np.errstate(all="ignore"):
        r, u = cpu.run(rho.copy(), [ux.copy(), uy.copy()], dt, dt)
    gpu.set_state(rho, ux, uy)
    gpu.step(1, dt)
    for got, ref in zip([t.cpu().numpy() for t in gpu.get_state()], [r, *u]):
        assert not (np.isfinite(got) & ~np.isfinite(ref)).any()
        far = np.ones(ref.shape, bool)
        far[16:25, 9:18] = False
        assert np.isfinite(ref[far]).all() and np.abs(got[far] - ref[far]).max() < 1e-11
    gpu.close()
