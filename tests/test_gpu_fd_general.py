"""The finite-difference update's general form at every point, which constants outside the
frames take (a time step of 1e-21): against the CPU oracle in the changes of one step, at the
edges of its 32 x 8 tiles."""
import numpy as np
import pytest

import lbm_inputs as I
from oracle import eos as E
from oracle import fd as F

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FORMS = {"constant": dict(tau_nu=0.8, tau_e=1.1), "kappa": dict(tau_nu=0.7, tau_e=1.0, kappa=0.3),
         "vary": dict(tau_e=1.0, tau_l=0.7, visc_ratio=5.0)}


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("nx, ny, walls", [(1, 33, False), (33, 9, False), (31, 40, True), (64, 33, True)])
def test_constants_outside_the_frames(form, nx, ny, walls):
    """Velocities of 1e-20 and a step of 1e-21, so that a step's change is seen to 1e-4 or better
    of the velocities and its rounding (2^-53 1e-20) is 1e-12 of the change. The right-hand
    side's terms cancel to a tenth at most, their 30 roundings leave 1e-13 of the largest change
    on nodes of the largest density, 1 / rho_v more on the others: 1e-11."""
    import paper_2107_06355_gb300 as P

    dx, dt = 0.5, 1e-21
    eosp = P.EOSParams(P.EOS_SMOOTH, 0.6, 0.387, 2.0, 0.834)
    oe = E.make_eos(E.MODE_SMOOTH, 0.6, 0.387, 2.0, 0.834)
    cpu = F.FDSolver(oe, P.eos_setup(eosp)["eps"], dx=dx, walls=walls, **FORMS[form])
    gpu = P.FDSolver(nx, ny, eosp, dx=dx, bc=P.BC_WALLS_Y if walls else P.BC_PERIODIC, **FORMS[form])
    if walls:
        rho = I.impact(nx, ny, 0.15 * ny, 0.25 * ny, oe.rho_v, oe.rho_l, 0.0, W=8.0)[0]
    else:
        rho = I.planar(nx, ny, oe.rho_v, oe.rho_l, W=8.0, axis="y" if ny > nx else "x")
    rho = I.perturbed(rho, 1e-3, 11)
    ux, uy = I.random_velocity((ny, nx), 1e-20, 12)
    _, u = cpu.step(rho.copy(), [ux.copy(), uy.copy()], dt)
    gpu.set_state(rho, ux, uy)
    gpu.step(1, dt)
    gr, gx, gy = [t.cpu().numpy() for t in gpu.get_state()]
    gpu.close()
    scale = max(np.abs(u[0] - ux).max(), np.abs(u[1] - uy).max())
    assert scale > 1e-23 and np.array_equal(gr, rho)
    assert np.abs(gx - u[0]).max() < 1e-11 * scale and np.abs(gy - u[1]).max() < 1e-11 * scale
