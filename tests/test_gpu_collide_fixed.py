"""The collision kernels' fixed-point path and its fall-back at the lattice shapes where
their neighbour indices and tiles can go wrong, against the oracle (1e-12 normwise per
step, as the other parity tests)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import lbm_inputs as I  # noqa: E402
from gpu_helpers import BC_PER, BC_WALLS, make_pair, normwise  # noqa: E402

SMOOTH06 = (1, 0.6, 0.387, 2.0, 0.834)
KINDS = {"unit": dict(), "kappa": dict(kappa=0.4), "two_phase": dict(kind=1, tau_l=0.6, visc_ratio=3.0),
         "two_phase_kappa": dict(kind=1, tau_l=0.6, visc_ratio=3.0, kappa=-0.3)}


def state(olat, nx, ny, speed, seed):
    e = olat.eos
    rng = np.random.default_rng(seed)
    rho = e.rho_v + (e.rho_l - e.rho_v) * (0.5 + 0.4 * np.sin(2 * np.pi * (np.arange(ny)[:, None] / ny
                                                                           + np.arange(nx)[None, :] / nx)))
    rho = I.perturbed(rho, 1e-2, seed)
    return rho, speed * rng.uniform(-1, 1, rho.shape), speed * rng.uniform(-1, 1, rho.shape)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("nx, ny, walls", [(1, 1, False), (1, 5, True), (2, 200, False), (3, 2, True), (31, 8, False),
                                           (32, 9, True), (33, 7, False), (65, 17, True)])
def test_shapes(kind, nx, ny, walls):
    olat, sim = make_pair(nx, ny, BC_WALLS if walls else BC_PER, SMOOTH06, KINDS[kind])
    rho, ux, uy = state(olat, nx, ny, 0.02, 3)
    sim.init_equilibrium(rho, ux, uy)
    f = olat.init_equilibrium(rho, ux, uy)
    for _ in range(3):
        sim.step(1)
        f = olat.step(f)
        assert normwise(sim.get_f().cpu().numpy(), f) <= 1e-12
        sim.set_f(f)
    sim.close()


@pytest.mark.parametrize("kind", KINDS)
def test_fast_nodes_take_the_general_collision(kind):
    """|u| up to 1.3: beyond the fixed-point path's bounds on many nodes, inside on others."""
    olat, sim = make_pair(48, 20, BC_WALLS, SMOOTH06, KINDS[kind])
    rho, ux, uy = state(olat, 48, 20, 1.3, 4)
    sim.init_equilibrium(rho, ux, uy)
    f = olat.init_equilibrium(rho, ux, uy)
    sim.step(1)
    assert normwise(sim.get_f().cpu().numpy(), olat.step(f)) <= 1e-12
    sim.close()
