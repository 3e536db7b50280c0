"""Kernels launched dependent on their predecessors: bitwise the same results when the steps
are captured in a CUDA graph, between other work on the stream, and on lattices whose tile
rows exceed one grid axis."""
import numpy as np
import pytest

import lbm_inputs as I
from oracle import eos as E
from oracle import fd as F

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EOS = (0.6, 0.387, 2.0, 0.834)
KINDS = {"unit": dict(), "kappa": dict(kappa=0.4), "two_phase": dict(kind=1, tau_l=0.6, visc_ratio=3.0),
         "mrt": dict(tau_e=1.1, tau_nu=0.8, tau_q=1.2)}


def make(P, kind, nx, ny, seed=3):
    sim = P.Simulation(nx, ny, P.BC_PERIODIC, P.EOSParams(P.EOS_SMOOTH, *EOS), P.Relax(**KINDS[kind]))
    d = sim.derived()
    rho = I.perturbed(I.planar(nx, ny, d["rho_v"], d["rho_l"], W=10.0), 1e-3, seed)
    return sim, (rho, *I.random_velocity((ny, nx), 0.01, seed))


def same(a, b):
    return bool(torch.isfinite(a).all()) and torch.equal(a.view(torch.int64), b.view(torch.int64))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("nx, ny", [(32, 32), (131, 77), (1, 9001)])
def test_captured_steps(kind, nx, ny):
    import paper_2107_06355_gb300 as P

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ref, init = make(P, kind, nx, ny)
        ref.init_equilibrium(*init)
        f0 = ref.get_f()
        ref.step(4)
        ref.step(4)
        want = ref.get_f()
        sim, _ = make(P, kind, nx, ny)
        src, buf = f0.clone(), torch.zeros_like(f0)
        sim.set_f(f0)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            buf.copy_(src)
            sim.step(4)
        g.replay()
        g.replay()
        s.synchronize()
        assert same(sim.get_f(), want) and same(buf, src)
    ref.close()
    sim.close()


@pytest.mark.parametrize("kind", ["unit", "two_phase"])
def test_more_tile_rows_than_a_grid_axis(kind):
    import paper_2107_06355_gb300 as P

    nx, ny = 1, 131_073 + 2 * 4096
    sim, init = make(P, kind, nx, ny)
    b = P.Batch([(nx, ny, P.BC_PERIODIC)], [P.EOSParams(P.EOS_SMOOTH, *EOS)], [P.Relax(**KINDS[kind])])
    sim.init_equilibrium(*init)
    b.init_equilibrium(0, *init)
    sim.step(3)
    b.step(3)
    assert same(sim.get_f(), b.get_f(0))
    sim.close()
    b.close()


def test_fd_more_tile_rows_than_a_grid_axis():
    """(1, 262,145): one step against the oracle, to the bounds of the fixed-point update's
    test (a third of the roundings)."""
    import paper_2107_06355_gb300 as P

    ny, dx, dt = 4 * 65_536 + 1, 0.5, 0.05
    eosp = P.EOSParams(P.EOS_SMOOTH, *EOS)
    oe = E.make_eos(E.MODE_SMOOTH, *EOS)
    rho = I.perturbed(I.planar(1, ny, oe.rho_v, oe.rho_l, W=10.0), 1e-3, 5)
    ux, uy = I.random_velocity((ny, 1), 0.004, 6)
    r, u = F.FDSolver(oe, P.eos_setup(eosp)["eps"], tau_nu=0.8, tau_e=1.0, dx=dx).step(rho, [ux, uy], dt)
    gpu = P.FDSolver(1, ny, eosp, tau_nu=0.8, tau_e=1.0, dx=dx)
    gpu.set_state(rho, ux, uy)
    gpu.step(1, dt)
    gr, gx, gy = [t.cpu().numpy() for t in gpu.get_state()]
    assert np.abs(gr - r).max() < 1e-11 * r.max()
    assert np.abs(gx - u[0]).max() < 1e-11 and np.abs(gy - u[1]).max() < 1e-11
    gpu.close()
