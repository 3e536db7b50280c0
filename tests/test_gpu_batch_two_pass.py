"""Batches whose launches and graph plans run the two step kernels (one lattice is beyond the
clusters' 4,096 nodes) at every tile width, and batches of six relaxation times in clusters (at
most 2,048 nodes per lattice): walls, odd sizes, several equations of state, kappa on some
lattices only; bitwise the single lattices."""
import pytest

import lbm_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2107_06355_gb300")

RELAX = {"unit": {}, "two_phase": dict(kind=1, tau_l=0.6, visc_ratio=2.0),
         "mrt": dict(tau_e=0.8, tau_zeta=1.1, tau_q=1.2, tau_nu=0.9)}
SMALL = [(4, 90, P.BC_PERIODIC, 0.8), (33, 33, P.BC_PERIODIC, 0.35), (48, 40, P.BC_WALLS_Y, 0.6), (3, 5, P.BC_PERIODIC, 0.6),
         (1, 1, P.BC_PERIODIC, 0.7), (130, 9, P.BC_WALLS_Y, 0.5)]
LARGE = [(70, 61, P.BC_PERIODIC, 0.6), (5, 901, P.BC_WALLS_Y, 0.5)]  # 4,270 and 4,505 nodes


def check(sizes, kind, kappas, mode, width):
    eos = [P.EOSParams(P.EOS_SMOOTH, Tr, 0.363, 2.0, 0.775) for _, _, _, Tr in sizes]
    relax = [P.Relax(**RELAX[kind], kappa=kappas[k % len(kappas)]) for k in range(len(sizes))]
    b = P.Batch([s[:3] for s in sizes], eos, relax)
    b.set_plan(mode, width)
    sims = []
    for k, (nx, ny, bc, _) in enumerate(sizes):
        s = P.Simulation(nx, ny, bc, eos[k], relax[k])
        d = s.derived()
        if bc == P.BC_WALLS_Y:  # a film on the bottom wall
            rho = I.impact(nx, ny, 0.15 * ny, 0.3 * ny, d["rho_v"], d["rho_l"], 0.0, W=6.0)[0]
        else:
            rho = I.planar(nx, ny, d["rho_v"], d["rho_l"], W=6.0, axis="y" if ny > nx else "x")
        init = (I.perturbed(rho, 1e-3, k), *I.random_velocity(rho.shape, 0.01, k))
        s.init_equilibrium(*init)
        b.init_equilibrium(k, *init)
        sims.append(s)
    for n in (1, 6, 7):
        b.step(n)
        for k, s in enumerate(sims):
            s.step(n)
            got, want = b.get_f(k), s.get_f()
            assert bool(torch.isfinite(want).all()) and torch.equal(got.view(torch.int64), want.view(torch.int64)), (n, k)
    for k, s in enumerate(sims):
        assert all(torch.equal(x, y) for x, y in zip(b.fields(k), s.fields()))
        s.close()
    b.close()


@pytest.mark.parametrize("kind", RELAX)
@pytest.mark.parametrize("kappas", [(0.0,), (0.4, 0.0, -0.6)])
@pytest.mark.parametrize("mode, width", [(0, 0), (0, 4), (0, 32), (0, 256), (1, 0), (1, 4), (1, 256)])
def test_two_step_kernels(kind, kappas, mode, width):
    check(SMALL + LARGE, kind, kappas, mode, width)


@pytest.mark.parametrize("kappas", [(0.0,), (0.4, 0.0, -0.6)])
@pytest.mark.parametrize("mode", [0, 1])
def test_six_rates_in_clusters(kappas, mode):
    check(SMALL + [(64, 32, P.BC_PERIODIC, 0.6)], "mrt", kappas, mode, 0)


@pytest.mark.parametrize("kind", RELAX)
def test_clusters_with_kappa_on_some_lattices(kind):
    check(SMALL, kind, (0.4, 0.0, -0.6), 1, 0)
