"""Small lattices advance all steps of a call in one cluster launch: bitwise the two step
kernels (which run while per-kernel timing is on), at the edges of the shapes' ranges,
single lattices and batches."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import lbm_inputs as I  # noqa: E402

KINDS = {"unit": dict(), "kappa": dict(kappa=0.4), "two_phase": dict(kind=1, tau_l=0.6, visc_ratio=3.0),
         "mrt": dict(tau_e=1.1, tau_nu=0.8, tau_q=1.2)}
SIZES = [(1, 1, False), (1, 5, True), (2, 200, False), (127, 1, False), (129, 1, False), (32, 64, True), (2049, 1, False),
         (64, 64, False), (4096, 1, False), (17, 241, True)]


def make(P, kind, nx, ny, walls, seed):
    eos = P.EOSParams(P.EOS_SMOOTH, 0.6, 0.387, 2.0, 0.834)
    sim = P.Simulation(nx, ny, P.BC_WALLS_Y if walls else P.BC_PERIODIC, eos, P.Relax(**KINDS[kind]))
    d = sim.derived()
    # a film on the bottom wall, or a slab of liquid: states that stay finite
    rho = I.impact(nx, ny, 0.2 * ny, 0.3 * ny, d["rho_v"], d["rho_l"], 0.0)[0] if walls else \
        I.planar(nx, ny, d["rho_v"], d["rho_l"], W=10.0)
    rho = I.perturbed(rho, 1e-2, seed)
    u = I.random_velocity(rho.shape, 0.01, seed)
    return sim, (rho, *u)


def same(a, b):
    return bool(torch.isfinite(a).all()) and torch.equal(a.view(torch.int64), b.view(torch.int64))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("nx, ny, walls", SIZES)
def test_single_lattice_bitwise(kind, nx, ny, walls):
    import paper_2107_06355_gb300 as P

    sim, init = make(P, kind, nx, ny, walls, 5)
    ref, _ = make(P, kind, nx, ny, walls, 5)
    ref.enable_kernel_timing(64)
    sim.init_equilibrium(*init)
    ref.init_equilibrium(*init)
    for n in (1, 2, 5, 0, 8):
        sim.step(n)
        ref.step(n)
        assert same(sim.get_f(), ref.get_f()), n
    assert ref.kernel_times()[1] == (16, 16) and sim.sync() == 16 and ref.sync() == 16
    sim.close()
    ref.close()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("plan", [0, 1])
def test_batch_bitwise(kind, plan):
    import paper_2107_06355_gb300 as P

    sizes = [(1, 5, True), (2, 200, False), (40, 33, True), (16, 16, False), (64, 64, False)]
    refs = [make(P, kind, *s, 7 + k) for k, s in enumerate(sizes)]
    eos = P.EOSParams(P.EOS_SMOOTH, 0.6, 0.387, 2.0, 0.834)
    b = P.Batch([(nx, ny, P.BC_WALLS_Y if w else P.BC_PERIODIC) for nx, ny, w in sizes], [eos] * 5,
                [P.Relax(**KINDS[kind])] * 5)
    b.set_plan(plan, 0)
    for k, (ref, init) in enumerate(refs):
        ref.enable_kernel_timing(64)
        ref.init_equilibrium(*init)
        b.init_equilibrium(k, *init)
    for n in (1, 4, 3):
        b.step(n)
        for k, (ref, _) in enumerate(refs):
            ref.step(n)
            assert same(b.get_f(k), ref.get_f()), (n, k)
    b.close()
