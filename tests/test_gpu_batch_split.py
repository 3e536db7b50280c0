"""Work items of a batch, each shared by two blocks of 128 threads, few and many of them:
bitwise the single lattices, for every collision kind and the
narrowest and widest tiles."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import lbm_inputs as I  # noqa: E402

KINDS = {"unit": dict(), "kappa": dict(kappa=0.4), "two_phase": dict(kind=1, tau_l=0.6, visc_ratio=3.0),
         "mrt": dict(tau_e=1.1, tau_nu=0.8, tau_q=1.2)}


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("sizes", [((70, 67), (5, 901)), ((640, 640), (641, 640))])
@pytest.mark.parametrize("plan, width", [(0, 0), (1, 4), (0, 256)])
def test_batch_bitwise(kind, sizes, plan, width):
    import paper_2107_06355_gb300 as P

    eos = P.EOSParams(P.EOS_SMOOTH, 0.6, 0.387, 2.0, 0.834)
    b = P.Batch([(nx, ny, P.BC_PERIODIC) for nx, ny in sizes], [eos] * 2, [P.Relax(**KINDS[kind])] * 2)
    b.set_plan(plan, width)
    refs = []
    for k, (nx, ny) in enumerate(sizes):
        ref = P.Simulation(nx, ny, P.BC_PERIODIC, eos, P.Relax(**KINDS[kind]))
        d = ref.derived()
        rho = I.perturbed(I.planar(nx, ny, d["rho_v"], d["rho_l"], W=10.0), 1e-3, k)
        init = (rho, *I.random_velocity(rho.shape, 0.01, k))
        ref.init_equilibrium(*init)
        b.init_equilibrium(k, *init)
        ref.step(5)
        refs.append(ref)
    b.step(5)
    for k, ref in enumerate(refs):
        got, want = b.get_f(k), ref.get_f()
        assert bool(torch.isfinite(want).all()) and torch.equal(got.view(torch.int64), want.view(torch.int64))
        ref.close()
    b.close()
