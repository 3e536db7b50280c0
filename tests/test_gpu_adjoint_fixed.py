"""The adjoint passes at the edges of their warps and blocks (rows of 32 nodes, two rows per
block) against the oracle's autograd: lambda, the kappa and alpha gradients, and the same
lambda from the kernels with and without the constants' sums.

Tolerances are those of the larger lattices' tests: lambda to 1e-12 of its largest value (a
few hundred roundings of 2^-53, amplified by 1/rho_v of at most 2e3 on vapour nodes only
where lambda is as large), dL/dkappa to 1e-9 and dL/dalpha to 1e-6 (the differences of the
set-up behind it) of the largest per-constant contribution."""
import ctypes as C

import numpy as np
import pytest

import lbm_inputs as I
from gpu_helpers import BC_PER, BC_WALLS, make_pair, normwise
from oracle import adjoint as A
from oracle import eos as E

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2107_06355_gb300")
from paper_2107_06355_gb300 import _lib as L  # noqa: E402

CASE = (E.MODE_SMOOTH, 0.5, 0.363, 2.0, 0.775)
RELAX = {"unit": {}, "two_phase": dict(kind=P.RELAX_TWO_PHASE, tau_l=0.6, visc_ratio=3.0)}


@pytest.mark.parametrize("relax", RELAX)
@pytest.mark.parametrize("kappa", [0.0, 0.6])
@pytest.mark.parametrize("nx, ny, bc", [(1, 40, BC_PER), (31, 33, BC_PER), (32, 40, BC_PER), (33, 41, BC_PER),
                                        (65, 32, BC_PER), (2, 41, BC_WALLS), (33, 40, BC_WALLS), (64, 37, BC_WALLS)])
def test_adjoint_step_at_the_edges(relax, kappa, nx, ny, bc):
    olat, sim = make_pair(nx, ny, bc, CASE, dict(RELAX[relax], kappa=kappa))
    e = olat.eos
    if bc == BC_WALLS:
        rho = I.impact(nx, ny, 0.15 * ny, 0.3 * ny, e.rho_v, e.rho_l, 0.0, W=8.0)[0]
    else:
        rho = I.planar(nx, ny, e.rho_v, e.rho_l, W=8.0)
    rho = I.perturbed(rho, 1e-3, 4)
    f = olat.step(olat.init_equilibrium(rho, *I.random_velocity((ny, nx), 0.005, 6)), 3)
    lam1 = np.random.default_rng(17).standard_normal((9, ny, nx))
    c = A.constants_as_tensors(e)
    c["kappa"] = torch.tensor(kappa, dtype=torch.float64, requires_grad=True)
    x = torch.tensor(f, requires_grad=True)
    (A.step(x, olat, c) * torch.tensor(lam1)).sum().backward()
    dc = A.constants_derivative(*CASE[:4], CASE[4])
    parts = [float(c[k].grad) * dc[k] for k in A.CONST_NAMES]
    fd, l1 = torch.tensor(f, device="cuda"), torch.tensor(lam1, device="cuda")
    nbytes = L.lib().pplbm_adjoint_workspace_bytes(C.byref(sim.lattice))
    p = lambda t: C.c_void_p(t.data_ptr())  # noqa: E731
    lams = []
    for mask in ((1 << L.NGRAD) - 1, 0):
        assert L.lib().pplbm_adjoint_set_slots(sim.ctx, mask) == 0
        l0, grad = torch.empty_like(l1), torch.zeros(L.NGRAD, dtype=torch.float64, device="cuda")
        ws = torch.full((nbytes // 8 + 1,), float("nan"), dtype=torch.float64, device="cuda")
        assert L.lib().pplbm_adjoint_step(sim.ctx, p(fd), p(l1), p(l0), p(grad), p(ws), nbytes) == 0
        torch.cuda.synchronize()
        lams.append(l0.cpu())
        if mask:
            full = grad.cpu()
        else:
            assert bool((grad == 0).all())
    assert torch.equal(*lams) and normwise(lams[0].numpy(), x.grad.numpy()) < 1e-12
    k = float(c["kappa"].grad)
    assert float(full[L.GRAD_NAMES.index("kappa")]) == pytest.approx(k, rel=1e-9, abs=1e-9 * np.abs(lam1).sum() * 1e-3)
    grad = full.cuda()
    assert L.lib().pplbm_adjoint_set_param(sim.ctx, 0, 1e-4) == 0
    out = (C.c_double * 1)()
    assert L.lib().pplbm_adjoint_param_gradient(sim.ctx, p(grad), out) == 0
    assert abs(out[0] - sum(parts)) < 1e-6 * max(abs(v) for v in parts)
    sim.close()
