"""The reverse pass over the whole range of cotangents: a loss scaled by a power of two gives
the gradient scaled by it. Host build of csrc/adjoint_fixed.cuh (rows that it accepts are
bitwise the scaled rows, the others are reported), and rollouts on the GPU."""
from fractions import Fraction as Fr

import numpy as np
import pytest

import lbm_inputs as I
from test_adjoint_fixed_host import CX, CY, WT, af, nodes, reverse  # noqa: F401


@pytest.mark.parametrize("shear", [0, 1])
def test_scaled_cotangents(af, shear):  # noqa: F811
    """Every value is linear in mu, and a power of two only shifts the frame: bitwise."""
    rows = nodes(np.random.default_rng(5), 40, -3, -0.5, 0.1, 0.1, 0.5)
    rows[:, 14:] *= 2.0 ** -np.floor(np.log2(np.abs(rows[:, 14:]).max(axis=1, keepdims=True)))  # largest in [1, 2)
    want, ok = reverse(af, rows, shear, (0.6, 0.0))
    assert ok.all()
    linear = [0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11]
    for k in (-300, -100, 100, 250, 300, 340, 400, 600, 699, 700, 701, 760, 900, 1000, 1030, 1040):
        r = rows.copy()
        r[:, 14:] = np.ldexp(r[:, 14:], -k)
        got, acc = reverse(af, r, shear, (0.6, 0.0))
        assert np.array_equal(acc, np.full(len(rows), k <= 700)), k
        if k <= 700:
            assert np.array_equal(got[:, linear], np.ldexp(want[:, linear], -k)), k


@pytest.mark.parametrize("shear", [0, 1])
def test_small_psi_beside_small_cotangents(af, shear):  # noqa: F811
    """zs_b is a product of mu and psi^2: accepted rows are exact multiples of the unscaled ones
    as long as it stays a normal double, and the rest is reported."""
    rows = nodes(np.random.default_rng(7), 20, -3, -0.5, 0.1, 0.1, 0.5)
    rows[:, 14:] *= 2.0 ** -np.floor(np.log2(np.abs(rows[:, 14:]).max(axis=1, keepdims=True)))
    seen = set()
    for psi, k in ((0, 690), (80, 600), (80, 690), (150, 500), (150, 690), (150, 100)):
        base, r = rows.copy(), rows.copy()
        base[:, :9] = np.ldexp(base[:, :9], -psi)
        r[:, :9] = base[:, :9]
        r[:, 14:] = np.ldexp(r[:, 14:], -k)
        want, ok = reverse(af, base, shear, (0.6, 0.0))
        assert ok.all()
        got, acc = reverse(af, r, shear, (0.6, 0.0))
        seen |= set(acc.tolist())
        assert np.array_equal(got[acc, :12], np.ldexp(want[acc, :12], -k)), (psi, k)
    assert seen == {True, False}


@pytest.mark.parametrize("shear", [0, 1])
def test_zero_cotangents_are_inside(af, shear):  # noqa: F811
    rows = nodes(np.random.default_rng(6), 3, -1, -1, 0.05, 0.05, 0.5)
    rows[:, 14:] = 0.0
    rows[1, 14:18] = -0.0
    rows[2, 20] = 1e-310
    got, acc = reverse(af, rows, shear, (0.6, 0.0))
    assert acc.tolist() == [True, True, False]
    assert not got[:2, :12].any()


@pytest.mark.parametrize("shear", [0, 1])
@pytest.mark.parametrize("octaves", [2, 4, 6])
def test_small_density_adjoint_beside_large_momentum_adjoint(af, shear, octaves):  # noqa: F811
    """mu_i = r + c_i . J with |J| = 2^octaves |r| in a fluid at rest: rho_b = sum w_i mu_i exactly.
    With M the largest |mu|, every mu is rounded to nearest in units of 2^-55 M at most, ties to
    even (beyond the second dropped bit to 1/8 unit): rho_b's error is below a unit, 2^-55 M, plus
    its own rounding 2^-53 |r|, and its mean in r's direction below 2^-58 M plus four standard
    errors of 0.3 2^-55 M / sqrt(2000): 2^-57 M. Cut off towards zero it was 2^-55 M."""
    rng = np.random.default_rng(octaves)
    n = 2000
    rows = np.zeros((n, 23))
    rows[:, :9], rows[:, 9] = np.sqrt(0.3), 0.4
    r = rng.choice([-1.0, 1.0], n) * rng.uniform(1.0, 2.0, n)
    a = rng.uniform(0.0, 2.0 * np.pi, n)
    J = 2.0**octaves * np.abs(r)[:, None] * np.stack([np.cos(a), np.sin(a)], 1)
    for i in range(9):
        rows[:, 14 + i] = r + CX[i] * J[:, 0] + CY[i] * J[:, 1]
    got, ok = reverse(af, rows, shear, (0.6, 0.0))
    assert ok.all()
    mean = 0.0
    for k in range(n):
        M = float(np.abs(rows[k, 14:]).max())
        want = sum(w * Fr(float(v)) for w, v in zip(WT, rows[k, 14:]))
        e = float(Fr(float(got[k, 0])) - want)
        assert abs(e) <= 2.0**-55 * M + 2.0**-53 * abs(float(want))
        mean += e * np.sign(float(want)) / M / n
    assert abs(mean) < 2.0**-57


@pytest.mark.gpu
@pytest.mark.parametrize("relax, kappa", [(dict(), 0.0), (dict(), 0.3), (dict(kind=1, tau_l=0.6, visc_ratio=3.0), 0.0),
                                          (dict(kind=1, tau_l=0.6, visc_ratio=3.0), 0.3)])
@pytest.mark.parametrize("k", [250, 640, 700, 800])
def test_scaled_loss(relax, kappa, k):
    """20 steps on 40 x 36: the nodes outside the frames take the double-precision form, which
    agrees with the fixed-point one to a few hundred roundings of 2^-53 of the largest lambda,
    amplified by 1/rho_v on vapour nodes (1e-12 in the tests of one step): 1e-10 of the
    largest value over 20 steps. dL/dalpha is a sum over the nodes with random weights: 1e-10
    of its terms, four digits left for what they cancel."""
    torch = pytest.importorskip("torch")
    import paper_2107_06355_gb300 as P
    from paper_2107_06355_gb300 import adjoint as A

    eos = P.EOSParams(P.EOS_SMOOTH, 0.5, 0.363, 2.0, 0.775)
    d = P.eos_setup(eos)
    nx, ny = 40, 36
    rho = torch.tensor(I.perturbed(I.planar(nx, ny, d["rho_v"], d["rho_l"], W=8.0), 1e-3, 2), device="cuda")
    spec = A.RolloutSpec(nx, ny, P.BC_PERIODIC, eos, P.Relax(kappa=kappa, **relax), nsteps=20)
    w = torch.tensor(np.random.default_rng(3).standard_normal((ny, nx)), device="cuda")

    def gradient(scale):
        x = rho.clone().requires_grad_(True)
        t = torch.tensor(0.775, dtype=torch.float64, requires_grad=True)
        (A.rollout(x, t, spec) * (w * scale)).sum().backward()
        return x.grad, float(t.grad)

    g0, a0 = gradient(1.0)
    g1, a1 = gradient(2.0 ** -k)
    assert bool(torch.isfinite(g0).all()) and float(g0.abs().max()) > 0.0
    assert float((g1 * 2.0 ** k - g0).abs().max()) < 1e-10 * float(g0.abs().max())
    assert abs(a1 * 2.0 ** k - a0) < 1e-6 * abs(a0)


@pytest.mark.gpu
@pytest.mark.parametrize("relax", [dict(), dict(kind=1, tau_l=0.6, visc_ratio=1.5)])
def test_long_rollout(relax):
    """400 steps on 28 x 24: the fixed-point reverse against the double-precision form, which the
    loss scaled by 2^-900 takes at every node. Each has an error of about 1e-16 of the gradient per
    step from the stored lambda's and the stages' roundings, 4e-14 in all: 1e-13 between the two."""
    torch = pytest.importorskip("torch")
    import paper_2107_06355_gb300 as P
    from paper_2107_06355_gb300 import adjoint as A

    eos = P.EOSParams(P.EOS_SMOOTH, 0.6, 0.387, 2.0, 0.834)
    d = P.eos_setup(eos)
    nx, ny = 28, 24
    y, x = np.mgrid[0:ny, 0:nx]
    phi = 0.5 * (1.0 - np.tanh(4.6 * (np.hypot(x - 13.6, y - 11.7) - 6.0) / 8.0))
    rho = torch.tensor(d["rho_v"] + (d["rho_l"] - d["rho_v"]) * phi, device="cuda")
    spec = A.RolloutSpec(nx, ny, P.BC_PERIODIC, eos, P.Relax(**relax), nsteps=400)
    w = torch.tensor(np.random.default_rng(4).standard_normal((ny, nx)), device="cuda")
    g = []
    for scale in (1.0, 2.0 ** -900):
        r = rho.clone().requires_grad_(True)
        (A.rollout(r, torch.tensor(0.834, dtype=torch.float64), spec) * (w * scale)).sum().backward()
        g.append(r.grad / scale)
    assert float((g[0] - g[1]).square().mean().sqrt()) < 1e-13 * float(g[1].square().mean().sqrt())
