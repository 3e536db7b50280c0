"""f^eq of given densities and velocities (Eq. EquilibriumDistribution): exactly w_i rho at
rest, and within 6 roundings of the formula otherwise (weight, four in the polynomial, the
product; |c.u| < 0.3 keeps the polynomial above 0.4: 2^-50 relative)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CX, CY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
W = [4.0 / 9] + [1.0 / 9] * 4 + [1.0 / 36] * 4


@pytest.mark.parametrize("nx, ny", [(1, 1), (255, 1), (257, 3)])
@pytest.mark.parametrize("moving", [(), ("x",), ("y",), ("x", "y")])
def test_equilibrium(nx, ny, moving):
    import paper_2107_06355_gb300 as P

    sim = P.Simulation(nx, ny, P.BC_PERIODIC, P.EOSParams(P.EOS_SMOOTH, 0.6, 0.387, 2.0, 0.834), P.Relax())
    g = torch.Generator(device="cuda").manual_seed(nx)
    new = lambda: torch.rand(ny, nx, dtype=torch.float64, device="cuda", generator=g)  # noqa: E731
    rho, zero = new() + 1e-3, torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
    u = [0.1 * (new() - 0.5) if d in moving else zero for d in "xy"]
    sim.init_equilibrium(rho, *[u[i] if d in moving else None for i, d in enumerate("xy")])
    f = sim.get_f()
    for i in range(9):
        cu = CX[i] * u[0] + CY[i] * u[1]
        want = W[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u[0] ** 2 + u[1] ** 2))
        if not moving:
            assert torch.equal(f[i], want)
        assert bool(((f[i] - want).abs() <= 2.0**-50 * want).all())
    sim.close()
