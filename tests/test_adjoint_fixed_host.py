"""The fixed-point reverse of the collision (csrc/adjoint_fixed.cuh), built for the host from
the same source, against forward-mode differentiation in exact rational arithmetic (dual
numbers over fractions.Fraction) of the populations' definition."""
import ctypes as C
import os
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WT = [Fr(4, 9)] + [Fr(1, 9)] * 4 + [Fr(1, 36)] * 4
HF, ZS = 1.0 / 24.0, 0.12 / 432.0
NAMES = ("rho", "jx", "jy", "m7", "m8", "psi", "gx", "gy", "zs")


class Dual:
    def __init__(self, v, d=0):
        self.v, self.d = Fr(v), Fr(d)

    @staticmethod
    def of(x):
        return x if isinstance(x, Dual) else Dual(x)

    def __add__(self, o):
        o = Dual.of(o)
        return Dual(self.v + o.v, self.d + o.d)

    def __mul__(self, o):
        o = Dual.of(o)
        return Dual(self.v * o.v, self.v * o.d + self.d * o.v)

    def inverse(self):
        return Dual(1 / self.v, -self.d / self.v**2)

    __radd__, __rmul__ = __add__, __mul__

    def __sub__(self, o):
        return self + Dual.of(o) * -1


@pytest.fixture(scope="module")
def af(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("adjfix") / "libadjoint_fixed_host.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-o", so,
                    os.path.join(ROOT, "tests", "native", "adjoint_fixed_host.cpp")], check=True)
    lib = C.CDLL(so)
    lib.af_reverse.argtypes = [C.c_longlong, C.c_int] + [C.c_void_p] * 3
    lib.af_slope.argtypes = [C.c_void_p, C.c_double, C.c_int, C.c_longlong] + [C.c_void_p] * 5
    return lib


def reverse(lib, rows, shear, tau):
    out = np.zeros((len(rows), 17))
    rows, c = np.ascontiguousarray(rows), np.array([HF, ZS, *tau])
    lib.af_reverse(len(rows), shear, c.ctypes.data, rows.ctypes.data, out.ctypes.data)
    return out[:, :16], out[:, 16] == 1.0


def objective(x, mu, shear, tau):
    """sum_i mu_i f*_i of (rho, jx, jy, m7, m8, psi, gx, gy, zs)."""
    rho, jx, jy, m7, m8, psi, gx, gy, zs = x
    hx, hy = Fr(HF) * psi * gx, Fr(HF) * psi * gy
    inv = rho.inverse()
    ux, uy = (jx + hx) * inv, (jy + hy) * inv
    Px, Py = jx + 2 * hx, jy + 2 * hy
    xx, yy, xy = ux * (Px + hx), uy * (Py + hy), ux * Py + uy * hx
    tr, d = xx + yy, xx - yy
    zz = zs * (gx * gx + gy * gy)
    if shear:
        w = Dual(1) - (Fr(tau[0]) + Fr(tau[1]) * rho).inverse()
        d = d + w * (m7 - ux * (jx - hx) + uy * (jy - hy))
        xy = xy + w * (m8 - ux * jy + uy * hx)
    xx, yy = (tr + d) * Fr(1, 2), (tr - d) * Fr(1, 2)
    total = Dual(0)
    for i in range(9):
        f = WT[i] * (rho + 3 * (CX[i] * Px + CY[i] * Py)
                     + Fr(9, 2) * (CX[i]**2 * xx + CY[i]**2 * yy + 2 * CX[i] * CY[i] * xy - tr * Fr(1, 3)))
        total = total + Fr(float(mu[i])) * (f + (-8 if i == 0 else 1) * zz)
    return total


def nodes(rng, n, lo, hi, amp, u, spread):
    rho = 10.0 ** rng.uniform(lo, hi, size=(n, 1))
    psi = np.sqrt(0.6 * rho) * (1 + amp * rng.uniform(-1, 1, size=(n, 9)))
    j = rho * u * rng.uniform(-1, 1, size=(n, 2))
    m = 0.05 * rho * rng.uniform(-1, 1, size=(n, 2))
    mu = rng.normal(size=(n, 1)) * (1 + spread * rng.normal(size=(n, 9)))
    return np.hstack([psi, rho, j, m, mu])


@pytest.mark.parametrize("shear", [0, 1])
@pytest.mark.parametrize("lo, hi, amp, u, spread", [(-5, -2, 0.1, 0.1, 1.0), (-0.7, -0.3, 0.05, 0.05, 0.1),
                                                    (-1, 0.5, 1e-6, 1e-6, 1e-3), (-3, 0, 0.0, 0.0, 0.5)])
def test_adjoints_against_dual_numbers(af, shear, lo, hi, amp, u, spread):
    """Absolute errors against the largest |mu| = M. rho_b, j_b, m7_b, m8_b: the nine
    truncated mu (2^-54 M each, coefficients summing to 72 over 36, squared into velocities
    below 1: 4 units), at most 16 products of 8 units over 36, then the conversion: 2^-50 M.
    The source's sums 6 t, sd, xd: at most 12 truncations of 2^-59 psi_max, then the
    conversion, 2^-53 of at most 12 psi_max: 2^-51 P. psi_b, g_b and zs_b carry the factors half_force psi (g) and zz_scale g psi, g up to
    6 psi_max = P: 2^-48 M half_force P, 2^-48 M (half_force psi + zz_scale P) and
    2^-48 M P^2."""
    rng = np.random.default_rng(60 + shear)
    rows = nodes(rng, 60, lo, hi, amp, u, spread)
    tau = ((2.0, -0.4), (0.6, 0.0))[int(lo > -2)]
    out, ok = reverse(af, rows, shear, tau)
    assert ok.all()
    for r, got in zip(rows, out):
        p = [Fr(float(v)) for v in r[:9]]
        gx = 4 * (p[1] - p[2]) + (p[5] - p[7]) + (p[8] - p[6])
        gy = 4 * (p[3] - p[4]) + (p[5] - p[7]) - (p[8] - p[6])
        base = [Fr(float(r[9])), Fr(float(r[10])), Fr(float(r[11])), Fr(float(r[12])), Fr(float(r[13])), p[0], gx, gy,
                Fr(ZS)]
        M, P = Fr(float(np.abs(r[14:]).max())), 6 * max(p)
        tol = [M / 2**50] * 5 + [M * Fr(HF) * P / 2**48] + [M * (Fr(HF) * p[0] + Fr(ZS) * P) / 2**48] * 2 + [M * P * P / 2**48]
        t6 = sum(p[1:5]) + sum(p[5:9]) / 2 - 6 * p[0]
        sums = (t6, p[1] + p[2] - p[3] - p[4], p[5] + p[7] - p[6] - p[8])
        assert all(abs(Fr(float(g)) - want) <= P / 2**51 for g, want in zip(got[13:], sums))
        for i, name in enumerate(NAMES):
            if not shear and name in ("m7", "m8"):
                continue
            x = [Dual(v, 1 if k == i else 0) for k, v in enumerate(base)]
            want = objective(x, r[14:], shear, tau).d
            assert abs(Fr(float(got[i])) - want) <= tol[i], (name, got[i], float(want))


@pytest.mark.parametrize("mode, Tr, al, av, b, alpha, G", [(0, 0.6, 0.387, 0.387, 4.0, 0.5, -1.0),
                                                           (1, 0.35, 0.363, 2.0, 4.0, 0.838, -1.0),
                                                           (1, 0.8, 0.5, 0.5, 4.0, 0.342, -3.0),
                                                           (1, 0.5, 0.363, 2.0, 2.0, 0.775, -0.25)])
@pytest.mark.parametrize("branch", [0, 1])
def test_slope_of_the_cs_branches(af, mode, Tr, al, av, b, alpha, G, branch):
    """d psi^2 / d rho in units of 2^s (|2/(3 G)| 2^-s in [1/2, 1)), with v = 1/(1 - eta): v is
    within v/2 units of 2^-58 (reciprocal_q63), v^2 within v^2 + 2, so the polynomial v^2 t +
    1/2, t = 3 v^2 - 2 v - 1, within (v^2 + 2)(t + 3 v^2) + v^3 + 9; times c1, plus 6 units of
    2^-56 (the products and constants), then the conversion. 1/(2 rho): 2^-52 relative."""
    rng = np.random.default_rng(9)
    rho = np.concatenate([10.0 ** rng.uniform(-9, np.log10(1.99 / b), 200), [1.0 / b, np.nextafter(2.0 / b, 0.0), 2.0 / b]])
    n, k, par = len(rho), np.zeros(3), np.array([mode, Tr, al, av, b, 1.0, alpha])
    slope, half, ok = np.zeros(n), np.zeros(n), np.zeros(n, np.int32)
    assert af.af_slope(par.ctypes.data, G, branch, n, rho.ctypes.data, k.ctypes.data, slope.ctypes.data,
                       half.ctypes.data, ok.ctypes.data) == 0
    assert ok[:-1].all() and not ok[-1]  # eta = 1/2 is outside
    bb, RT, a = (Fr(float(x)) for x in k)
    sc = Fr(2) / Fr(G)
    s = int(np.floor(np.log2(2 / (3 * abs(G))))) + 1
    for r, got, h in zip(rho[:-1], slope, half):
        r = Fr(float(r))
        v = 1 / (1 - bb / 4 * r)
        t = 3 * v * v - 2 * v - 1
        want = sc * (2 * RT * (v * v * t + Fr(1, 2)) - 2 * a * r - Fr(1, 3))
        c1 = abs(2 * sc * RT) / Fr(2) ** s
        units = c1 * ((v * v + 2) * (t + 3 * v * v) + v**3 + 9) / 4 + 6  # of 2^-56
        assert abs(Fr(float(got)) - want) <= units * Fr(2) ** (s - 56) + abs(want) / 2**53, float(r)
        assert abs(Fr(float(h)) * 2 * r - 1) <= Fr(1, 2**52)


def test_outside_the_domain(af):
    base = nodes(np.random.default_rng(8), 1, -1, -1, 0.05, 0.05, 0.5)[0]
    rows = []
    for k, v in ((9, 0.0), (9, np.nan), (9, 1e-200), (0, np.nan), (3, np.inf), (1, -0.2), (10, 0.11), (11, np.inf),
                 (14, np.nan), (20, np.inf), (17, 1e200)):
        r = base.copy()
        r[k] = v
        rows.append(r)
    for shear in (0, 1):
        assert not reverse(af, np.array(rows), shear, (0.6, 0.0))[1].any()
    assert not reverse(af, base[None], 1, (0.4, 0.0))[1].any()
