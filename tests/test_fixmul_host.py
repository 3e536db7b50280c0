"""The fixed-point collision (csrc/collide_fixed.cuh, csrc/fixmul.cuh), built for the
host from the same source, against exact rational arithmetic: the post-collision
populations w_i [rho + 3 c_i.P + 4.5 (c_i c_i - I/3) : Pi*] + z_i (-8, 1, ..., 1) of the
node's doubles, for unit relaxation times and the two-phase set, with and without the
surface-tension source."""
import ctypes as C
import math
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


@pytest.fixture(scope="module")
def fm(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fixmul") / "libfixmul_host.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-o", so,
                    os.path.join(ROOT, "tests", "native", "fixmul_host.cpp")], check=True)
    lib = C.CDLL(so)
    lib.fm_collide.argtypes = [C.c_longlong, C.c_int, C.c_int] + [C.c_void_p] * 3
    for name in ("fm_reciprocal", "fm_to_double"):
        getattr(lib, name).argtypes = [C.c_longlong, C.c_void_p, C.c_void_p]
    return lib


RATES, LI = (1 / 1.1, 1 / 0.9, 1 / 1.2, 1 / 0.8), (0.12 * 12 / 0.6 / 144, 0.12 * 12 / 0.4 / 144)


def collide(lib, rows, shear, st, kq, tau=(1.0, 0.0)):
    out = np.zeros((len(rows), 10))
    c = np.array([HF, ZS, kq, *tau, *RATES, *LI])
    rows = np.ascontiguousarray(np.hstack([rows, np.zeros((len(rows), 18 - rows.shape[1]))]))
    lib.fm_collide(len(rows), shear, st, c.ctypes.data, rows.ctypes.data, out.ctypes.data)
    return out[:, :9], out[:, 9] == 1.0


def exact(r, shear, st, kq, tau):
    p = [Fr(float(v)) for v in r]
    rho, jx, jy, m7, m8 = p[9:]
    gx = 4 * (p[1] - p[2]) + (p[5] - p[7]) + (p[8] - p[6])
    gy = 4 * (p[3] - p[4]) + (p[5] - p[7]) - (p[8] - p[6])
    hx, hy = Fr(HF) * p[0] * gx, Fr(HF) * p[0] * gy
    ux, uy = (jx + hx) / rho, (jy + hy) / rho
    Px, Py = jx + 2 * hx, jy + 2 * hy
    xx, yy, xy = ux * (Px + hx), uy * (Py + hy), ux * Py + uy * hx
    tr, d = xx + yy, xx - yy
    zz = Fr(ZS) * (gx * gx + gy * gy)
    om = 1 / (Fr(tau[0]) + Fr(tau[1]) * rho) if shear else Fr(1)
    if shear:
        d += (1 - om) * (m7 - ux * (jx - hx) + uy * (jy - hy))
        xy += (1 - om) * (m8 - ux * jy + uy * hx)
    if st:
        k = Fr(kq) * p[0]
        zz += k * (Fr(1, 6) * sum(p[1:5]) + Fr(1, 12) * sum(p[5:9]) - p[0])
        d -= 4 * om * k * (p[1] + p[2] - p[3] - p[4])
        xy -= om * k * (p[5] + p[7] - p[6] - p[8])
    xx, yy = (tr + d) / 2, (tr - d) / 2
    return [WT[i] * (rho + 3 * (CX[i] * Px + CY[i] * Py)
                     + Fr(9, 2) * (CX[i]**2 * xx + CY[i]**2 * yy + 2 * CX[i] * CY[i] * xy - tr / 3))
            + (-8 if i == 0 else 1) * zz for i in range(9)]


MOM = ((1,) * 9, (-4, -1, -1, -1, -1, 2, 2, 2, 2), (4, -2, -2, -2, -2, 1, 1, 1, 1), CX, (0, -2, 0, 2, 0, 1, -1, -1, 1),
       CY, (0, 0, -2, 0, 2, 1, 1, -1, -1), (0, 1, -1, 1, -1, 0, 0, 0, 0), (0, 0, 0, 0, 0, 1, -1, 1, -1))


def exact_mrt(r, st, kq):
    """m* = m - omega (m - m_eq) + (1 - omega/2) S in rational arithmetic, f* = M^-1 m*."""
    p = [Fr(float(v)) for v in r]
    rho, jx, jy = p[9:12]
    gx = 4 * (p[1] - p[2]) + (p[5] - p[7]) + (p[8] - p[6])
    gy = 4 * (p[3] - p[4]) + (p[5] - p[7]) - (p[8] - p[6])
    Fx, Fy = 2 * Fr(HF) * p[0] * gx, 2 * Fr(HF) * p[0] * gy
    Jx, Jy = jx + Fx / 2, jy + Fy / 2
    ux, uy = Jx / rho, Jy / rho
    m = [rho, p[12], p[13], jx, p[14], jy, p[15], p[16], p[17]]
    u2, uF, F2 = ux * Jx + uy * Jy, ux * Fx + uy * Fy, gx * gx + gy * gy
    eq = [rho, 3 * u2 - 2 * rho, rho - 3 * u2, Jx, -Jx, Jy, -Jy, ux * Jx - uy * Jy, ux * Jy]
    S = [0, 6 * uF + Fr(LI[0]) * F2, -6 * uF - Fr(LI[1]) * F2, Fx, -Fx, Fy, -Fy, 2 * (ux * Fx - uy * Fy), ux * Fy + uy * Fx]
    if st:
        k = Fr(kq) * p[0]
        t = Fr(1, 6) * sum(p[1:5]) + Fr(1, 12) * sum(p[5:9]) - p[0]
        eq[1] += 36 * k * t
        eq[2] -= 36 * k * t
        eq[7] -= 4 * k * (p[1] + p[2] - p[3] - p[4])
        eq[8] -= k * (p[5] + p[7] - p[6] - p[8])
    om = [Fr(1), *[Fr(RATES[i]) for i in (0, 1)], Fr(1), Fr(RATES[2]), Fr(1), Fr(RATES[2]), Fr(RATES[3]), Fr(RATES[3])]
    ms = [a - w * (a - e) + (1 - w / 2) * s for a, w, e, s in zip(m, om, eq, S)]
    norm = [sum(c * c for c in row) for row in MOM]
    return [sum(MOM[k][i] * ms[k] / norm[k] for k in range(9)) for i in range(9)]


@pytest.mark.parametrize("st", [0, 1])
@pytest.mark.parametrize("lo, hi, amp, u", [(-5, -2, 0.2, 0.15), (-0.7, -0.3, 0.1, 0.1), (-3, 0, 0.0, 0.0)])
def test_six_relaxation_times_against_exact_rational_arithmetic(fm, st, lo, hi, amp, u):
    """As for the other forms: each relaxed moment carries its own truncation, twice those of
    the equilibrium and the source (2 units per product and shift, coefficients up to 12 in
    the source) and the rate's product: at most 40 units, the second moments' 24; they enter a
    population with coefficients 4 (r), 1, 2 (rows 1, 2), 6 + 6 (rows 3 to 6) and 9: 500 units,
    300 more for the source; the rest population's sum is scaled by 4."""
    rng = np.random.default_rng(40 + st)
    rows = nodes(rng, 300, lo, hi, amp, u)
    rho = rows[:, 9:10]
    mom = np.hstack([rho * (-2 + 0.1 * rng.uniform(-1, 1, rho.shape)), rho * (1 + 0.1 * rng.uniform(-1, 1, rho.shape)),
                     -rows[:, 10:12] + 0.02 * rho * rng.uniform(-1, 1, (len(rho), 2)),
                     0.05 * rho * rng.uniform(-1, 1, (len(rho), 2))])
    rows = np.hstack([rows[:, :12], mom])
    kq = -0.5 / 24 if st else 0.0
    f, ok = collide(fm, rows, 2, st, kq)
    assert ok.mean() > 0.95
    for r, got in zip(rows[ok], f[ok]):
        unit = Fr(2) ** (math.frexp(r[9])[1] - 64)
        for i, e in enumerate(exact_mrt(r, st, kq)):
            tol = Fr(math.ulp(got[i])) / 2 + (500 + 300 * st) * unit * (4 if i == 0 else 1)
            assert abs(Fr(float(got[i])) - e) <= tol, (i, got[i], float(e))


def nodes(rng, n, lo, hi, amp, u):
    """Densities in 10^[lo, hi], psi ~ sqrt(0.6 rho) varying by amp, momenta up to u rho."""
    rho = 10.0 ** rng.uniform(lo, hi, size=(n, 1))
    psi = np.sqrt(0.6 * rho) * (1 + amp * rng.uniform(-1, 1, size=(n, 9)))
    j = rho * u * rng.uniform(-1, 1, size=(n, 2))
    m = 0.05 * rho * rng.uniform(-1, 1, size=(n, 2))
    return np.hstack([psi, rho, j, m])


def seed_of(lo):
    return {-5: 0, -0.7: 1, -1: 2, -3: 0}[lo]


@pytest.mark.parametrize("st", [0, 1])
@pytest.mark.parametrize("shear", [0, 1])
@pytest.mark.parametrize("lo, hi, amp, u", [(-5, -2, 0.25, 0.2), (-0.7, -0.3, 0.1, 0.1), (-1, 0.5, 1e-9, 1e-9),
                                            (-3, 0, 0.0, 0.0)])
def test_populations_against_exact_rational_arithmetic(fm, shear, st, lo, hi, amp, u):
    """Each population is within half its own ulp (the one rounding) plus the frame's
    truncations: at most 2 units of 2^(e - 1086) per product (e the biased exponent of
    rho), carried through the sums with their coefficients (18 on the diagonal moments, 9
    on the mixed one, 12 on the momenta, 16 on rho): 150 units, 120 more for the rows 7, 8
    corrections and 120 more for the source; the rest population's sum is scaled by 4."""
    rng = np.random.default_rng(20 + 2 * shear + st)
    rows = nodes(rng, 300, lo, hi, amp, u)
    tau = ((2.0, -0.4), (0.6, 0.0), (0.55, 0.9))[seed_of(lo)]
    kq = -0.5 / 24 if st else 0.0
    f, ok = collide(fm, rows, shear, st, kq, tau)
    assert ok.mean() > 0.95  # the few others are handed to the general collision
    rows, f = rows[ok], f[ok]
    units = 150 + 120 * shear + 120 * st
    for r, got in zip(rows, f):
        unit = Fr(2) ** (math.frexp(r[9])[1] - 64)  # 2^(e - 1086)
        for i, e in enumerate(exact(r, shear, st, kq, tau)):
            tol = Fr(math.ulp(got[i])) / 2 + units * unit * (4 if i == 0 else 1)
            assert abs(Fr(float(got[i])) - e) <= tol, (i, got[i], float(e))


def test_rest_state_is_exact_and_transverse_momentum_stays_zero(fm):
    """Equal psi and zero momentum give w_i rho to half an ulp with equal values per class;
    a profile along x alone keeps the y mirror pairs bitwise equal."""
    rng = np.random.default_rng(5)
    rows = nodes(rng, 200, -4, 0, 0.0, 0.0)
    rows[:, 10:] = 0.0
    f, ok = collide(fm, rows, 0, 0, 0.0)
    assert ok.all()
    assert (f[:, 1:2] == f[:, 1:5]).all() and (f[:, 5:6] == f[:, 5:]).all()
    rows = nodes(rng, 200, -4, 0, 0.1, 0.1)
    p = rows[:, :9]
    p[:, 3] = p[:, 4] = p[:, 0]
    p[:, 5] = p[:, 8] = p[:, 1]
    p[:, 6] = p[:, 7] = p[:, 2]
    rows[:, 11:] = 0.0
    f, ok = collide(fm, rows, 0, 0, 0.0)
    assert ok.all()
    for a, b in ((2, 4), (5, 8), (6, 7)):
        assert (f[:, a] == f[:, b]).all()


def test_nodes_outside_the_domain_are_reported(fm):
    """Densities, psi or momenta the frames cannot hold, populations at or below zero: the
    caller must run the general collision."""
    base = nodes(np.random.default_rng(6), 1, -1, -1, 0.05, 0.05)[0]
    cases = []
    for k, v in ((9, 0.0), (9, -0.1), (9, np.nan), (9, np.inf), (9, 1e-300), (9, 1e300), (0, np.nan), (3, np.inf),
                 (5, -0.2), (10, 0.09), (11, -0.3), (10, np.nan), (11, np.inf), (2, 40.0)):
        r = base.copy()
        r[k] = v
        cases.append(r)
    for shear in (0, 1):
        for st in (0, 1):
            _, ok = collide(fm, np.array(cases), shear, st, -0.02 * st)
            assert not ok.any(), (shear, st, ok)
    r = np.array([base] * 2)
    r[0, 12], r[1, 13] = np.nan, 1.0
    assert not collide(fm, r, 1, 0, 0.0, (0.6, 0.0))[1].any()
    # tau below 1/2 or from 16 on
    for tau in ((0.4, 0.0), (-3.0, 0.0), (15.9, 2.0), (1.0, -40.0)):
        assert not collide(fm, r[:1] * 0 + base, 1, 0, 0.0, tau)[1].any()


def test_reciprocal_and_conversion(fm):
    rng = np.random.default_rng(7)
    L = (rng.integers(0, 2**52, 4000, dtype=np.uint64) << np.uint64(11)) | np.uint64(1 << 63)
    L[:3] = [1 << 63, (2**53 - 1) << 11, (2**52 + 1) << 11]
    out = np.zeros(len(L), np.int64)
    fm.fm_reciprocal(len(L), L.ctypes.data, out.ctypes.data)
    for a, b in zip(L.tolist(), out.tolist()):
        e = Fr(9 * 2**122, a)
        assert abs(Fr(b) - e) <= e / 2**60
    n = rng.integers(2**32, 2**63 - 1, 4000, dtype=np.int64) >> rng.integers(0, 30, 4000)
    n = np.maximum(n, 2**32)
    n[:6] = [2**32, 2**63 - 1, 2**53 + 1, 2**54 + 2, 2**54 + 6, 2**60 - 1]
    d = np.zeros(len(n))
    fm.fm_to_double(len(n), n.ctypes.data, d.ctypes.data)
    assert d.tolist() == [float(v) for v in n.tolist()]
