"""The fixed-point products (csrc/fixmul.cuh) have no mean error, so that a step adds no
momentum: host build against exact integers, and a droplet at rest on the GPU."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def mh(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("mulhi") / "libmulhi_host.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-o", so,
                    os.path.join(ROOT, "tests", "native", "mulhi_host.cpp")], check=True)
    lib = C.CDLL(so)
    lib.mh_product.argtypes = [C.c_longlong] + [C.c_void_p] * 3
    lib.mh_pair.argtypes = [C.c_longlong] + [C.c_void_p] * 5
    lib.mh_constant.argtypes = [C.c_longlong, C.c_longlong] + [C.c_void_p] * 2
    return lib


def errors(lib, *f):
    f = [np.ascontiguousarray(v, dtype=np.int64) for v in f]
    out = np.zeros(len(f[0]), np.int64)
    (lib.mh_product if len(f) == 2 else lib.mh_pair)(len(out), *(v.ctypes.data for v in f), out.ctypes.data)
    exact = [sum(int(a[i]) * int(b[i]) for a, b in zip(f[::2], f[1::2])) for i in range(len(out))]
    return np.array([((int(o) << 64) - e) / 2.0**64 for o, e in zip(out, exact)])


@pytest.mark.parametrize("bits", [(62, 62), (62, 58), (58, 50), (62, 40), (40, 33)])
@pytest.mark.parametrize("terms", [1, 2])
def test_mean_error(mh, bits, terms):
    """An error has the shift's half unit, the low halves' product (1/4, by the addend's mean
    zero) and each factor's dropped bit (below a quarter of a unit, of either sign): a standard
    deviation below 0.5 per term, 0.5 / sqrt(40,000) = 0.0025 for the mean, so 0.02 is asked for; every single error
    stays below 2 units a term."""
    rng = np.random.default_rng(sum(bits) + terms)
    n = 40_000
    f = [rng.integers(-(1 << b), 1 << b, n) for b in bits * terms]
    err = errors(mh, *f)
    assert np.abs(err).max() < 2.0 * terms and abs(err.mean()) < 0.02 * terms


@pytest.mark.parametrize("k", [0x71C71C71C71C71C7, 0x1999999999999A00, -0x1999999999999A00, 0x2B7E151628AED2A6,
                               -0x3243F6A8885A308D, 0x123456789ABCDEF0, 0x26D5A1B400000002, 0x3B9AC9FFFFFFFFFE])
@pytest.mark.parametrize("bits", [62, 50, 40])
def test_mean_error_with_a_constant(mh, k, bits):
    """As above with the low halves' product at its mean for this constant (half its low half), for
    factors whose lowest bit is zero: the same bounds; zero stays zero."""
    x = 2 * np.random.default_rng(bits).integers(-(1 << (bits - 1)), 1 << (bits - 1), 40_000)
    x[0] = 0
    out = np.zeros(len(x), np.int64)
    mh.mh_constant(len(x), k, x.ctypes.data, out.ctypes.data)
    err = np.array([((int(o) << 64) - k * int(v)) / 2.0**64 for o, v in zip(out, x)])
    assert out[0] == 0 and np.abs(err).max() < 2.0 and abs(err.mean()) < 0.02


def test_zero_factors(mh):
    rng = np.random.default_rng(1)
    x, z = rng.integers(-(1 << 62), 1 << 62, 500), np.zeros(500, np.int64)
    for f in ((x, z), (z, x), (z, z), (x, z, z, x), (z, z, z, z)):
        assert not errors(mh, *f).any()


@pytest.mark.gpu
@pytest.mark.parametrize("relax", [dict(), dict(kind=1, tau_l=0.6, visc_ratio=1.5), dict(tau_e=1.1, tau_nu=0.8, tau_q=1.2)])
def test_a_droplet_at_rest_gains_no_momentum(relax):
    """400 steps on 28 x 24. The nine populations of 672 nodes are rounded to 2^-53 of
    themselves (0.29 of that rms): a momentum of 2^-53 0.29 sqrt(sum f^2 c^2) / mass, about 5e-19
    of the mass per step and component (the liquid's 130 nodes carry it), a random walk of 1e-17
    in 400 steps, and the same from the moments' roundings. 1e-16 is asked for; products rounded
    down gave -2.3e-16 in both components."""
    torch = pytest.importorskip("torch")
    import paper_2107_06355_gb300 as P

    nx, ny = 28, 24
    eos = P.EOSParams(P.EOS_SMOOTH, 0.6, 0.387, 2.0, 0.834)
    sim = P.Simulation(nx, ny, P.BC_PERIODIC, eos, P.Relax(**relax))
    d = sim.derived()
    y, x = np.mgrid[0:ny, 0:nx]
    r = np.hypot(x - 13.6, y - 11.7)
    rho = d["rho_v"] + (d["rho_l"] - d["rho_v"]) * 0.5 * (1.0 - np.tanh(4.6 * (r - 6.0) / 8.0))
    sim.init_equilibrium(torch.tensor(rho, device="cuda"))
    sim.step(400)
    f = sim.get_f().cpu().numpy().astype(np.longdouble)
    sim.close()
    jx = (f[1] + f[5] + f[8] - f[3] - f[6] - f[7]).sum()
    jy = (f[2] + f[5] + f[6] - f[4] - f[7] - f[8]).sum()
    assert np.isfinite(f).all()
    assert abs(jx) < 1e-16 * f.sum() and abs(jy) < 1e-16 * f.sum()
