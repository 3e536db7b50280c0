"""The fixed-point EOS and psi (csrc/eos_fixed.cuh), built for the host from the same
source, against 60-digit decimal arithmetic on the set-up's own constants: every branch
of the C-S, Smooth C-S and Modified Smooth equations of state, several T_r, G and b."""
import ctypes as C
import math
import os
import subprocess
from decimal import Decimal as D
from decimal import getcontext

import numpy as np
import pytest

getcontext().prec = 60
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NAMES = "G b RT_l RT_v a_l a_v dP rho_v rho_max rho_min rho_l p_max b1 a1sq p_min b3 a3sq".split()


@pytest.fixture(scope="module")
def ef(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("eosfix") / "libeos_fixed_host.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-o", so,
                    os.path.join(ROOT, "tests", "native", "eos_fixed_host.cpp")], check=True)
    lib = C.CDLL(so)
    lib.ef_setup.argtypes = [C.c_void_p, C.c_double, C.c_void_p]
    lib.ef_psi.argtypes = [C.c_void_p, C.c_double, C.c_longlong, C.c_void_p, C.c_void_p, C.c_void_p]
    lib.ef_sqrt.argtypes = [C.c_longlong, C.c_void_p, C.c_void_p, C.c_void_p]
    return lib


def exact_psi(mode, e, rho):
    r = D(float(rho))
    cs = lambda a, RT: r * RT * (1 + h + h * h - h**3) / (1 - h)**3 - a * r * r  # noqa: E731
    h = e["b"] / 4 * r
    if mode == 0 or r >= e["rho_l"]:
        p = cs(e["a_l"], e["RT_l"]) + (e["dP"] if mode else 0)
    elif r <= e["rho_v"]:
        p = cs(e["a_v"], e["RT_v"])
    elif r <= e["rho_max"]:
        p = e["p_max"] - e["b1"] + e["b1"] * (1 - (r - e["rho_max"])**2 / e["a1sq"]).sqrt()
    elif r < e["rho_min"]:
        t = (r - e["rho_max"]) / (e["rho_min"] - e["rho_max"])
        p = e["p_max"] + (e["p_min"] - e["p_max"]) * t * t * (3 - 2 * t)
    else:
        p = e["p_min"] + e["b3"] - e["b3"] * (1 - (r - e["rho_min"])**2 / e["a3sq"]).sqrt()
    return (2 / e["G"] * (p - r / 3)).sqrt(), abs(2 / e["G"]) * max(abs(p), abs(r / 3))


CASES = [(0, 0.6, 0.387, 0.387, 4.0, 0.5, -1.0), (0, 0.9, 0.5, 0.5, 4.0, 0.5, -1.0),
         (1, 0.35, 0.363, 2.0, 4.0, 0.838, -1.0), (1, 0.5, 0.363, 2.0, 4.0, 0.775, -1.0),
         (1, 0.5, 0.5, 0.5, 4.0, 0.610, -1.0), (1, 0.8, 0.5, 0.5, 4.0, 0.342, -1.0),
         (1, 0.95, 0.363, 2.0, 4.0, 0.775, -1.0), (1, 0.6, 0.387, 2.0, 4.0, 0.834, -3.0),
         (1, 0.5, 0.363, 2.0, 2.0, 0.775, -0.25), (3, 0.6, 0.387, 2.0, 4.0, 0.446, -1.0)]


@pytest.mark.parametrize("mode, Tr, al, av, b, alpha, G", CASES)
def test_psi_of_every_branch(ef, mode, Tr, al, av, b, alpha, G):
    """psi is within half its ulp plus the error of psi^2, halved and divided by psi: on the
    C-S branches at most 24 units of 2^-57 of rho (three products and the constants, each
    below 4 units of x's frame, and the final product), on the loop 2^-57 of the largest
    constant of the branch, divided by the ellipse's root s (an error of the radicand is
    divided by 2 s), and 6 units of the sum's frame 2^(e - 1081 + s) <= 2 k3 rho 2^-58 (the
    three terms' products and shifts)."""
    par = np.array([mode, Tr, al, av, b, 1.0, alpha, 0.0])
    v = np.zeros(17)
    assert ef.ef_setup(par.ctypes.data, G, v.ctypes.data) == 0
    e = {k: D(x) for k, x in zip(NAMES, v.tolist())}
    rng = np.random.default_rng(3)
    f = dict(zip(NAMES, v.tolist()))
    edges = [f["rho_v"] * 0.3, f["rho_v"], f["rho_max"], f["rho_min"], f["rho_l"], min(1.1 * f["rho_l"], 2.39 / b)]
    rho = np.concatenate([np.exp(rng.uniform(np.log(lo), np.log(hi), 120)) for lo, hi in zip(edges, edges[1:])])
    rho = np.concatenate([rho, [np.nextafter(x, s) for x in edges[1:5] for s in (0.0, 1.0)], edges[1:5]])
    psi, ok = np.zeros(len(rho)), np.zeros(len(rho), np.int32)
    assert ef.ef_psi(par.ctypes.data, G, len(rho), rho.ctypes.data, psi.ctypes.data, ok.ctypes.data) == 0
    assert ok.all()
    sc = abs(2 / e["G"])
    for r, got in zip(rho, psi):
        want, size = exact_psi(mode, e, r)
        bulk = mode == 0 or r <= f["rho_v"] or r >= f["rho_l"]
        k3 = 2 ** D(math.ceil(math.log2(2 / (3 * abs(G)))))
        if bulk:
            err2 = k3 * D(float(r)) * 24 / D(2)**57
        else:
            big = max(D(abs(x)) for x in ((e["b1"], e["p_max"]) if r <= f["rho_max"] else
                                          (e["b3"], e["p_min"]) if r >= f["rho_min"] else (e["p_max"], e["p_min"])))
            root = D(1)
            if r <= f["rho_max"]:
                root = (1 - (D(float(r)) - e["rho_max"])**2 / e["a1sq"]).sqrt()
            elif r >= f["rho_min"]:
                root = (1 - (D(float(r)) - e["rho_min"])**2 / e["a3sq"]).sqrt()
            err2 = sc * big / D(2)**57 / root + 6 * size / D(2)**57
        tol = D(math.ulp(got)) / 2 + err2 / (2 * want)
        assert abs(D(float(got)) - want) <= tol, (float(r), float(got), float((D(float(got)) - want) / D(math.ulp(got))))


def test_outside_the_domain(ef):
    """b not a power of two, the Peng loop, eta from 0.6 on, psi^2 <= 0: reported."""
    def ok_of(par, G, rho):
        par, rho = np.array(par), np.array(rho)
        psi, ok = np.zeros(len(rho)), np.zeros(len(rho), np.int32)
        assert ef.ef_psi(par.ctypes.data, G, len(rho), rho.ctypes.data, psi.ctypes.data, ok.ctypes.data) == 0
        return ok.tolist()

    assert ok_of([0, 0.6, 0.387, 0.387, 3.0, 1.0, 0.5, 0.0], -1.0, [0.1, 0.5]) == [0, 0]
    # Peng: the bulk branches in fixed point, the loop not
    assert ok_of([2, 0.6, 0.387, 0.387, 4.0, 1.0, 0.5, 0.45], -1.0, [1e-3, 0.1, 0.42]) == [1, 0, 1]
    smooth = [1, 0.5, 0.363, 2.0, 4.0, 1.0, 0.775, 0.0]
    assert ok_of(smooth, -1.0, [0.59, 0.6, 0.9, 1.0, 5.0, 1e300]) == [1, 0, 0, 0, 0, 0]


def test_square_root(ef):
    rng = np.random.default_rng(4)
    P = np.maximum(rng.integers(2**32, 2**63 - 1, 3000, dtype=np.int64) >> rng.integers(0, 30, 3000), 2**32)
    P[:5] = [2**62, 2**62 - 1, 2**62 + 1, 2**32, 2**63 - 1]
    ex = rng.integers(-120, 120, 3000).astype(np.int32)
    out = np.zeros(3000)
    ef.ef_sqrt(3000, P.ctypes.data, ex.ctypes.data, out.ctypes.data)
    for p, k, got in zip(P.tolist(), ex.tolist(), out.tolist()):
        want = (D(p) * D(2)**k).sqrt()
        assert abs(D(got) - want) <= D(math.ulp(got)) * (D(1) / 2 + D(3) / 2**7)
