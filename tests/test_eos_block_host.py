"""Fixed-point factors of derived EOS blocks that no set-up made (unset, with a loop that has
no width, or not finite) and of collision constants that are not finite: they end, and the
nodes that they spoil are left to the double-precision form, which raises the error word
where psi is not finite."""
import os
import subprocess

import numpy as np
import pytest

from test_fixmul_host import HF, LI, RATES, ZS, fm, nodes  # noqa: F401

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("eosblock") / "eos_fix_block")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-o", exe,
                    os.path.join(ROOT, "tests", "native", "eos_fix_block_host.cpp")], check=True)
    return exe


def factors(exe, mode=1, **change):
    """(ok, loop, nodes in fixed point on the vapour branch, the loop, the liquid branch)"""
    args = [k if v is None else f"{k}={v!r}" for k, v in change.items()]
    out = subprocess.run([exe, str(mode), *args], capture_output=True, text=True, timeout=20, check=True)
    return tuple(map(int, out.stdout.split()))


@pytest.mark.parametrize("mode", [1, 3])
def test_a_block_of_a_set_up(program, mode):
    assert factors(program, mode) == (1, 1, 100, 100, 100)


@pytest.mark.parametrize("mode", [1, 3])
@pytest.mark.parametrize("change", [dict(rho_max=0.1, rho_min=0.1), dict(rho_max=0.1, rho_min=0.09),
                                    dict(rho_max=0.1, rho_min=0.1 + 1.4e-17),
                                    dict(rho_max=float("nan")), dict(rho_min=float("inf")), dict(a1sq=0.0),
                                    dict(a3sq=-1.0), dict(a1sq=float("inf")), dict(zero=None)])
def test_loops_without_a_width(program, mode, change):
    assert factors(program, mode, **change)[1] == 0


@pytest.mark.parametrize("mode", [1, 3])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_constants_that_are_not_finite(program, mode, bad):
    for key in ("p_max", "p_min"):  # the loop's branches with that constant; the C-S branches stay
        got = factors(program, mode, **{key: bad})[2:]
        assert got[0] == got[2] == 100 and got[1] < 100, key
    assert factors(program, mode, dP=bad)[2:] == (100, 100, 0)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("form, st, places", [(0, 0, (0, 1)), (0, 1, (0, 1, 2)), (1, 0, (0, 1, 4)), (1, 1, (0, 1, 2, 4)),
                                              (2, 0, (0, 9, 10)), (2, 1, (0, 2, 9, 10))])
def test_collision_constants_that_are_not_finite(fm, bad, form, st, places):  # noqa: F811
    """c: half_force, zz_scale, kappa_q, tau_a, tau_b, four rates, the Li term's scales; a node at
    rest in a uniform fluid, where every force is zero, included."""
    rows = np.zeros((20, 18))
    rows[:, :12] = nodes(np.random.default_rng(2), 20, -1, -0.5, 0.05, 0.05)[:, :12]
    rows[0, :9], rows[0, 10:12] = 0.5, 0.0
    if form == 2:
        rows[:, 12:14], rows[:, 14:16] = rows[:, 9:10] * [-2.0, 1.0], -rows[:, 10:12]
    good = np.array([HF, ZS, -0.5 / 24, 1.0, 0.0, *RATES, *LI])
    for k in (None, *places):
        c, out = good.copy(), np.zeros((20, 10))
        if k is not None:
            c[k] = bad
        fm.fm_collide(20, form, st, c.ctypes.data, rows.ctypes.data, out.ctypes.data)
        assert out[:, 9].tolist() == [float(k is None)] * 20, k


@pytest.mark.gpu
@pytest.mark.parametrize("key", ["p_max", "p_min", "dP", "eps"])
def test_step_noalloc_reports_a_block_that_is_not_finite(key):
    import ctypes as C

    torch = pytest.importorskip("torch")
    import lbm_inputs as I
    import paper_2107_06355_gb300 as P
    from paper_2107_06355_gb300 import _lib as L

    nx, ny = 32, 24
    sim = P.Simulation(nx, ny, P.BC_PERIODIC, P.EOSParams(P.EOS_SMOOTH, 0.6, 0.387, 2.0, 0.834), P.Relax())
    d = L.pplbm_eos_derived()
    assert L.lib().pplbm_get_derived(sim.ctx, C.byref(d)) == 0
    sim.init_equilibrium(I.planar(nx, ny, d.rho_v * 0.99, d.rho_l * 1.01, W=10.0))
    f, msg = sim.get_f(), C.c_char_p()
    g, h = torch.empty_like(f), torch.empty_like(f)
    relax, s = P.Relax().c(), C.c_void_p(torch.cuda.current_stream().cuda_stream)

    def step(src, dst):
        return L.lib().pplbm_step_noalloc(C.byref(sim.lattice), C.byref(d), C.byref(relax), C.c_void_p(src.data_ptr()),
                                          C.c_void_p(dst.data_ptr()), s, C.byref(msg))

    assert step(f, g) == L.PPLBM_OK and step(g, h) == L.PPLBM_OK
    setattr(d, key, float("nan"))
    # eps enters the collision: its populations are NaN, which the next step reports
    first = step(f, g)
    assert first == (L.PPLBM_OK if key == "eps" else L.PPLBM_ERR_DIVERGED)
    assert step(g, h) == L.PPLBM_ERR_DIVERGED
    sim.close()
