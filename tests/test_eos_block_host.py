"""Fixed-point factors of derived EOS blocks that no set-up made (unset, or with a loop that
has no width): they end, and the loop's branches are left to the double-precision form."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LOOP = dict(rho_v=1e-3, rho_max=0.05, rho_min=0.3, rho_l=0.4, p_max=6e-3, p_min=4e-3, a1sq=0.01, a3sq=0.04)


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("eosblock") / "eos_fix_block")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-o", exe,
                    os.path.join(ROOT, "tests", "native", "eos_fix_block_host.cpp")], check=True)
    return exe


def factors(exe, mode=1, b=4.0, G=-1.0, **loop):
    v = [mode, b, G, *(loop.get(k, 0.0) for k in LOOP)]
    out = subprocess.run([exe, *map(repr, map(float, v))], capture_output=True, text=True, timeout=20, check=True)
    ok, on = map(int, out.stdout.split())
    return ok, on


def test_a_block_of_a_set_up(program):
    assert factors(program, **LOOP) == (1, 1)


@pytest.mark.parametrize("mode", [1, 3])
@pytest.mark.parametrize("change", [dict(rho_min=0.05), dict(rho_min=0.04), dict(rho_min=0.05 + 7e-18),
                                    dict(rho_max=float("nan")), dict(rho_min=float("inf")), dict(a1sq=0.0),
                                    dict(a3sq=-1.0), dict(a1sq=float("inf")),
                                    dict.fromkeys(LOOP, 0.0)])
def test_loops_without_a_width(program, mode, change):
    assert factors(program, mode, **{**LOOP, **change})[1] == 0
