"""The EOS set-up on a caller's thread with a small stack: its quadrature nodes (150 KB) are not
kept there. Run in a child process, which an overflow would end."""
import subprocess
import sys

import pytest

CHILD = """
import ctypes as C, threading
import paper_2107_06355_gb300 as P
from paper_2107_06355_gb300 import _lib as L
lib, p, d, out = L.lib(), P.EOSParams(%d, 0.6, 0.387, %r, %r, r_theta=%r).c(), L.pplbm_eos_derived(), []
threading.stack_size(96 * 1024)
t = threading.Thread(target=lambda: out.append(lib.pplbm_eos_setup(C.byref(p), -1.0, C.byref(d))))
t.start()
t.join()
print(out, d.psi_l > 0.0)
"""


@pytest.mark.parametrize("mode, a_v, alpha, r_theta", [(0, 0.387, 0.5, 0.0), (1, 2.0, 0.834, 0.0), (2, 0.387, 0.5, 0.45),
                                                       (3, 2.0, 0.446, 0.0)])
def test_set_up_on_a_small_stack(mode, a_v, alpha, r_theta):
    from paper_2107_06355_gb300 import build

    build.build()
    r = subprocess.run([sys.executable, "-c", CHILD % (mode, a_v, alpha, r_theta)], capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and r.stdout.split("\n")[0] == "[0] True", (r.returncode, r.stderr[-500:])
