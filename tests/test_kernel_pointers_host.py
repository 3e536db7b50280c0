"""Fields that a kernel writes are not marked `const __restrict__` where they are read: the
mark lets the compiler take the read-only path, for data unchanged during the whole kernel.
A kernel launched dependent on its predecessor is resident while that one still writes the
field, and the kernels that run several steps write it themselves."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_06355_gb300", "csrc")


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_no_read_only_mark_on_a_field(path):
    src = open(path).read()
    assert not re.findall(r"const\s+double\s*\*\s*__restrict__\s*\w+|__ldg\s*\(|ld\.global\.nc", src)
    # a dependent kernel's own parameters carry no alias promise across its wait
    for head in re.findall(r"__global__[^{]*\)\s*\{\s*(?:using namespace \w+;\s*)?begin_dependent", src):
        assert "__restrict__" not in head, head
