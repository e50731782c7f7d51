"""A kernel that may start while its predecessor still writes must not read that data as if it were read-only for the
kernel's lifetime: a const __restrict__ parameter or __ldg lets the compiler use the non-coherent path and move the load
above the wait.  That cannot be provoked at will, so the sources are checked."""
import os
import re

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2608_23834_b200", "csrc")


@pytest.mark.parametrize("name", ["lifecycle_kernels.cu", "demote_warp.cuh", "promote_warp.cuh", "decode_tensor.cu", "decode_cut.cuh"])
def test_no_read_only_loads_in_kernels_that_start_early(name):
    with open(os.path.join(CSRC, name)) as f:
        code = re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)
    assert not re.findall(r"__ldg\b|ld\.global\.nc|\bconst\s+\w+\s*\*\s*__restrict__", code)
