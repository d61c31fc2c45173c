"""Loads through the non-coherent path (ld.global.nc, __ldg, const __restrict__)
are for memory that nothing writes while a kernel runs.  Kernels launched with
programmatic stream serialisation run while the previous kernel still writes its
results, so only what has to be in place before that may be read so: the block
table."""
import glob
import os
import re

import pytest

from paper_2505_12728_gb300 import build_lib

FILES = sorted(glob.glob(os.path.join(build_lib.CSRC, "*.cu*")))


@pytest.mark.parametrize("path", FILES, ids=[os.path.basename(f) for f in FILES])
def test_no_noncoherent_loads_of_what_a_previous_kernel_writes(path):
    code = re.sub(r"//[^\n]*", "", open(path).read())
    loads = [line.strip() for line in code.splitlines()
             if re.search(r"__ldg\s*\(|\.nc\b|__restrict__", line) and "p.block_table" not in line]
    assert not loads
