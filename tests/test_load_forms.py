"""Loads that the kernels may not use: every kernel may be resident while the one
that writes its inputs still runs, and the non-coherent path (ld.global.nc, __ldg,
const __restrict__) is for data that nothing writes during a kernel's life."""
import glob
import os
import re

import pytest

from paper_2608_02625_gb300 import build


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(build.CSRC, "*.cu*"))), ids=os.path.basename)
def test_no_non_coherent_loads(path):
    code = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
    assert not re.search(r"ld\.global[.\w:]*\.nc\b|\b__ldg\b|__restrict", code)
