"""Resources of the compiled kernels, from the compiler's own report (no GPU)."""

import os
import re

import pytest

from paper_1408_4675_gb300 import build


@pytest.mark.parametrize("unit", ["kernels_x", "kernels_xvel", "kernels_adj"])
def test_row_kernels_reserve_only_the_barriers_they_use(unit):
    """The CTA's barrier and one per team of a CTA (two teams at most).  A barrier
    id that is not a literal reserves all 16, which limits the CTAs per SM."""
    build.build()
    log = open(os.path.join(build.BUILD, unit + ".ptxas.txt")).read()
    used = [int(n) for n in re.findall(r"used (\d+) barriers", log)]
    assert used and max(used) <= 3
