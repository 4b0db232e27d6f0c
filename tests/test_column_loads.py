"""Launches that may start while the kernel that writes the column still runs
never read the column through the read-only path (`ld.global.nc`, __ldg), whose
data must not change while the kernel runs.  (The block pipeline of
fp_decoder.cuh starts by ordinary launches.)"""
import os
import re

import pytest

from paper_2609_15034_gb300 import _build


@pytest.mark.parametrize("name", ["fp_warp.cuh", "fp_reduce.cuh", "fp_cluster.cuh"])
def test_no_read_only_loads_of_the_column(name):
    with open(os.path.join(_build.CSRC, name)) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    assert "global.nc" not in code
    assert not re.search(r"__ldg\([^;]*\b(codes|code_offsets)\b", code)
