"""The built-in decode shapes, with no tuned ones loaded: OnPair-12 stages its
table in shared memory at every size."""
import os

import pytest


@pytest.mark.parametrize("bytes_", [16, 1 << 16, 1 << 18, 3 << 18, 1 << 20, 1 << 22, 1 << 23, 1 << 24, 1 << 30])
def test_onpair12_stages_its_table(bytes_):
    import paper_2609_15034_gb300 as fp
    fp.tune_clear()
    try:
        v = fp.variant_for(fp.ONPAIR12, bytes_)   # read width 8
        assert fp.variant_width(fp.ONPAIR12, v) == 8
        assert fp.variant_info(fp.ONPAIR12, v)["dict_in_smem"]
    finally:
        fp.tune_load(os.path.join(os.path.dirname(fp.__file__), "tuning", "gb300.txt"))
