"""GPU parity of small columns around the lines of the one-cluster decode: by
code slots and by strings (columns of many mostly empty strings take three
launches), for whole columns and for selected rows.  Decoding is exact: no tolerance."""
import numpy as np
import pytest

import synth
from gpu_util import DeviceColumn, assert_same, make_column
from test_gpu_rows import Rows
from test_gpu_rows_gather import CODECS, TOKENS, fp, same  # noqa: F401  (fp: the module's fixture)

pytestmark = pytest.mark.gpu


def column(codec, n_slots, n_strings, rng):
    offs = np.sort(np.concatenate([[0, n_slots], rng.integers(0, n_slots + 1, n_strings - 1)]))
    return make_column(codec, TOKENS, rng.integers(0, 4, n_slots), offs)


@pytest.mark.parametrize("codec", CODECS)
def test_line_by_slots(fp, codec):  # noqa: F811
    rng = np.random.default_rng(codec)
    for n_slots, launches in (((1 << 17) - 2, 1), (1 << 17, 3)):
        dc = DeviceColumn(column(codec, n_slots, 5000, rng))
        v = fp.variant_for_dict(dc.dict, dc.codes_bytes)
        assert fp.variant_info(codec, v)["launches_per_call"] == launches
        assert_same(dc.col, dc)


@pytest.mark.parametrize("codec", CODECS)
@pytest.mark.parametrize("n_strings", [(1 << 17) - 1, 1 << 17, (1 << 17) + 1, 1_000_000])
@pytest.mark.parametrize("n_slots", [0, 1, 40_000, 130_000])
def test_line_by_strings(fp, codec, n_strings, n_slots):  # noqa: F811
    rng = np.random.default_rng(n_strings + codec)
    assert_same(column(codec, n_slots, n_strings, rng))


@pytest.mark.parametrize("codec", CODECS)
@pytest.mark.parametrize("n_rows", [(1 << 17) - 1, 1 << 17])
def test_rows_by_strings(fp, codec, n_rows):  # noqa: F811
    rng = np.random.default_rng(n_rows + codec)
    same(Rows(fp, column(codec, 9000, 30_000, rng)), rng.integers(0, 30_000, n_rows).astype(np.uint32))
