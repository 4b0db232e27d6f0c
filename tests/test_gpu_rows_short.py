"""GPU parity of the selective decode's gather with short rows: as many rows as
a chunk's window holds and one more or less, several windows a chunk, and more
rows than all of a chunk's windows hold (nearly all empty).  Decoding is exact:
no tolerance."""
import numpy as np
import pytest

import synth
from gpu_util import make_column
from test_gpu_rows import Rows
from test_gpu_rows_gather import CODECS, TOKENS, fp, same  # noqa: F401  (fp: the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("codec", CODECS)
@pytest.mark.parametrize("empty", [0, 1, 2, 40])
def test_windows(fp, codec, empty):  # noqa: F811
    """Rows of one or two codes with `empty` empty rows on average between them."""
    rng = np.random.default_rng(10 * codec + empty)
    lens = rng.integers(1, 3, 5000) * (rng.random(5000) * (empty + 1) < 1)
    offs = np.concatenate([[0], np.cumsum(lens)])
    r = Rows(fp, make_column(codec, TOKENS, rng.integers(0, 4, offs[-1]), offs))
    for m in (1, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1024, 5000):
        same(r, np.arange(m, dtype=np.uint32))
        same(r, rng.integers(0, 5000, m).astype(np.uint32))


@pytest.mark.parametrize("codec", CODECS)
@pytest.mark.parametrize("gap", [17, 300, 5000])
def test_rows_past_all_windows(fp, codec, gap):  # noqa: F811
    rng = np.random.default_rng(codec + gap)
    lens = np.zeros(60 * gap, int)
    lens[gap - 1::gap] = rng.integers(1, 30, 60)
    offs = np.concatenate([[0], np.cumsum(lens)])
    r = Rows(fp, make_column(codec, TOKENS, rng.integers(0, 4, offs[-1]), offs))
    same(r, np.arange(lens.size, dtype=np.uint32))
    same(r, np.arange(lens.size, dtype=np.uint32)[::-1].copy())
