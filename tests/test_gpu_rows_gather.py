"""GPU parity of the selective decode's gather where a chunk's rows leave its
window: many short or empty rows, rows longer than chunks, the last bytes of
the stored stream, selections of more than 8 M rows (the block sums scanned by
a launch of their own).  Decoding is exact: no tolerance."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import make_column
from test_gpu_rows import Rows

pytestmark = pytest.mark.gpu

CODECS = [synth.ONPAIR16, synth.ONPAIR12, synth.FSST8, synth.FSST12]
TOKENS = [b"a", b"bcd", b"efghijkl", b"mn"]


@pytest.fixture(scope="module")
def fp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15034_gb300 as m
    return m


def same(r, rows):
    st, ref, out, offs, guard_ok = r.run(rows)
    assert ref.status == oracle.OK
    assert st == r.fp.OK and guard_ok, r.fp.last_error()
    np.testing.assert_array_equal(offs, ref.offsets)
    assert np.array_equal(out[:ref.total], ref.data)


@pytest.mark.parametrize("codec", CODECS)
@pytest.mark.parametrize("kind", ["mostly_empty", "one_code", "long", "mixed"])
@pytest.mark.parametrize("extra", [0, 1, 2, 3])
def test_rows_outside_the_window(fp, codec, kind, extra):
    rng = np.random.default_rng(codec * 10 + extra)
    n = 4000
    lens = {"mostly_empty": (rng.random(n) < 0.01) * rng.integers(1, 40, n), "one_code": np.ones(n, int),
            "long": rng.integers(900, 3000, 60), "mixed": rng.integers(0, 2, n) * rng.integers(0, 30, n)}[kind]
    lens[-1] += extra
    offs = np.concatenate([[0], np.cumsum(lens)])
    r = Rows(fp, make_column(codec, TOKENS, rng.integers(0, 4, offs[-1]), offs))
    m = len(lens)
    same(r, rng.integers(0, m, 2 * m).astype(np.uint32))
    same(r, np.arange(m, dtype=np.uint32))
    same(r, np.full(300, m - 1, np.uint32))


def test_more_rows_than_blocks_add_up(fp):
    rng = np.random.default_rng(1)
    offs = np.concatenate([[0], np.cumsum(rng.integers(0, 3, 5000))])
    r = Rows(fp, make_column(synth.ONPAIR12, TOKENS, rng.integers(0, 4, offs[-1]), offs))
    same(r, rng.integers(0, 5000, 8_400_000).astype(np.uint32))
