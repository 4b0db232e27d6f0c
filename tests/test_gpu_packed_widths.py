"""Cascaded codes at every width: each has its own unpacking body, odd widths
put every second lane's codes in the middle of a word, and a lane reads only
the words that hold its codes -- up to the very end of the code buffer."""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_packed import fp, pack_bits, run, small_dict  # noqa: F401  (fp: the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("codec,b", [(c, b) for c in (synth.ONPAIR16, synth.ONPAIR12, synth.FSST12)
                                     for b in range(1, synth.CODE_BITS[c] + 1)])
def test_width(fp, codec, b):  # noqa: F811
    rng = np.random.default_rng(900 + b)
    n_entries = min(1 << b, 5000 if b > 12 else 4096)
    d = small_dict(codec, n_entries, rng)
    for n in (16, 31, 512, 1024, 1025, 5 * 512 + 16, 8192 + 496):
        codes = rng.integers(0, n_entries, n).astype(np.uint32)
        codes[-16:] = n_entries - 1
        stream = pack_bits(codes, b)   # ends with the last code's byte: no padding to a word
        cuts = np.sort(rng.integers(0, n, n // 9))
        for first in (0, n // 3):      # whole, and a slice from an odd slot on
            co = np.concatenate([[first], np.maximum(cuts, first), [n]]).astype(np.uint32)
            st, ref, out, offs, guard_ok = run(fp, codec, d, b, stream, co)
            assert ref.status == oracle.OK and st == fp.OK and guard_ok, (b, n, first)
            np.testing.assert_array_equal(offs, ref.offsets)
            assert np.array_equal(out[:ref.total], ref.data), (b, n, first)
