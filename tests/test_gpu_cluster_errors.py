"""The one-cluster decode of columns that are corrupt in some lanes only: the
lanes that found nothing wrong meet the others at the last barrier, the call
reports the corruption, keeps every write in bounds, and the next call is
normal."""
import numpy as np
import pytest

import synth
from gpu_util import DeviceColumn, assert_same, make_column

pytestmark = pytest.mark.gpu

CODECS = [synth.ONPAIR16, synth.ONPAIR12, synth.FSST8, synth.FSST12]


@pytest.mark.parametrize("codec", CODECS)
@pytest.mark.parametrize("step", [17, 256, 1021, 30_000])
def test_corrupt_in_some_lanes(codec, step):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15034_gb300 as fp
    rng = np.random.default_rng(step + codec)
    toks = [b"ab", b"c", b"defg", b"hi"]
    n = 60_000
    slots = rng.integers(0, len(toks), n)
    offs = np.sort(np.concatenate([[0, n], rng.integers(0, n + 1, n // 9)]))
    good = make_column(codec, toks, slots, offs)
    bad = slots.copy()
    bad[step // 2::step] = len(toks)   # a code past the dictionary
    dc = DeviceColumn(make_column(codec, toks, bad, offs))
    launches = fp.variant_info(codec, fp.variant_for_dict(dc.dict, dc.codes_bytes))["launches_per_call"]
    assert launches == 1
    for _ in range(3):
        st, _, _, guard_ok, _ = dc.decode(capacity=8 * n)
        assert st == fp.ERR_CORRUPT and guard_ok
    assert_same(good)
