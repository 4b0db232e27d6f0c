"""GPU parity of columns with as many strings as the API takes: every code is the
token "a", so the output offsets are the code offsets.  With a long last string
the last tile owns one boundary, the last before 2^32.  Decoding is exact: no
tolerance."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("last", [0, 5000])
def test_most_strings(last):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15034_gb300 as fp
    if torch.cuda.mem_get_info()[0] < 50 << 30:
        pytest.skip("not enough device memory")
    n, slots = (1 << 32) - 2, 1 << 30
    dic = fp.Dict(synth.ONPAIR16, np.frombuffer(b"a", np.uint8), np.array([0, 1], np.uint32))
    codes = torch.zeros(2 * slots, dtype=torch.uint8, device="cuda")
    co = torch.empty(n + 1, dtype=torch.int32, device="cuda")
    step = 1 << 27
    for a in range(0, n + 1, step):
        i = torch.arange(a, min(a + step, n + 1), dtype=torch.int64, device="cuda")
        co[a:a + step] = torch.where(i < n, (i * slots // n).clamp_(max=slots - last), slots).to(torch.int32)
    out = torch.zeros(slots, dtype=torch.uint8, device="cuda")
    offs = torch.full((n + 1,), -1, dtype=torch.int32, device="cuda")
    fp.decode(synth.ONPAIR16, dic, codes.data_ptr(), codes.numel(), co.data_ptr(), n, out.data_ptr(), out.numel(),
              offs.data_ptr())
    assert fp.sync_status() == fp.OK, fp.last_error()
    assert bool((out == 97).all())
    for a in range(0, n + 1, step):
        assert torch.equal(offs[a:a + step], co[a:a + step])
    del codes, co, out, offs
    torch.cuda.empty_cache()
