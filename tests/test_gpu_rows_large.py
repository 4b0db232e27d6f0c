"""GPU parity of the selective decode on code buffers of 16 GiB and more (the
rows in use lie at the front, or just below slot 2^32): the gather's words are
counted without loss.  Decoding is exact: no tolerance."""
import numpy as np
import pytest

import synth
from gpu_util import store_slots

pytestmark = pytest.mark.gpu

TOKENS = [b"a", b"bcd", b"efghijkl", b"mn", b"opq"]


@pytest.mark.parametrize("codec", [synth.ONPAIR16, synth.ONPAIR12, synth.FSST8, synth.FSST12])
@pytest.mark.parametrize("size", [1 << 34, (1 << 34) + 258])
@pytest.mark.parametrize("place", ["front", "far"])
def test_rows_of_a_large_buffer(codec, size, place):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15034_gb300 as fp
    if torch.cuda.mem_get_info()[0] < size + (2 << 30):
        pytest.skip("not enough device memory")
    rng = np.random.default_rng(codec)
    n = 700
    starts = np.concatenate([[0], np.cumsum(rng.integers(0, 40, n))])
    slots = rng.integers(0, len(TOKENS), int(starts[-1]))
    first = 0 if place == "front" else ((1 << 32) - 1 - slots.size) // 32 * 32
    stored = store_slots(codec, slots)
    buf = torch.empty(size, dtype=torch.uint8, device="cuda")
    at = first * synth.CODE_BITS[codec] // 8
    buf[at:at + stored.size] = torch.from_numpy(np.ascontiguousarray(stored)).cuda()
    co = torch.from_numpy((starts + first).astype(np.uint32).view(np.int32)).cuda()
    d = synth.Dictionary.from_tokens(codec, TOKENS)
    dic = fp.Dict(codec, d.data, d.offsets)
    rows = rng.integers(0, n, 1500)
    ids = torch.from_numpy(rows.astype(np.int32)).cuda()
    strings = [b"".join(TOKENS[s] for s in slots[starts[r]:starts[r + 1]]) for r in rows]
    want = np.frombuffer(b"".join(strings), np.uint8)
    want_offsets = np.concatenate([[0], np.cumsum([len(s) for s in strings])])
    st, n_slots, n_bytes = fp.rows_size(codec, dic, buf.data_ptr(), size, co.data_ptr(), n, ids.data_ptr(), rows.size)
    assert st == fp.OK and n_bytes == want.size, fp.last_error()
    out = torch.zeros(n_bytes, dtype=torch.uint8, device="cuda")
    offs = torch.zeros(rows.size + 1, dtype=torch.int32, device="cuda")
    fp.decode_rows(codec, dic, buf.data_ptr(), size, co.data_ptr(), n, ids.data_ptr(), rows.size, n_slots,
                   out.data_ptr(), n_bytes, offs.data_ptr())
    assert fp.sync_status() == fp.OK, fp.last_error()
    np.testing.assert_array_equal(offs.cpu().numpy(), want_offsets)
    assert np.array_equal(out.cpu().numpy(), want)
