"""GPU parity of the staged assembly of a warp tile: tiles whose bytes pass
the staging area (several rounds), tiles of one-byte tokens, every alignment
of the output, tiles that end inside a word or a 16-byte chunk, and strings
denser than the boundaries fetched ahead.  Decoding is exact: no tolerance."""
import numpy as np
import pytest

import synth
from gpu_util import DeviceColumn, assert_same, make_column

pytestmark = pytest.mark.gpu

CODECS = [synth.ONPAIR16, synth.ONPAIR12, synth.FSST8, synth.FSST12]


@pytest.fixture(scope="module")
def fp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15034_gb300 as m
    yield m
    for c in CODECS:
        m.variant_select(c, -1)


def tokens(codec, lengths, rng):
    top = synth.MAX_TOKEN[codec]
    return [rng.integers(0, 256, top if L == 0 else min(L, top), dtype=np.uint8).tobytes() for L in lengths]


# token lengths of the dictionary (0: the codec's longest)
LENGTHS = {"longest": [0], "one": [1], "mixed": list(range(1, 17)), "edges": [1, 3, 4, 5, 8, 12, 15, 0]}


@pytest.mark.parametrize("codec", CODECS)
@pytest.mark.parametrize("kind", list(LENGTHS))
@pytest.mark.parametrize("n_slots", [1, 17, 512, 1024, 1025, 5003])
def test_staged_tiles(fp, codec, kind, n_slots):
    rng = np.random.default_rng(n_slots * 10 + codec)
    toks = tokens(codec, LENGTHS[kind], rng)
    slots = rng.integers(0, len(toks), n_slots)
    for start, per in ((0, 1), (min(3, n_slots), 40)):
        # strings of 0..2 per slots; a start past slot 0 moves every tile's alignment
        cuts = np.unique(np.concatenate([[start, n_slots], rng.integers(start, n_slots + 1, n_slots // per + 1)]))
        offs = np.sort(np.concatenate([cuts, cuts[: len(cuts) // 2]]))
        col = make_column(codec, toks, slots, offs)
        dc = DeviceColumn(col)
        try:
            for v in range(fp.variant_count(codec)):
                fp.variant_select(codec, v)
                assert_same(col, dc)
        finally:
            fp.variant_select(codec, -1)


@pytest.mark.parametrize("codec", [synth.ONPAIR16, synth.ONPAIR12, synth.FSST12])
def test_staged_tiles_of_packed_codes(fp, codec):
    import torch
    rng = np.random.default_rng(codec)
    toks = tokens(codec, LENGTHS["edges"] + [0] * 8, rng)
    slots = rng.integers(0, len(toks), 4099)
    offs = np.concatenate([[0], np.sort(rng.integers(0, 4100, 3000)), [4099]])
    col = make_column(codec, toks, slots, offs)
    dc = DeviceColumn(col)
    _, data, want, _, _ = dc.decode()
    packed = torch.from_numpy(synth.pack_bits(slots, 5)).cuda()
    out = torch.zeros(data.size, dtype=torch.uint8, device="cuda")
    out_offsets = torch.zeros(offs.size, dtype=torch.int32, device="cuda")
    fp.decode_packed(codec, dc.dict, 5, packed.data_ptr(), packed.numel(), dc.code_offsets.data_ptr(), dc.n_strings,
                     out.data_ptr(), out.numel(), out_offsets.data_ptr())
    assert fp.sync_status() == fp.OK
    np.testing.assert_array_equal(out.cpu().numpy(), data)
    np.testing.assert_array_equal(out_offsets.cpu().numpy().view(np.uint32), want)
