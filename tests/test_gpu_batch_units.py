"""GPU parity of the staged batch configuration (units of a chunk's tiles,
tables in shared memory): chunks around unit and warp edges, chunks that share
a dictionary and chunks that do not, slices, empty chunks, every codec mix, an
error that stays with its chunk.  Decoding is exact: no tolerance."""
import numpy as np
import pytest

import synth
from gpu_util import DeviceColumn, make_column, oracle_decode

pytestmark = pytest.mark.gpu

CODECS = [synth.ONPAIR16, synth.ONPAIR12, synth.FSST8, synth.FSST12]
TILE = {synth.ONPAIR16: 512, synth.ONPAIR12: 512, synth.FSST8: 1024, synth.FSST12: 512}
TILES = [0, 1, 2, 15, 16, 17, 127, 128, 129, 300]


@pytest.fixture(scope="module")
def fp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15034_gb300 as m
    return m


def column(codec, tiles, k, rng, shared):
    toks = shared[codec] if k % 3 else [rng.integers(0, 256, 1 + i % synth.MAX_TOKEN[codec], dtype=np.uint8).tobytes()
                                        for i in range(100)]
    n = max(0, tiles * TILE[codec] - (k % 4))   # short of a tile's end by 0 .. 3 slots
    first = min(n, 5 * (k % 2))
    slots = rng.integers(0, len(toks), n)
    offs = np.sort(np.concatenate([[first, n], rng.integers(first, n + 1, n // 11)]))
    return make_column(codec, toks, slots, offs)


def run(fp, cols, dicts=None):
    import torch
    config = fp.batch_config_count() - 1
    dcs = [DeviceColumn(c) for c in cols]
    refs = [oracle_decode(c) for c in cols]
    outs = [torch.full((r.total + 64,), 0xA5, dtype=torch.uint8, device="cuda") for r in refs]
    offs = [torch.full((c.n_strings + 1,), -1, dtype=torch.int32, device="cuda") for c in cols]
    by_dict = {}   # chunks with the same tokens share one device dictionary
    chunks = []
    for c, dc, r, o, f in zip(cols, dcs, refs, outs, offs):
        d = by_dict.setdefault((c.codec, c.dictionary.data.tobytes()), dc.dict)
        chunks.append(fp.chunk(c.codec, d, dc.codes.data_ptr(), dc.codes_bytes, dc.code_offsets.data_ptr(), c.n_strings,
                               o.data_ptr(), r.total, f.data_ptr()))
    plan = fp.Plan(chunks, config=config)
    for _ in range(3):
        plan.decode()
    st, sts, tot = plan.sync_status()
    return st, sts, tot, refs, outs, offs


@pytest.mark.parametrize("codecs", [[c] for c in CODECS] + [CODECS, CODECS[1:3]])
def test_units(fp, codecs):
    rng = np.random.default_rng(len(codecs) * 10 + codecs[0])
    shared = {c: [rng.integers(0, 256, 1 + i % synth.MAX_TOKEN[c], dtype=np.uint8).tobytes() for i in range(90)]
              for c in CODECS}
    cols = [column(c, t, k, rng, shared) for k, t in enumerate(TILES) for c in codecs]
    st, sts, tot, refs, outs, offs = run(fp, cols)
    assert st == fp.OK, fp.last_error()
    for k, (r, o, f) in enumerate(zip(refs, outs, offs)):
        assert tot[k] == r.total
        h = o.cpu().numpy()
        assert np.array_equal(h[:r.total], r.data), k
        assert np.all(h[r.total:] == 0xA5), k
        np.testing.assert_array_equal(f.cpu().numpy().view(np.uint32), r.offsets, err_msg=str(k))


def test_an_error_stays_with_its_chunk(fp):
    rng = np.random.default_rng(3)
    shared = {c: [b"ab", b"c"] * 20 for c in CODECS}
    cols = [column(c, t, 1, rng, shared) for t in (3, 130) for c in CODECS]
    few = make_column(synth.ONPAIR16, [b"ab", b"c"], [0, 1] * 4000, [0, 8000])
    cols.append(few)
    few_bad = make_column(synth.ONPAIR12, [b"ab", b"c"], [0, 1] * 4000, [0, 7, 3, 8000][:1] + [8000])
    few_bad.code_offsets = np.array([0, 900, 500, 8000], np.uint32)   # decreasing
    dcs = oracle_decode(few)
    assert dcs.total == 12000
    import torch
    config = fp.batch_config_count() - 1
    good = [DeviceColumn(c) for c in cols]
    bad = DeviceColumn(few_bad)
    refs = [oracle_decode(c) for c in cols]
    outs = [torch.zeros(r.total, dtype=torch.uint8, device="cuda") for r in refs]
    offs = [torch.zeros(c.n_strings + 1, dtype=torch.int32, device="cuda") for c in cols]
    bo, bf = torch.zeros(12000, dtype=torch.uint8, device="cuda"), torch.zeros(4, dtype=torch.int32, device="cuda")
    chunks = [fp.chunk_tensors(c.codec, d.dict, d.codes, d.code_offsets, c.n_strings, o, f)
              for c, d, o, f in zip(cols, good, outs, offs)]
    chunks.insert(3, fp.chunk_tensors(few_bad.codec, bad.dict, bad.codes, bad.code_offsets, 3, bo, bf))
    plan = fp.Plan(chunks, config=config)
    plan.decode()
    st, sts, _ = plan.sync_status()
    assert st == fp.ERR_CORRUPT
    assert sts[3] == fp.ERR_CORRUPT and all(s == fp.OK for k, s in enumerate(sts) if k != 3)
    for k, (r, o) in enumerate(zip(refs, outs)):
        assert np.array_equal(o.cpu().numpy(), r.data), k
