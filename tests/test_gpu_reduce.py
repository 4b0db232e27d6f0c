"""GPU parity of the pass before the decode: the index pass over offsets that are unaligned, dense, sparse or corrupt.  Decoding is
exact: no tolerance."""
import numpy as np
import pytest

import synth
from gpu_util import DeviceColumn, make_column, oracle_decode

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15034_gb300 as m
    yield m


def check(fp, col, dc=None, code_offsets=None):
    dc = dc or DeviceColumn(col)
    ref = oracle_decode(col, threads=8)
    st, data, offs, guard_ok, _ = dc.decode(capacity=ref.total, code_offsets=code_offsets)
    assert st == fp.OK, fp.last_error()
    assert guard_ok
    np.testing.assert_array_equal(offs, ref.offsets)
    assert np.array_equal(data, ref.data)


@pytest.mark.parametrize("codec", [synth.ONPAIR16, synth.ONPAIR12, synth.FSST8, synth.FSST12])
@pytest.mark.parametrize("kind", ["unaligned", "dense", "sparse", "empty_ends"])
def test_index_pass(fp, codec, kind):
    import torch
    rng = np.random.default_rng(codec)
    n_slots = 300_001
    toks = [b"a", b"bcd", b"efghijkl"]
    slots = rng.integers(0, 3, n_slots)
    inner = {"unaligned": rng.integers(0, n_slots + 1, 20_000), "dense": np.repeat(np.arange(n_slots), 2),
             "sparse": np.array([299_000]),
             "empty_ends": np.concatenate([np.zeros(3000, int), np.full(3000, n_slots), np.arange(0, n_slots, 512)])}[kind]
    col = make_column(codec, toks, slots, np.sort(np.concatenate([[0, n_slots], inner])))
    dc = DeviceColumn(col)
    co = None
    if kind == "unaligned":
        buf = torch.zeros(dc.n_strings + 2, dtype=torch.int32, device="cuda")
        co = buf[1:]
        co.copy_(dc.code_offsets)
    check(fp, col, dc, co)


@pytest.mark.parametrize("at", [1, 255, 256, 4_000, 9_999])
def test_decreasing_offsets_are_corrupt(fp, at):
    offs = np.arange(0, 300_001, 30)
    offs[at] = offs[at - 1] - 1 if at > 1 else 299_999
    col = make_column(synth.FSST12, [b"xy", b"z"], np.zeros(300_001, int), offs)
    dc = DeviceColumn(col)
    st, _, _, guard_ok, _ = dc.decode(capacity=1 << 20)
    assert st == fp.ERR_CORRUPT and guard_ok
