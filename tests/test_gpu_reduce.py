"""GPU parity of the passes before the decode: the reduce of large columns
(lengths in a gather table, FSST-8's literals and entry states), and the index
pass over offsets that are unaligned, dense, sparse or corrupt.  Decoding is
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


@pytest.mark.parametrize("n_slots,first", [(4 << 20, 0), ((4 << 20) + 513, 700), (5_000_011, 1)])
def test_large_onpair16(fp, n_slots, first):
    rng = np.random.default_rng(n_slots)
    toks = [rng.integers(0, 256, 1 + k % 16, dtype=np.uint8).tobytes() for k in range(65536)]
    slots = rng.integers(0, 65536, n_slots)
    offs = np.sort(np.concatenate([[first, n_slots], rng.integers(first, n_slots + 1, n_slots // 9)]))
    check(fp, make_column(synth.ONPAIR16, toks, slots, offs))


@pytest.mark.parametrize("bad", [0, 511, 512, 2_000_003, (4 << 20) - 1])
def test_large_onpair16_code_without_a_token(fp, bad):
    slots = np.random.default_rng(bad).integers(0, 1000, 4 << 20)
    slots[bad] = 1000
    col = make_column(synth.ONPAIR16, [b"ab"] * 500 + [b"x" * 16] * 500, slots, [0, 100, 4 << 20])
    dc = DeviceColumn(col)
    st, _, _, guard_ok, _ = dc.decode(capacity=64 << 20)
    assert st == fp.ERR_CORRUPT and guard_ok


@pytest.mark.parametrize("n_slots", [40 << 20, (40 << 20) + 1025])
def test_large_fsst8(fp, n_slots):
    rng = np.random.default_rng(n_slots)
    slots = rng.integers(0, 255, n_slots).astype(np.uint8)
    slots[rng.integers(0, n_slots, n_slots // 60)] = 255
    # runs of 0xFF of every parity, over lane and tile edges and whole tiles
    for k, run in enumerate([1, 2, 31, 32, 33, 1023, 1024, 1025, 2048, 3071, 5000]):
        for at in (1024 * (50 + 20 * k) - k, 1024 * (1000 + 20 * k) + 32 * k, 1024 * (9000 + 20 * k) - 1):
            slots[at:at + run] = 255
    slots[-2:] = 7
    # strings begin on codes: walk the escapes once
    lit = np.zeros(n_slots + 1, bool)
    is_ff = np.concatenate([slots == 255, [False]])
    starts = np.flatnonzero(is_ff & ~np.concatenate([[False], is_ff[:-1]]))
    ends = np.flatnonzero(~is_ff & np.concatenate([[False], is_ff[:-1]]))
    for s, e in zip(starts, ends):
        lit[s + 1:e + 1:2] = True
    toks = [bytes([k]) * (1 + k % 8) for k in range(255)]
    cuts = np.sort(rng.integers(1, n_slots, n_slots // 13))
    offs = np.concatenate([[0], cuts[~lit[cuts]], [n_slots]])
    check(fp, make_column(synth.FSST8, toks, slots, offs))


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
