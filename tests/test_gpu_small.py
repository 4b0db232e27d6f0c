"""GPU parity of the one-cluster decode of small columns, and of the launches
that overlap: sizes around the line between one cluster and three launches,
tile and block edges, escape runs that cross lanes, warps and blocks, slices,
errors; a producer kernel right before the decode; stream capture.  Decoding
is exact: no tolerance."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import DeviceColumn, assert_same, make_column, oracle_decode

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


def cluster_variant(fp, codec):
    one = [v for v in range(fp.variant_count(codec)) if fp.variant_info(codec, v)["launches_per_call"] == 1]
    return one[-1]   # the cooperative launches come first


@pytest.mark.parametrize("codec", CODECS)
@pytest.mark.parametrize("n_slots", [0, 1, 255, 256, 257, 8191, 8193, 65537, 131071, 131072, 200001])
def test_cluster_sizes(fp, codec, n_slots):
    rng = np.random.default_rng(n_slots + codec)
    toks = [rng.integers(0, 256, 1 + k % synth.MAX_TOKEN[codec], dtype=np.uint8).tobytes() for k in range(200)]
    slots = rng.integers(0, len(toks), n_slots)
    fp.variant_select(codec, cluster_variant(fp, codec))
    try:
        for first in (0, min(n_slots, 777)):
            offs = np.sort(np.concatenate([[first, n_slots], rng.integers(first, n_slots + 1, n_slots // 7)]))
            assert_same(make_column(codec, toks, slots, offs))
    finally:
        fp.variant_select(codec, -1)


@pytest.mark.parametrize("run", [512, 8193, 40000, 40001])
def test_cluster_escape_runs(fp, run):
    """0xFF slots over whole lanes, warps and blocks: the entering state of
    every later slot comes from before the run."""
    rng = np.random.default_rng(run)
    slots = np.concatenate([rng.integers(0, 255, 301), np.full(run, 255), rng.integers(0, 255, 20000), [7]])
    col = make_column(synth.FSST8, [bytes([k]) * (1 + k % 8) for k in range(255)], slots, [0, len(slots)])
    fp.variant_select(synth.FSST8, cluster_variant(fp, synth.FSST8))
    try:
        assert_same(col)
    finally:
        fp.variant_select(synth.FSST8, -1)


@pytest.mark.parametrize("codec", CODECS)
def test_cluster_errors(fp, codec):
    col = synth.column(codec, 5, 900)
    dc = DeviceColumn(col)
    ref = oracle_decode(col)
    fp.variant_select(codec, cluster_variant(fp, codec))
    try:
        st, _, _, guard_ok, _ = dc.decode(capacity=ref.total - 1)
        assert st == fp.ERR_CAPACITY and guard_ok
        few = make_column(codec, [b"ab", b"c"], [0, 1, 0, 2, 1], [0, 2, 5])
        st, _, _, guard_ok, _ = DeviceColumn(few).decode(capacity=64)
        assert st == fp.ERR_CORRUPT and guard_ok
        # the stall hook: nothing waits here, the call reports it and the next one is normal
        assert fp.debug_stall_next(64) == fp.OK
        st, _, _, guard_ok, _ = dc.decode(capacity=ref.total)
        assert st == fp.ERR_TIMEOUT and guard_ok
        assert_same(col, dc)
    finally:
        fp.variant_select(codec, -1)


@pytest.mark.parametrize("codec", CODECS)
@pytest.mark.parametrize("n", [300, 30_000])
def test_decode_right_after_its_producer(fp, codec, n):
    """The column is written by a kernel just before the decode (whose first
    launch may start early) and the output read by one just after it."""
    import torch
    cols = [synth.column(codec, s, n) for s in (1, 2)]
    d = cols[0].dictionary
    dic = fp.Dict(codec, d.data, d.offsets)
    size = max(c.stream.size for c in cols)
    top = max(c.n_slots for c in cols)
    src, want = [], []
    for c in cols:
        col = synth.Column(codec, d, c.stream, c.code_offsets, c.n_slots)
        ref = oracle_decode(col)
        pad = np.zeros(size, np.uint8)
        pad[:c.stream.size] = c.stream
        src.append((torch.from_numpy(pad).cuda(), torch.from_numpy(c.code_offsets.view(np.int32)).cuda()))
        want.append((torch.from_numpy(ref.data).cuda(), torch.from_numpy(ref.offsets.view(np.int32)).cuda()))
    assert top
    codes, co = torch.empty_like(src[0][0]), torch.empty_like(src[0][1])
    out = torch.zeros(max(w[0].numel() for w in want), dtype=torch.uint8, device="cuda")
    offs = torch.empty(n + 1, dtype=torch.int32, device="cuda")
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        for k in range(60):
            codes.copy_(src[k & 1][0])
            torch.add(src[k & 1][1], 0, out=co)   # a kernel writes the offsets last
            fp.decode(codec, dic, codes.data_ptr(), size, co.data_ptr(), n, out.data_ptr(), out.numel(),
                      offs.data_ptr(), s)
            w = want[k & 1]
            bad += (out[:w[0].numel()] != w[0]).sum() + (offs != w[1]).sum()
    assert fp.sync_status(s) == fp.OK
    assert int(bad.item()) == 0


@pytest.mark.parametrize("codec,n", [(synth.ONPAIR12, 400), (synth.ONPAIR16, 40_000), (synth.FSST8, 700)])
def test_capture(fp, codec, n):
    """Captured as a graph's first node, after a copy, and after a join of two streams."""
    import torch
    col = synth.column(codec, 3, n)
    dc = DeviceColumn(col)
    ref = oracle_decode(col)
    out = torch.zeros(ref.total, dtype=torch.uint8, device="cuda")
    offs = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    codes = torch.zeros_like(dc.codes)
    s, side = torch.cuda.Stream(), torch.cuda.Stream()

    def call(buf):
        fp.decode(codec, dc.dict, buf.data_ptr(), dc.codes_bytes, dc.code_offsets.data_ptr(), n, out.data_ptr(),
                  out.numel(), offs.data_ptr(), s)

    call(dc.codes)   # the stream's workspace exists before the capture
    torch.cuda.synchronize()
    for how in ("first", "copy", "join"):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(s), torch.cuda.graph(g, stream=s):
            if how == "join":
                side.wait_stream(s)
                with torch.cuda.stream(side):
                    codes.copy_(dc.codes)
                s.wait_stream(side)
            elif how == "copy":
                codes.copy_(dc.codes)
            call(dc.codes if how == "first" else codes)
        for _ in range(3):
            out.zero_()
            offs.zero_()
            codes.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert fp.sync_status(s) == fp.OK, how
            np.testing.assert_array_equal(out.cpu().numpy(), ref.data, err_msg=how)
            np.testing.assert_array_equal(offs.cpu().numpy().view(np.uint32), ref.offsets, err_msg=how)
    assert ref.status == oracle.OK
