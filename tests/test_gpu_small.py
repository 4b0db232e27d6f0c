"""GPU parity where the launches of a call overlap with what comes before
them: a producer kernel right before the decode; stream capture.  Decoding is
exact: no tolerance."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import DeviceColumn, oracle_decode

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
