"""A call's first launch may start before the work ahead of it on the stream
has ended, and its later launches before the first has: columns that a kernel
writes just before the call, with older columns' lines in the caches -- packed
codes, selected rows (whose codes and offsets the call itself makes), an event
of another stream waited for, the legacy default stream behind a blocking one.
Every result is compared on the stream.  Decoding is exact: no tolerance."""
import ctypes

import numpy as np
import pytest

import oracle
import synth
from gpu_util import make_column, oracle_decode
from test_gpu_packed import pack_bits

pytestmark = pytest.mark.gpu

CODECS = [synth.ONPAIR16, synth.ONPAIR12, synth.FSST8, synth.FSST12]
SIZES = [300, 30_000]   # one cluster, three launches


@pytest.fixture(scope="module")
def fp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15034_gb300 as m
    return m


@pytest.fixture(scope="module")
def streams(fp):
    """Two streams for the whole file (torch hands out 32 and then the first again)."""
    import torch
    return torch.cuda.Stream(), torch.cuda.Stream()


def device(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def columns(codec, n):
    """Two columns of n strings and as many codes, with one dictionary."""
    rng = np.random.default_rng(n + codec)
    toks = [rng.integers(0, 256, 1 + k % synth.MAX_TOKEN[codec], dtype=np.uint8).tobytes() for k in range(200)]
    total = 14 * n
    return [make_column(codec, toks, rng.integers(0, len(toks), total),
                        np.sort(np.concatenate([[0, total], rng.integers(0, total + 1, n - 1)]))) for _ in range(2)]


class Pair:
    """Two inputs of one call, copied in turn into the buffers that it reads."""

    def __init__(self, fp, cols, streams, refs, ids=None):
        import torch
        d = cols[0].dictionary
        self.dic = fp.Dict(cols[0].codec, d.data, d.offsets)
        self.src = [[device(s), device(c.code_offsets.view(np.int32))] for s, c in zip(streams, cols)]
        if ids is not None:
            for s, i in zip(self.src, ids):
                s.append(device(i.view(np.int32)))
        self.want = [(device(r.data), device(r.offsets.view(np.int32))) for r in refs]
        self.buf = [torch.empty_like(b) for b in self.src[0]]
        self.out = torch.zeros(max(r.total for r in refs), dtype=torch.uint8, device="cuda")
        self.offs = torch.zeros(refs[0].offsets.size, dtype=torch.int32, device="cuda")
        self.bad = torch.zeros(1, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()

    def produce(self, k):
        import torch
        for b, s in zip(self.buf, self.src[k & 1]):
            torch.add(s, 0, out=b)   # kernels, the last of them right before the call

    def compare(self, k):
        data, offs = self.want[k & 1]
        self.bad += (self.out[:data.numel()] != data).sum() + (self.offs != offs).sum()


@pytest.mark.parametrize("codec", CODECS)
@pytest.mark.parametrize("n", SIZES)
def test_rows_right_after_their_producer(fp, streams, codec, n):
    import torch
    cols = columns(codec, n)
    ids = [np.random.default_rng(s).integers(0, n, n // 2).astype(np.uint32) for s in (1, 2)]
    refs = [oracle.decode_rows(codec, c.dictionary.data, c.dictionary.offsets, c.stream, c.code_offsets, i)
            for c, i in zip(cols, ids)]
    x = Pair(fp, cols, [c.stream for c in cols], refs, ids)
    slots = max(int((c.code_offsets[i + 1] - c.code_offsets[i]).sum()) for c, i in zip(cols, ids))
    s = streams[0]
    with torch.cuda.stream(s):
        for k in range(60):
            x.produce(k)
            codes, co, rows = x.buf
            fp.decode_rows(codec, x.dic, codes.data_ptr(), codes.numel(), co.data_ptr(), n, rows.data_ptr(), n // 2,
                           slots, x.out.data_ptr(), x.out.numel(), x.offs.data_ptr(), s)
            x.compare(k)
    assert fp.sync_status(s) == fp.OK, fp.last_error()
    assert int(x.bad.item()) == 0


@pytest.mark.parametrize("codec,bits", [(synth.ONPAIR16, 13), (synth.ONPAIR12, 11), (synth.FSST12, 10),
                                        (synth.FSST12, 9)])
@pytest.mark.parametrize("n", SIZES)
def test_packed_right_after_its_producer(fp, streams, codec, bits, n):
    import torch
    cols = columns(codec, n)
    rng = np.random.default_rng(bits)
    codes_of = [rng.integers(0, 200, c.n_slots).astype(np.uint32) for c in cols]
    packed = [pack_bits(c, bits) for c in codes_of]
    refs = [oracle.decode_packed(codec, bits, c.dictionary.data, c.dictionary.offsets, st, c.code_offsets)
            for c, st in zip(cols, packed)]
    x = Pair(fp, cols, packed, refs)
    s = streams[0]
    with torch.cuda.stream(s):
        for k in range(60):
            x.produce(k)
            codes, co = x.buf
            fp.decode_packed(codec, x.dic, bits, codes.data_ptr(), codes.numel(), co.data_ptr(), n, x.out.data_ptr(),
                             x.out.numel(), x.offs.data_ptr(), s)
            x.compare(k)
    assert fp.sync_status(s) == fp.OK, fp.last_error()
    assert int(x.bad.item()) == 0


def call(fp, x, codec, n, stream):
    codes, co = x.buf
    fp.decode(codec, x.dic, codes.data_ptr(), codes.numel(), co.data_ptr(), n, x.out.data_ptr(), x.out.numel(),
              x.offs.data_ptr(), stream)


@pytest.mark.parametrize("codec", CODECS)
@pytest.mark.parametrize("n", SIZES)
def test_decode_behind_an_event(fp, streams, codec, n):
    """The column is written on another stream, whose event the call's stream
    waits for, with the call before it still on the stream."""
    import torch
    cols = columns(codec, n)
    x = Pair(fp, cols, [c.stream for c in cols], [oracle_decode(c) for c in cols])
    a, b = streams
    for k in range(30):
        a.wait_stream(b)
        with torch.cuda.stream(a):
            torch.cuda._sleep(200_000)   # the event is far from recorded when the call is made
            x.produce(k)
        b.wait_stream(a)
        with torch.cuda.stream(b):
            call(fp, x, codec, n, b)
            x.compare(k)
    assert fp.sync_status(b) == fp.OK, fp.last_error()
    assert int(x.bad.item()) == 0


@pytest.mark.parametrize("codec", CODECS)
@pytest.mark.parametrize("n", SIZES)
def test_legacy_stream_behind_a_blocking_one(fp, codec, n):
    import torch
    cols = columns(codec, n)
    x = Pair(fp, cols, [c.stream for c in cols], [oracle_decode(c) for c in cols])
    cudart = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    handle = ctypes.c_void_p()
    assert cudart.cudaStreamCreate(ctypes.byref(handle)) == 0   # a blocking stream
    try:
        p = torch.cuda.ExternalStream(handle.value)
        for k in range(30):
            with torch.cuda.stream(p):
                torch.cuda._sleep(200_000)
                x.produce(k)
            call(fp, x, codec, n, None)   # the legacy stream waits for p by itself
            x.compare(k)
        assert fp.sync_status() == fp.OK, fp.last_error()
        assert int(x.bad.item()) == 0
    finally:
        torch.cuda.synchronize()
        assert cudart.cudaStreamDestroy(handle) == 0
