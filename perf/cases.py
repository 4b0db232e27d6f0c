"""Performance cases: decoding dictionary-compressed string columns.

Each case is one call, or one batch or request burst, as a program that holds
compressed columns on the GPU makes it: codes, code offsets and a dictionary
go in, string bytes and string offsets come out.  The sizes are those of the
benchmark workloads and of the committed tuning table (1 k to 16 M strings);
the inputs are seeded synthetic columns with the benchmark's distributions:
token lengths and Zipf exponents per codec, string lengths uniform or
lognormal, escapes in one unit out of a hundred for FSST-8.

A case is a dict of plain values:
  form     "decode"   fp_decode of one column
           "packed"   fp_decode_packed: codes bit-packed at `bits` bits
           "rows"     fp_decode_rows: `rows` random rows of a column
           "sidecar"  fp_decode_sidecar from a stored table
           "batch"    one fp_decode_batch of `chunks` columns, mixed codecs
           "serve"    a burst of `chunks` requests to a server, mixed codecs
  codec    "onpair16", "onpair12", "fsst8" or "fsst12" (single columns)
  strings, codes, spread   number of strings, codes per string, and how that
           number is spread: "uniform" over 1 .. 2 codes - 1, "lognormal" with
           that median (sigma 0.6), "documents" lognormal with sigma 1.0
  low, high   decoded bytes of a chunk, log-uniform (batch, serve)
"""
import math
import random

import numpy as np
import torch

import paper_2609_15034_gb300 as fp

CODECS = {"onpair16": fp.ONPAIR16, "onpair12": fp.ONPAIR12, "fsst8": fp.FSST8, "fsst12": fp.FSST12}
CODE_BITS = {"onpair16": 16, "onpair12": 12, "fsst8": 8, "fsst12": 12}
SIGMA = {"lognormal": 0.6, "documents": 1.0}
ZIPF = {"onpair16": 1.1, "onpair12": 1.2, "fsst8": 1.0, "fsst12": 1.0}
ESCAPES = 0.01   # FSST-8: share of units that are an escape and a literal byte
LITERALS = 0.12  # OnPair-12: share of codes that are one-byte literals (the ends of strings)
# codecs of a batch or burst, chunk by chunk: OnPair-16 twice as often as the others
MIX = ("onpair16", "onpair12", "onpair16", "fsst8", "fsst12")
# decoded bytes a string of a chunk has on average, and its spread
CHUNK_CODES = {"onpair16": 20, "onpair12": 18, "fsst8": 11, "fsst12": 9}
CHUNK_SPREAD = {"onpair16": "uniform", "onpair12": "uniform", "fsst8": "lognormal", "fsst12": "lognormal"}


def listed():
    return [
        # the smallest call: one page of a log column, where launches and latency count
        dict(name="onpair12_1k", form="decode", codec="onpair12", strings=1001, codes=18, spread="uniform"),
        # a row group of identifiers
        dict(name="fsst8_30k", form="decode", codec="fsst8", strings=30011, codes=11, spread="lognormal"),
        # a row group with the large dictionary (1 MiB), the benchmark's small column
        dict(name="onpair16_100k", form="decode", codec="onpair16", strings=100_000, codes=20, spread="uniform"),
        # an ordinary column with the large dictionary
        dict(name="onpair16_2m", form="decode", codec="onpair16", strings=1_999_993, codes=20, spread="uniform"),
        # documents: few strings of kilobytes each, so that many tiles hold no string start
        dict(name="fsst12_docs_20k", form="decode", codec="fsst12", strings=20_011, codes=1200, spread="documents"),
        # the headline column: log lines of 20-200 bytes
        dict(name="onpair12_10m", form="decode", codec="onpair12", strings=10_000_000, codes=18, spread="uniform"),
        # URLs and identifiers with escapes, the most strings of any case
        dict(name="fsst8_16m", form="decode", codec="fsst8", strings=16_000_000, codes=11, spread="lognormal"),
        # a cascaded column: 10-bit codes of a 1,024-symbol table, unpacked by the decode
        dict(name="fsst12_packed10_16m", form="packed", codec="fsst12", strings=16_000_000, codes=9,
             spread="lognormal", bits=10),
        # selective decode: a filter kept one row in ten, in join order
        dict(name="onpair12_rows_1m", form="rows", codec="onpair12", strings=10_000_000, codes=18, spread="uniform",
             rows=1_000_000),
        # a column stored with its table of output positions
        dict(name="onpair12_sidecar_5m", form="sidecar", codec="onpair12", strings=5_000_011, codes=18,
             spread="uniform"),
        # a scan over many column chunks, each with its own dictionary, planned once
        dict(name="batch_256", form="batch", chunks=256, low=4096, high=16 << 20),
        # a burst of page requests to the server
        dict(name="serve_32", form="serve", chunks=32, low=65536, high=16 << 20),
    ]


def draw(rng):
    form = rng.choice(("decode", "decode", "decode", "packed", "rows", "sidecar", "batch", "serve"))

    def log_between(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if form == "batch":
        return dict(form=form, chunks=log_between(8, 256), low=4096, high=log_between(1 << 20, 16 << 20))
    if form == "serve":
        return dict(form=form, chunks=rng.randint(4, 32), low=65536, high=log_between(1 << 20, 16 << 20))
    codecs = ("onpair16", "onpair12", "fsst12") if form == "packed" else tuple(CODECS)
    codec = rng.choice(codecs)
    spread = rng.choice(("uniform", "lognormal", "lognormal", "documents"))
    codes = log_between(300, 3000) if spread == "documents" else log_between(2, 40)
    case = dict(form=form, codec=codec, strings=1, codes=codes, spread=spread)
    strings = log_between(1000, min(16_000_000, int(150e6 / _mean_codes(case))))
    case["strings"] = strings
    if form == "packed":
        case["bits"] = rng.randint(9, CODE_BITS[codec])
    if form == "rows":
        case["rows"] = max(1, strings // log_between(2, 50))
    return case


# ---- dictionaries ------------------------------------------------------------

def _entries(case):
    codec = case["codec"]
    full = {"onpair16": 65536, "onpair12": 4096, "fsst8": 255, "fsst12": 4096}[codec]
    return min(full, 1 << case["bits"]) if "bits" in case else full


def _lengths(codec, entries):
    """Token lengths by popularity rank, the same for every seed, and the
    entries that are one-byte literals at the front of the table."""
    rng = np.random.Generator(np.random.Philox([11, CODECS[codec], entries]))
    if codec == "onpair16":
        lens = rng.geometric(1.0 / 6.0, entries)
        while (lens > 16).any():
            lens[lens > 16] = rng.geometric(1.0 / 6.0, int((lens > 16).sum()))
        return lens, 0
    if codec == "onpair12":
        p = np.array([0, 0, 52, 102, 117, 72, 124, 118, 97, 92, 59, 37, 18, 21, 20, 6, 7], np.float64)
        front = min(256, entries // 2)
        return rng.choice(17, entries - front, p=p / p.sum()), front
    if codec == "fsst8":
        p = np.array([0, 92, 120, 141, 229, 143, 114, 75, 86], np.float64)
        return rng.choice(9, entries, p=p / p.sum()), 0
    p = np.array([0, 62, 91, 172, 182, 123, 121, 124, 125], np.float64)
    return rng.choice(9, entries, p=p / p.sum()), 0


def _weights(codec, n):
    w = np.arange(1, n + 1, dtype=np.float64) ** -ZIPF[codec]
    return w / w.sum()


def _dictionary(case, rng):
    """Token bytes, token offsets and the table code of each popularity rank."""
    codec, entries = case["codec"], _entries(case)
    by_rank, front = _lengths(codec, entries)
    perm = front + rng.permutation(entries - front)
    lens = np.ones(entries, np.int64)
    lens[perm] = by_rank
    offsets = np.zeros(entries + 1, np.uint32)
    offsets[1:] = np.cumsum(lens)
    alphabet = np.frombuffer(b"ABCDEFGHIJKLMNOPQRSTUVWXYZabcdefghijklmnopqrstuvwxyz0123456789-_", np.uint8)
    data = alphabet[rng.integers(0, 64, int(offsets[-1]))]
    data[:front] = np.arange(front)
    return data, offsets, perm


def _mean_bytes(case):
    """Expected decoded bytes of a code (FSST-8: of a unit) and slots of it."""
    codec = case["codec"]
    by_rank, front = _lengths(codec, _entries(case))
    mean = float((_weights(codec, by_rank.size) * by_rank).sum())
    if front:
        mean = LITERALS + (1 - LITERALS) * mean
    if codec == "fsst8":
        return ESCAPES + (1 - ESCAPES) * mean, 1 + ESCAPES
    return mean, 1.0


def _mean_codes(case):
    s = SIGMA.get(case["spread"])
    return case["codes"] * (math.exp(s * s / 2) if s else 1.0)


# ---- columns -------------------------------------------------------------------

def _column(case, seed, part=0):
    """A column: its dictionary, its units (FSST-8: 256 + b is the literal b)
    and the number of units of each string."""
    codec, n = case["codec"], case["strings"]
    rng = np.random.Generator(np.random.Philox([seed, part, CODECS[codec]]))
    data, offsets, perm = _dictionary(case, rng)
    g = torch.Generator(device="cuda")
    g.manual_seed(int(rng.integers(0, 1 << 62)))
    if case["spread"] == "uniform":
        counts = torch.randint(1, 2 * case["codes"], (n,), generator=g, device="cuda")
    else:
        z = torch.randn(n, generator=g, device="cuda", dtype=torch.float32)
        counts = (case["codes"] * torch.exp(SIGMA[case["spread"]] * z)).clamp(0, 30.0 * case["codes"]).round().long()
    total = int(counts.sum())
    cdf = torch.tensor(np.cumsum(_weights(codec, perm.size)), dtype=torch.float32, device="cuda")
    to_code = torch.tensor(perm, dtype=torch.int32, device="cuda")
    front = offsets.size - 1 - perm.size
    parts = []
    for a in range(0, total, 1 << 25):
        m = min(1 << 25, total - a)
        r = torch.searchsorted(cdf, torch.rand(m, generator=g, device="cuda"), out_int32=True, right=True)
        units = to_code[r.clamp_(max=perm.size - 1)]
        if front:
            literal = torch.rand(m, generator=g, device="cuda") < LITERALS
            low, high = (32, 127) if front == 256 else (0, front)
            byte = torch.randint(low, high, (m,), generator=g, device="cuda", dtype=torch.int32)
            units = torch.where(literal, byte, units)
        if codec == "fsst8":
            escape = torch.rand(m, generator=g, device="cuda") < ESCAPES
            byte = torch.randint(256, 512, (m,), generator=g, device="cuda", dtype=torch.int32)
            units = torch.where(escape, byte, units)
        parts.append(units.to(torch.int32))
    units = torch.cat(parts) if parts else torch.zeros(0, dtype=torch.int32, device="cuda")
    return data, offsets, units, counts


def _starts(counts):
    out = torch.zeros(counts.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(counts, 0, out=out[1:])
    return out


def _pack(units, bits):
    """Codes bit-packed LSB-first at `bits` bits per code."""
    n = units.numel()
    out = []
    for a in range(0, n, 1 << 25):
        c = units[a:a + (1 << 25)].to(torch.int64)
        c = torch.nn.functional.pad(c, (0, -c.numel() % 32)).view(-1, 32)
        words = torch.zeros(c.shape[0], bits, dtype=torch.int64, device="cuda")
        for k in range(32):
            w, s = divmod(k * bits, 32)
            words[:, w] |= (c[:, k] << s) & 0xffffffff
            if s + bits > 32:
                words[:, w + 1] |= c[:, k] >> (32 - s)
        out.append(torch.where(words > 0x7fffffff, words - (1 << 32), words).to(torch.int32).view(-1).view(torch.uint8))
    stream = torch.cat(out) if out else torch.zeros(0, dtype=torch.uint8, device="cuda")
    return stream[:(n * bits + 7) // 8].clone()


def _stored(case, units, counts):
    """The stored code buffer and the code offsets of a column."""
    codec = case["codec"]
    starts = _starts(counts)
    if codec == "fsst8":
        width = 1 + (units >= 256).to(torch.int64)
        at = _starts(width)
        stream = torch.full((int(at[-1]),), 255, dtype=torch.uint8, device="cuda")
        stream[at[1:] - 1] = (units & 255).to(torch.uint8)   # the unit's last slot: its code, or its literal
        starts = at[starts]
    elif codec == "onpair16" and "bits" not in case:
        wrapped = torch.where(units > 32767, units - 65536, units)
        stream = wrapped.to(torch.int16).view(torch.uint8)
    else:
        stream = _pack(units, case.get("bits", CODE_BITS[codec]))
    return stream, starts.to(torch.int32)


def _capacity(case):
    """Bytes a program sets aside for the decoded strings: what the column's
    statistics promise and eight standard deviations, whole 256-byte lines.
    The part past the decoded size stays zero."""
    n = case.get("rows", case["strings"])
    s = SIGMA.get(case["spread"])
    string_spread = math.sqrt(math.exp(s * s) - 1) if s else 0.6
    codes = n * _mean_codes(case)
    expected = codes * _mean_bytes(case)[0]
    return int(expected * (1 + 8 * string_spread / math.sqrt(n) + 8 / math.sqrt(codes)) + 4096) // 256 * 256


def _layout(chunks):
    """Where each chunk's strings and string offsets lie in a batch's or
    burst's two result buffers, and the sizes of the two."""
    places, at, at_offsets = [], 0, 0
    for c in chunks:
        places.append((at, at_offsets))
        at += _capacity(c)
        at_offsets += (c["strings"] + 4) // 4 * 4
    return places, at, at_offsets


def _buffers(size, entries):
    return (torch.zeros(size, dtype=torch.uint8, device="cuda"),
            torch.zeros(entries, dtype=torch.int32, device="cuda"))


def _chunks(case):
    """The chunks of a batch or burst as single-column cases (their sizes are
    the case's, their contents the seed's)."""
    rng = random.Random(case["chunks"] * 1000003 + case["high"])
    out = []
    for i in range(case["chunks"]):
        codec = MIX[i % len(MIX)]
        c = dict(codec=codec, codes=CHUNK_CODES[codec], spread=CHUNK_SPREAD[codec], strings=1)
        size = math.exp(rng.uniform(math.log(case["low"]), math.log(case["high"])))
        c["strings"] = max(1, int(size / (_mean_codes(c) * _mean_bytes(c)[0])))
        out.append(c)
    return out


# ---- the measured calls ----------------------------------------------------------

def prepare(case, seed):
    form = case["form"]
    if form in ("batch", "serve"):
        return _prepare_many(case, seed)
    codec = CODECS[case["codec"]]
    data, offsets, units, counts = _column(case, seed)
    codes, starts = _stored(case, units, counts)
    d = fp.Dict(codec, data, offsets)
    n = case["strings"]
    state = dict(form=form, codec=codec, dict=d, codes=codes, starts=starts, strings=n)
    if form == "packed":
        state["bits"] = case["bits"]
    elif form == "rows":
        n = case["rows"]
        state["rows"] = _row_ids(case, seed)
        _, state["slots"], _ = fp.rows_size(codec, d, codes.data_ptr(), codes.numel(), starts.data_ptr(),
                                            case["strings"], state["rows"].data_ptr(), n)
    elif form == "sidecar":
        state["column"] = fp.SidecarColumn(codec, d, codes, starts, n)
        state["column"].build()
    state["out"], state["out_offsets"] = _buffers(_capacity(case), n + 1)
    return state


def _prepare_many(case, seed):
    form, chunks = case["form"], _chunks(case)
    places, size, entries = _layout(chunks)
    out, out_offsets = _buffers(size, entries)
    server = fp.Server(hbm_budget=2 << 30, dict_cache_slots=64) if form == "serve" else None
    keep, calls = [], []
    for i, (c, (at, at_offsets)) in enumerate(zip(chunks, places)):
        codec, n = CODECS[c["codec"]], c["strings"]
        data, offsets, units, counts = _column(c, seed, i)
        codes, starts = _stored(c, units, counts)
        d = fp.Dict(codec, data, offsets)
        mine, my_offsets = out[at:at + _capacity(c)], out_offsets[at_offsets:at_offsets + n + 1]
        if form == "serve":
            server.dict_put(i, codec, data, offsets)
            _, total = fp.decoded_size_tensors(codec, d, codes, starts, n)   # a request carries its decoded size
            calls.append((codes, starts, n, total, mine, my_offsets))
        else:
            calls.append(fp.chunk_tensors(codec, d, codes, starts, n, mine, my_offsets))
            keep.append((d, codes, starts))
    torch.cuda.synchronize()   # the server's streams, or the plan's tuning, read these buffers
    state = dict(form=form, outs=[out, out_offsets])
    if form == "serve":
        state["server"], state["requests"] = server, calls
    else:
        state["keep"], state["plan"] = keep, fp.Plan(calls)
    return state


def _row_ids(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 13)
    return torch.randperm(case["strings"], generator=g, device="cuda")[:case["rows"]].to(torch.int32)


def run(state):
    form, stream = state["form"], torch.cuda.current_stream()
    if form == "serve":
        server, requests = state["server"], state["requests"]
        for i, (codes, starts, strings, total, _, _) in enumerate(requests):
            server.submit(i, codes.data_ptr(), codes.numel(), starts.data_ptr(), strings, total, user_tag=i)
        done = []
        while len(done) < len(requests):
            done += server.poll(timeout_s=1.0)
        for r in done:
            _, _, strings, total, out, out_offsets = requests[r["user_tag"]]
            out[:total].copy_(fp.device_bytes(r["d_out_bytes"], total))
            out_offsets.view(torch.uint8).copy_(fp.device_bytes(r["d_out_offsets"], 4 * (strings + 1)))
        stream.synchronize()   # the results are copied out before the server may reuse them
        for r in done:
            server.release(r["ticket"])
        return state["outs"]
    if form == "batch":
        state["plan"].decode(stream)
        return state["outs"]
    codec, d, codes, starts, n = state["codec"], state["dict"], state["codes"], state["starts"], state["strings"]
    out, out_offsets = state["out"], state["out_offsets"]
    if form == "sidecar":
        state["column"].decode(out, out_offsets, stream)
    elif form == "packed":
        fp.decode_packed(codec, d, state["bits"], codes.data_ptr(), codes.numel(), starts.data_ptr(), n,
                         out.data_ptr(), out.numel(), out_offsets.data_ptr(), stream)
    elif form == "rows":
        fp.decode_rows(codec, d, codes.data_ptr(), codes.numel(), starts.data_ptr(), n, state["rows"].data_ptr(),
                       state["rows"].numel(), state["slots"], out.data_ptr(), out.numel(), out_offsets.data_ptr(),
                       stream)
    else:
        fp.decode_tensors(codec, d, codes, starts, n, out, out_offsets, stream)
    return [out, out_offsets]


# ---- what a pass cannot do without, and what it returns -----------------------------

def work(case):
    """Bytes: the codes and code offsets read, the string bytes and offsets
    written, the dictionary read, the row ids or the stored table read."""
    if case["form"] in ("batch", "serve"):
        total = sum(work(dict(c, form="decode"))["bytes"] for c in _chunks(case))
        if case["form"] == "serve":   # results are copied out: the string bytes and offsets read and written once more
            for c in _chunks(case):
                total += 2 * (c["strings"] * _mean_codes(c) * _mean_bytes(c)[0] + 4 * c["strings"])
        return dict(bytes=float(total), flops=0.0)
    codec, n = case["codec"], case.get("rows", case["strings"])
    mean, slots = _mean_bytes(case)
    codes = n * _mean_codes(case)
    stored = codes * slots * case.get("bits", CODE_BITS[codec]) / 8
    by_rank, front = _lengths(codec, _entries(case))
    total = stored + codes * mean + 8 * n + float(by_rank.sum() + front)
    if case["form"] == "rows":
        total += 8 * n   # the row ids, and each selected row's second offset
    if case["form"] == "sidecar":
        total += 8 * codes * slots / fp.sidecar_tile_slots(CODECS[codec])
    return dict(bytes=float(total), flops=0.0)


def exact(case, seed):
    """The string bytes and offsets by table look-up and prefix sums."""
    if case["form"] in ("batch", "serve"):
        chunks = _chunks(case)
        places, size, entries = _layout(chunks)
        out, out_offsets = _buffers(size, entries)
        for i, (c, (at, at_offsets)) in enumerate(zip(chunks, places)):
            strings, offsets = _expand(*_column(c, seed, i))
            out[at:at + strings.numel()] = strings
            out_offsets[at_offsets:at_offsets + offsets.numel()] = offsets
        return [out, out_offsets]
    strings, offsets = _expand(*_column(case, seed), rows=_row_ids(case, seed).long() if case["form"] == "rows" else None)
    out, _ = _buffers(_capacity(case), 1)
    out[:strings.numel()] = strings
    return [out, offsets]


def _expand(data, offsets, units, counts, rows=None):
    if rows is not None:
        first, counts = _starts(counts)[rows], counts[rows]
        at = torch.repeat_interleave(first - _starts(counts)[:-1], counts)
        units = units[at + torch.arange(at.numel(), device="cuda")]
    lens = torch.ones(512 if offsets.size <= 256 else offsets.size - 1, dtype=torch.int64)
    lens[:offsets.size - 1] = torch.from_numpy(np.diff(offsets.astype(np.int64)))
    table = torch.zeros(lens.numel(), 16, dtype=torch.uint8)
    flat = torch.arange(16)[None, :] < lens[:offsets.size - 1, None]
    table[:offsets.size - 1][flat] = torch.from_numpy(data)
    if offsets.size <= 256:
        table[256:, 0] = torch.arange(256, dtype=torch.uint8)
    lens, table = lens.cuda(), table.cuda()
    total = int(units.numel())
    out, sums = [], torch.zeros(total + 1, dtype=torch.int64, device="cuda")
    for a in range(0, total, 1 << 24):
        u = units[a:a + (1 << 24)].long()
        out.append(table[u][torch.arange(16, device="cuda")[None, :] < lens[u][:, None]])
        sums[a + 1:a + 1 + u.numel()] = lens[u]
    sums.cumsum_(0)
    bytes_ = torch.cat(out) if out else torch.zeros(0, dtype=torch.uint8, device="cuda")
    return [bytes_, sums[_starts(counts)].to(torch.int32)]
