"""A server's waves on both sides of the size at which the staged launches are
taken: small and large ones in turn, on the same lanes, exact each time."""
import numpy as np
import pytest

import synth
from test_gpu_serve import Page, collect, fetch, fp, register  # noqa: F401  (fp: the module's fixture)

pytestmark = pytest.mark.gpu


def test_small_and_large_waves_in_turn(fp):  # noqa: F811
    codecs = [synth.ONPAIR16, synth.ONPAIR12, synth.FSST8, synth.FSST12]
    pages = [Page(synth.column(c, 4100 + i, 60000), key=i) for i, c in enumerate(codecs)]
    srv = fp.Server(hbm_budget=2 << 30, n_streams=2)
    register(srv, pages)
    total = sum(p.ref.total for p in pages)
    large = 4 * ((400 << 20) // total + 1)     # requests of about 400 MB
    for count in (2, large, 3, large):
        sent = {}
        for i in range(count):
            p = pages[i % 4]
            sent[p.submit(srv, tag=i)] = p
        got = collect(fp, srv, count)
        checked = set()
        for t, r in got.items():
            p = sent[t]
            assert r["status"] == fp.OK and r["bytes"] == p.ref.total
            if count < 10 or p.key not in checked or r["user_tag"] >= count - 8:
                checked.add(p.key)
                data, offs = fetch(fp, r)
                assert np.array_equal(data, p.ref.data)
                np.testing.assert_array_equal(offs, p.ref.offsets)
        for t in got:
            srv.release(t)
    srv.destroy()
