"""Which launches a server's wave takes: below 192 MiB of output capacity the
four of the warp-tile batch, from there on the staged ones, counted in the
server's statistics; an explicit configuration is taken for every wave.  One
request a wave, so the sizes are exact; every result equals the oracle's."""
import numpy as np
import pytest

import synth
from test_gpu_serve import Page, collect, fetch, fp, register  # noqa: F401  (fp: the module's fixture)

pytestmark = pytest.mark.gpu

LINE = 192 << 20


@pytest.mark.parametrize("config", [-1, 4, 5])
def test_staged_waves_are_counted(fp, config):  # noqa: F811
    codecs = [synth.ONPAIR16, synth.ONPAIR12, synth.FSST8, synth.FSST12]
    pages = [Page(synth.column(c, 4200 + c, 20000), key=c) for c in codecs]
    srv = fp.Server(hbm_budget=1 << 30, n_streams=1, max_wave=1, batch_config=config)
    register(srv, pages)
    staged = 0
    for capacity in (0, LINE, LINE - 1, LINE + 1, 0):
        for p in pages:
            p.submit(srv, tag=0, decoded_size=max(capacity, p.ref.total))
            (t, r), = collect(fp, srv, 1).items()
            assert r["status"] == fp.OK and r["bytes"] == p.ref.total
            data, offs = fetch(fp, r)
            assert np.array_equal(data, p.ref.data)
            np.testing.assert_array_equal(offs, p.ref.offsets)
            srv.release(t)
            staged += config == 5 or (config < 0 and capacity >= LINE)
            assert srv.stats()["staged_waves"] == staged
    srv.destroy()
