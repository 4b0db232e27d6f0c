"""A kernel launch that the runtime refuses in the middle of a call: the call
reports it, and the calls after it are exact.  A child process runs with a shim
in front of the runtime's cudaLaunchKernelExC that answers the n-th launch with
an error code instead of making it; nothing goes wrong on the GPU."""
import os
import subprocess
import sys

import pytest

from gpu_util import __file__ as GPU_UTIL

pytestmark = pytest.mark.gpu

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
static int left;
void shim_refuse(int n) { __atomic_store_n(&left, n, __ATOMIC_SEQ_CST); }
int cudaLaunchKernelExC(const void* config, const void* func, void** args) {
    static int (*real)(const void*, const void*, void**);
    if (!real) {
        void* rt = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
        *(void**)&real = dlsym(rt ? rt : RTLD_DEFAULT, "cudaLaunchKernelExC");
    }
    if (__atomic_load_n(&left, __ATOMIC_SEQ_CST) > 0 && __atomic_sub_fetch(&left, 1, __ATOMIC_SEQ_CST) == 0)
        return 701;   /* cudaErrorLaunchOutOfResources */
    return real(config, func, args);
}
"""

COLUMN = r"""
import ctypes, sys
import numpy as np
import synth
from gpu_util import DeviceColumn, assert_same, oracle_decode
import paper_2609_15034_gb300 as fp

refuse = ctypes.CDLL(None).shim_refuse
codec, k = int(sys.argv[1]), int(sys.argv[2])
cols = [synth.column(codec, s, n) for s, n in ((1, 60000), (2, 50000), (3, 9000))]
dcs = [DeviceColumn(c) for c in cols]
assert fp.variant_info(codec, fp.variant_for_dict(dcs[0].dict, dcs[0].codes_bytes))["launches_per_call"] == 3
caps = [oracle_decode(c).total for c in cols]
block = [v for v in range(fp.variant_count(codec)) if fp.variant_info(codec, v)["launches_per_call"] == 2]
for first in range(3):
    assert_same(cols[0], dcs[0])
    refuse(k)
    st, _, _, guard_ok, launch = dcs[0].decode(capacity=caps[0])
    assert launch == fp.ERR_CUDA and guard_ok, launch
    if first == 2 and block:   # the block pipeline's tickets are the same words
        fp.variant_select(codec, block[0])
        assert_same(cols[1], dcs[1], capacity=caps[1])
        fp.variant_select(codec, -1)
    for j in (1, 2, 0)[first:]:
        assert_same(cols[j], dcs[j], capacity=caps[j])
print("passed")
"""

SERVED = r"""
import ctypes, sys
import numpy as np
import synth
from test_gpu_serve import Page, collect, fetch, register
import paper_2609_15034_gb300 as fp

refuse = ctypes.CDLL(None).shim_refuse
k = int(sys.argv[1])
codecs = (synth.ONPAIR16, synth.ONPAIR12, synth.FSST8, synth.FSST12)
pages = [Page(synth.column(c, 800 + 10 * c + s, n), key=10 * c + s) for c in codecs for s, n in ((1, 9000), (2, 7000))]
srv = fp.Server(hbm_budget=256 << 20, n_streams=1, max_wave=1, batch_config=5)   # the staged launches
register(srv, pages)


def one(p):
    p.submit(srv, tag=0)
    (t, r), = collect(fp, srv, 1).items()
    if r["status"] == fp.OK:
        data, offs = fetch(fp, r)
        assert np.array_equal(data, p.ref.data)
        np.testing.assert_array_equal(offs, p.ref.offsets)
    srv.release(t)
    return r["status"]


for a, b in zip(pages[::2], pages[1::2]):
    assert one(a) == fp.OK
    refuse(k)
    assert one(b) == fp.ERR_CUDA
    for p in (a, b, a):
        assert one(p) == fp.OK
srv.destroy()
print("passed")
"""


def run(tmp_path, script, *args):
    c, so = tmp_path / "shim.c", tmp_path / "shim.so"
    c.write_text(SHIM)
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-O1", str(c), "-o", str(so), "-ldl"])
    tests = os.path.dirname(os.path.abspath(GPU_UTIL))
    env = dict(os.environ, LD_PRELOAD=str(so), PYTHONPATH=os.pathsep.join([os.path.dirname(tests), tests]))
    r = subprocess.run([sys.executable, "-c", script, *map(str, args)], env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "passed" in r.stdout, r.stdout + r.stderr


@pytest.fixture(autouse=True)
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("codec", [1, 2, 3, 4])
@pytest.mark.parametrize("launch", [1, 2, 3])
def test_decode_launch_refused(tmp_path, codec, launch):
    run(tmp_path, COLUMN, codec, launch)


# of a wave of one chunk: reduce, index pass, decode (the scan is launched another way)
@pytest.mark.parametrize("launch", [1, 2, 3])
def test_wave_launch_refused(tmp_path, launch):
    run(tmp_path, SERVED, launch)
