"""Failure detection without a fault: the waits for the decode's bulk copies
really run out.  The stored-sidecar calls are built once more with barriers
that wait for one arrival more than is ever made, and a limit of 20 ms: every
wait for the staged tables (OnPair, FSST-12) and for a tile's codes (FSST-8)
gives up.  The call decodes by ordinary loads, so its result equals the
oracle's, and its status word reports the time-out."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
import synth
from gpu_util import DeviceColumn, oracle_decode

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stalled(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15034_gb300 as fp
    from paper_2609_15034_gb300 import _build
    lib = fp.lib()
    out = str(tmp_path_factory.mktemp("stalled") / "libstalled.so")
    subprocess.check_call([_build.nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-DFP_COPY_ARRIVALS=2u",
                           "-DFP_WAIT_LIMIT_NS=20000000ull", "-shared", "--cudart", "shared",
                           os.path.join(_build.CSRC, "fp_sidecar.cu"), _build.LIB, "-o", out])
    s = ctypes.CDLL(out)
    s.fp_decode_sidecar.argtypes = lib.fp_decode_sidecar.argtypes
    return s


@pytest.mark.parametrize("codec", [synth.ONPAIR16, synth.ONPAIR12, synth.FSST8, synth.FSST12])
def test_copy_waits_give_up(stalled, codec):
    import torch
    import paper_2609_15034_gb300 as fp
    col = synth.column(codec, 70 + codec, 20_000)
    ref = oracle_decode(col)
    dc = DeviceColumn(col)
    sc = fp.SidecarColumn(codec, dc.dict, dc.codes, dc.code_offsets, dc.n_strings, dc.codes_bytes)
    sc.build()
    assert sc.status_bits() == 0
    out = torch.zeros(ref.total, dtype=torch.uint8, device="cuda")
    offs = torch.zeros(col.n_strings + 1, dtype=torch.int32, device="cuda")
    st = stalled.fp_decode_sidecar(codec, dc.dict.handle, dc.codes.data_ptr(), dc.codes_bytes,
                                   dc.code_offsets.data_ptr(), dc.n_strings, sc.sidecar.data_ptr(), sc.entries,
                                   out.data_ptr(), out.numel(), offs.data_ptr(), sc.scratch.data_ptr(),
                                   sc.scratch_bytes, sc.status.data_ptr(), None)
    assert st == fp.OK
    assert sc.status_bits() == 8   # a bounded device wait gave up, nothing else
    assert ref.status == oracle.OK
    np.testing.assert_array_equal(offs.cpu().numpy().view(np.uint32), ref.offsets)
    assert np.array_equal(out.cpu().numpy(), ref.data)
    sc.decode(out, offs)           # the library itself
    assert sc.status_bits() == 0
    assert np.array_equal(out.cpu().numpy(), ref.data)
