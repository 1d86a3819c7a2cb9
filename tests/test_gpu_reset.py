"""A process that resets the device between two stores."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = """
import ctypes as C
import numpy as np
import torch                                                    # (the CUDA runtime that the library is linked to)
from paper_2411_04975_b200 import binding

lib, rt = binding.library(), C.CDLL("libcudart.so.12")
rt.cudaMalloc.argtypes = [C.POINTER(C.c_void_p), C.c_size_t]
rt.cudaMemcpy.argtypes = [C.c_void_p, C.c_void_p, C.c_size_t, C.c_int]


def device(a):
    p = C.c_void_p()
    assert rt.cudaMalloc(C.byref(p), max(a.nbytes, 1)) == 0
    assert rt.cudaMemcpy(p, a.ctypes.data, a.nbytes, 1) == 0
    return p


for turn in range(2):
    prm, store = binding._BuildParams(50, 8, 2, 64, 64, -1, 0), C.c_void_p()
    assert lib.sd_build(C.byref(prm), None, None, 0, None, C.byref(store)) == 0
    tokens = (np.arange(40) % 7).astype(np.int32)
    rc = lib.sd_append(store, 2, device(np.array([-1, 0], np.int32)), device(np.array([0, 30, 40], np.int64)), device(tokens), None, None)
    assert rc == 0, (turn, rc)
    spec, M, out = binding._SpecParams(4, 2.0, 8, 0, 0.0), 64, [device(np.zeros(2 * 64, np.int64)) for _ in range(9)]
    for _ in range(2):
        rc = lib.sd_speculate(store, 1, device(np.array([0], np.int32)), C.byref(spec), None, *out, None)
        assert rc == 0, (turn, rc)
    n_draft = np.zeros(1, np.int32)
    assert rt.cudaMemcpy(n_draft.ctypes.data, out[0], 4, 2) == 0 and n_draft[0] > 0
    st = binding._Stats()
    assert lib.sd_stats(store, C.byref(st), None) == 0
    assert st.global_tokens == 30 and st.global_nodes == 7 * 8
    lib.sd_free(store)
    lib.sd_trim()
    assert rt.cudaDeviceReset() == 0
print("done")
"""


def test_appends_and_drafts_after_a_device_reset():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.endswith("done\n"), r.stderr
