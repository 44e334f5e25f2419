"""Products before and after a cudaDeviceReset of the calling process's own
context, in a child process without any other user of CUDA: the plans' kept words
and events and the kernels' shared-memory attributes (tables of more than 48 KB a
CTA) belong to the context that ended."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import ctypes, sys
sys.path.insert(0, ROOT)
import numpy as np
import oracle, synth
import paper_2408_14558_gb300 as g
lib = g.load_library()
rt = ctypes.CDLL("libcudart.so.13")
A = synth.uniform_columns(2000, 15, seed=1)      # about 210 rows a column: tables of 512 slots
ref = oracle.spgemm(A, A)
cp, ri = A.colptr.astype(np.int64), A.rowidx.astype(np.int32)
M = g.spg_csc(2000, 2000, ri.size, g.SPG_IDX_I64, g.SPG_IDX_I32, g.SPG_VAL_F64, 0, cp.ctypes.data, ri.ctypes.data,
              A.vals.ctypes.data)
lib.spgemm_1d_multiply_host.argtypes = [ctypes.POINTER(g.spg_csc), ctypes.POINTER(g.spg_csc),
                                        ctypes.POINTER(g.spg_options), ctypes.c_int32, g.HOST_ALLOC_FN,
                                        g.HOST_FREE_FN, ctypes.c_void_p, ctypes.POINTER(g.spg_csc)]
for turn in range(4):
    for again in range(2):
        held = {}
        def take(nbytes, ctx):
            a = np.empty(nbytes, np.uint8)
            held[a.ctypes.data] = a
            return a.ctypes.data
        o, C = g.spg_options(), g.spg_csc()
        lib.spgemm_default_options(ctypes.byref(o))
        o.P, o.b = 3, 64
        alloc, free = g.HOST_ALLOC_FN(take), g.HOST_FREE_FN(lambda p, n, c: None)
        s = lib.spgemm_1d_multiply_host(ctypes.byref(M), ctypes.byref(M), ctypes.byref(o), 2, alloc, free, None,
                                        ctypes.byref(C))
        assert s == 0, g.spgemm_last_error()
        view = lambda p, dt, n: held[p].view(dt)[:n]
        assert np.array_equal(view(C.colptr, np.int64, 2001), ref["colptr"])
        assert np.array_equal(view(C.rowidx, np.int32, C.nnz), ref["rowidx"])
        assert np.all(np.abs(view(C.vals, np.float64, C.nnz) - ref["vals"]) <= 1e-12 * ref["absum"])
    assert rt.cudaDeviceReset() == 0
print("resets ok")
'''


def test_products_around_device_resets():
    r = subprocess.run([sys.executable, "-c", f"ROOT = {ROOT!r}\n" + CHILD], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "resets ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
