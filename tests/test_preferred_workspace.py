"""The workspace size of a call's fastest path (fwi_workspace_preferred_bytes):
host-side checks."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_model_is_refused_before_the_grids_are_read():
    """(in a child process: grids points to no readable memory)"""
    code = """
import ctypes
from paper_1406_1864_gb300 import _lib as L
lib = L.load()
f = lib.fwi_workspace_preferred_bytes
f.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 3 + [ctypes.c_int, ctypes.c_void_p]
n, o = ctypes.c_size_t(7), L.FwiOptions(0, 0, -1, 1, 1e-3)
for models in (0, -1):
    assert f(models, 64, 64, ctypes.addressof(o), L.FWI_OP_GRADIENT, ctypes.addressof(n)) == L.FWI_ERR_INVALID_ARG
assert n.value == 7
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
