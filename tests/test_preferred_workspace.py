"""The workspace size of a call's fastest path (fwi_workspace_preferred_bytes):
host-side checks."""
import os
import subprocess
import sys

import numpy as np

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


class _Geometry:
    """fwi.Geometry without a GPU: the size queries do not read the wavelet"""

    def __init__(self, src, rec):
        self.src, self.rec = (np.ascontiguousarray(x, dtype=np.int32) for x in (src, rec))

    def c(self):
        from paper_1406_1864_gb300 import _lib as L
        return L.FwiGeometry(self.rec.shape[0], self.rec.shape[1], self.src.ctypes.data, self.rec.ctypes.data, 64)


def _problem(nz, nx, ns, rec, nt=60):
    from paper_1406_1864_gb300 import fwi
    src = np.stack([np.zeros(ns, int), np.zeros(ns, int), np.arange(ns) % nx], 1)
    return fwi.Grid(nz, nx, 10.0, 1e-3, nt, 8), _Geometry(src, np.broadcast_to(rec, (ns,) + rec.shape))


def _sizes(probs, opts):
    from paper_1406_1864_gb300 import fwi
    g, ge = [p[0] for p in probs], [p[1] for p in probs]
    return fwi.batch_workspace_bytes(g, ge, opts), fwi.preferred_workspace_bytes(g, ge, opts, "gradient")


def _line(nx):
    return np.stack([np.ones(nx, int), np.zeros(nx, int), np.arange(nx)], 1)


def test_levels_count_only_where_the_call_keeps_them():
    """Kept levels of the offset Hessian: none for pinned shapes, for receivers
    too dense for a resident pass, and in a batch that runs its models' forward
    passes in one launch per level."""
    from paper_1406_1864_gb300 import fwi
    opts = fwi.Options(hmax=10, precond="offset")
    small, large = _problem(37, 83, 3, _line(83)), _problem(400, 1200, 64, _line(1200))
    zz, xx = np.meshgrid(np.arange(37), np.arange(83), indexing="ij")
    dense = _problem(37, 83, 3, np.stack([zz.ravel(), 0 * zz.ravel(), xx.ravel()], 1))
    fwi.autotune_reset()
    need, more = _sizes([small], opts)
    assert more >= need + 59 * 3 * 37 * 83 * 4
    need, more = _sizes([large], opts)
    assert more == need
    need, more = _sizes([dense], opts)
    assert more == need
    need, more = _sizes([small, large], opts)
    assert more == need
    need, more = _sizes([small, small], opts)
    assert more >= need + 2 * 59 * 3 * 37 * 83 * 4
    try:
        fwi.autotune_set(small[0], small[1], opts, {"forward_variant": 2, "forward_chunk": 16, "backward_variant": 0,
                                                    "backward_chunk": 8})
        need, more = _sizes([small], opts)
        assert more == need
    finally:
        fwi.autotune_reset()
