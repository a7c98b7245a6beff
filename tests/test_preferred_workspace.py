"""The workspace size of a call's fastest path (fwi_workspace_preferred_bytes):
host-side checks."""
import os
import subprocess
import sys

import numpy as np
import pytest

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


def _tight(limit, device):
    """a Workspace on a device without room for more than limit bytes"""
    import torch
    from paper_1406_1864_gb300 import fwi

    class Tight(fwi.Workspace):
        tries = 0

        def get(self, nbytes):
            if nbytes > limit:
                Tight.tries += 1
                raise torch.cuda.OutOfMemoryError("no room")
            return super().get(nbytes)

    return Tight(torch.device(device))


def test_a_refused_allocation_falls_back_to_the_size_the_call_needs():
    import torch
    from paper_1406_1864_gb300 import fwi
    ws = _tight(1000, "cpu")
    for _ in range(2):  # (the second call does not try again)
        buf, n = fwi._ws(ws, 5000, lambda: 800)
        assert n >= 800 and buf is ws.buf and type(ws).tries == 1
    buf, n = fwi._ws(ws, 900, lambda: 300)
    assert n >= 900
    with pytest.raises(torch.cuda.OutOfMemoryError):
        fwi._ws(ws, 2000)
    with pytest.raises(torch.cuda.OutOfMemoryError):
        fwi._ws(_tight(1000, "cpu"), 5000, lambda: 4000)


@pytest.mark.gpu
def test_calls_without_room_for_their_levels_run():
    """Every call that asks for the preferred size runs with the required one:
    the sums after each level, the same to FP32 rounding (1e-5, as between a
    workspace with and without room for the levels)."""
    import torch
    from paper_1406_1864_gb300 import fwi, workloads as W
    p = W.dipping(nz=37, nx=83, nt=60, ns=3, nrec=83, sponge=7)
    grid, geom = fwi.from_problem(p)
    v = torch.as_tensor(p.v_init, device="cuda")
    d = fwi.forward(grid, geom, torch.as_tensor(p.v_true, device="cuda"))
    opts = fwi.Options(hmax=10, precond="offset")
    calls = {"gradient": lambda ws: fwi.adjoint_gradient(grid, geom, v, d, opts, ws=ws),
             "batch": lambda ws: fwi.batch_gradient([grid] * 2, [geom] * 2, [v] * 2, [d] * 2, opts, ws=ws)[1],
             "graph": lambda ws: fwi.GradientGraph([grid], [geom], [v], [d], opts, ws=ws).run()[0],
             "offset_hessian": lambda ws: {"offh": fwi.offset_hessian_diag(grid, geom, v, opts, ws=ws)}}
    need = {"gradient": fwi.workspace_bytes(grid, geom, opts, "gradient"),
            "batch": fwi.batch_workspace_bytes([grid] * 2, [geom] * 2, opts),
            "graph": fwi.batch_workspace_bytes([grid], [geom], opts),
            "offset_hessian": fwi.workspace_bytes(grid, geom, opts, "offset_hessian")}
    for name, call in calls.items():
        full, ws = call(None), _tight(need[name], "cuda")
        res = call(ws)
        assert type(ws).tries == 1, name
        for k in ("offh", "grad"):
            if k in full:
                assert float((res[k] - full[k]).double().norm()) <= 1e-5 * float(full[k].double().norm()), (name, k)
