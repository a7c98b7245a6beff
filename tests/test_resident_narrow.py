"""Models of one to three columns in the chip-resident loops: sponge cells on both
sides of the model within four columns, which share a float4 of the checkpoint."""
import numpy as np
import pytest

from paper_1406_1864_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hmax", [-1, 3])
@pytest.mark.parametrize("nx,P", [(1, 1), (1, 2), (1, 6), (2, 1), (2, 2), (2, 5), (3, 1), (3, 3)])
def test_narrow_models_match_the_streaming_steps(nx, P, hmax):
    """Both passes are resident (one launch each); traces bit for bit, sums in
    another order (relative L2 1e-6; the offset Hessian 1e-5, at most 60 products
    per point)."""
    import torch
    from paper_1406_1864_gb300 import fwi
    nt, ns = 30, 2
    rng = np.random.default_rng(10 * nx + P)
    p = W.homogeneous(40, nx, v=2500.0, dt=1e-3, nt=nt, f0=25.0, sponge=P, src=[[0, 0, 0], [39, 0, nx - 1]],
                      rec=np.stack([np.full(nx, 1), np.zeros(nx, int), np.arange(nx)], 1))
    p.wavelet[:] = rng.standard_normal(p.wavelet.shape).astype(np.float32)
    grid, geom = fwi.from_problem(p)
    v = torch.as_tensor((2500 + 300 * rng.random((40, nx))).astype(np.float32), device="cuda")
    d = torch.as_tensor(rng.standard_normal((ns, nt, geom.nrec)).astype(np.float32), device="cuda")
    opts = fwi.Options(hmax=hmax, precond="none")

    def call():
        fwi.profile(True)
        try:
            t = fwi.forward(grid, geom, v)
            g = fwi.adjoint_gradient(grid, geom, v, d, opts)
            return t, g, fwi.last_phase_times()
        finally:
            fwi.profile(False)

    fwi.autotune_reset()
    a = call()
    try:
        for o, variant in ((fwi.Options(precond="none"), 0), (opts, 2 if hmax >= 0 else 0)):
            fwi.autotune_set(grid, geom, o, {"forward_variant": variant, "forward_chunk": 8, "backward_variant": 0,
                                              "backward_chunk": 8})
        b = call()
    finally:
        fwi.autotune_reset()
    assert a[2]["forward_launches"] == (2 if hmax >= 0 else 1) and a[2]["adjoint_launches"] == 1
    assert b[2]["forward_launches"] == nt and b[2]["adjoint_launches"] == nt - 1
    assert torch.equal(a[0], b[0])
    for k, tol in (("grad", 1e-6), ("illum", 1e-6), ("offh", 1e-5)):
        if k in b[1]:
            assert float((a[1][k] - b[1][k]).double().norm()) <= tol * float(b[1][k].double().norm()), k
