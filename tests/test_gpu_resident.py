"""The chip-resident 2-D time loops against the streaming steps (pinned with
fwi_autotune_set) on the same inputs. Both evaluate the same per-point
arithmetic, so traces are equal bit for bit; sums over shots and levels are
taken in another order (relative L2 1e-6, as between the tile variants).
Sizes at the edges of the layout: padded widths that are no multiple of 4,
sponge rows that are not contiguous in the checkpoint, one tile per shot,
tiles a few rows high, several rounds of shots with an uneven last one, two
and three time levels, receivers on every cell of a row and two on some cells
(the streaming step adds three or more in no fixed order), sources in corners."""
import numpy as np
import pytest

from paper_1406_1864_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# nz, nx, shots, nt, sponge
CASES = [(37, 83, 3, 90, 7), (20, 20, 1, 60, 20), (5, 300, 2, 50, 3), (90, 31, 5, 40, 1), (64, 128, 40, 30, 8),
         (61, 203, 97, 25, 5), (300, 1000, 9, 24, 20), (150, 460, 80, 20, 20), (33, 47, 2, 2, 4), (33, 47, 3, 3, 4),
         (400, 1201, 3, 12, 15), (40, 3, 2, 30, 2)]


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    torch.cuda.set_device(0)
    return torch


def rel(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm().clamp(min=1e-300))


def problem(torch, nz, nx, ns, nt, P):
    from paper_1406_1864_gb300 import fwi
    rng = np.random.default_rng(nz + 7 * nx + ns)
    p = W.homogeneous(nz, nx, v=2500.0, dt=1e-3, nt=nt, f0=25.0, sponge=P,
                      src=np.stack([rng.integers(0, nz, ns), np.zeros(ns, int), rng.integers(0, nx, ns)], 1),
                      rec=np.stack([np.full(nx + 3, min(1, nz - 1)), np.zeros(nx + 3, int),
                                    np.r_[np.arange(nx), 0, nx // 2, nx - 1]], 1))
    p.src[0] = (0, 0, 0)
    p.src[-1] = (nz - 1, 0, nx - 1)
    p.wavelet[:] = rng.standard_normal(p.wavelet.shape).astype(np.float32)
    grid, geom = fwi.from_problem(p)
    v = torch.as_tensor((2500 + 300 * rng.random((nz, nx))).astype(np.float32), device="cuda")
    d = torch.as_tensor(rng.standard_normal((ns, nt, geom.nrec)).astype(np.float32), device="cuda")
    return grid, geom, v, d


def both(fwi, grid, geom, opts, call):
    """call() with the resident loops and with the streaming steps."""
    fwi.autotune_reset()
    a = call()
    try:
        fwi.autotune_set(grid, geom, opts, {"forward_variant": 0, "forward_chunk": 8, "backward_variant": 0,
                                             "backward_chunk": 8})
        b = call()
    finally:
        fwi.autotune_reset()
    return a, b


@pytest.mark.parametrize("nz,nx,ns,nt,P", CASES)
def test_resident_loops_match_the_streaming_steps(torch_cuda, nz, nx, ns, nt, P):
    from paper_1406_1864_gb300 import fwi
    torch = torch_cuda
    grid, geom, v, d = problem(torch, nz, nx, ns, nt, P)
    for illum in ("u2", "utt2"):
        opts = fwi.Options(illum=illum, precond="none")
        a, b = both(fwi, grid, geom, opts, lambda: (fwi.forward(grid, geom, v),
                                                    fwi.adjoint_gradient(grid, geom, v, d, opts)))
        assert torch.equal(a[0], b[0])
        assert abs(float(a[1]["misfit"]) - float(b[1]["misfit"])) <= 1e-12 * float(b[1]["misfit"])
        assert rel(a[1]["grad"], b[1]["grad"]) <= 1e-6
        assert rel(a[1]["illum"], b[1]["illum"]) <= 1e-6


@pytest.mark.parametrize("nx,P", [(1, 1), (2, 1), (1, 2), (2, 5)])
def test_models_of_one_or_two_columns(torch_cuda, nx, P):
    """Sponge cells on both sides of the model within four columns: these run
    the streaming steps."""
    from paper_1406_1864_gb300 import fwi
    torch = torch_cuda
    grid, geom, v, d = problem(torch, 40, nx, 2, 30, P)
    geom = fwi.Geometry(geom.src, geom.rec[:, :nx], geom.wavelet)
    d, opts = d[:, :, :nx].contiguous(), fwi.Options(precond="none")
    a, b = both(fwi, grid, geom, opts, lambda: (fwi.forward(grid, geom, v), fwi.adjoint_gradient(grid, geom, v, d, opts)))
    assert torch.equal(a[0], b[0])
    assert rel(a[1]["grad"], b[1]["grad"]) <= 1e-6 and rel(a[1]["illum"], b[1]["illum"]) <= 1e-6


def test_resident_forward_feeds_either_adjoint_pass(torch_cuda):
    """forward(save) and adjoint_apply, each resident or streaming: the
    checkpoints and final levels are the same."""
    from paper_1406_1864_gb300 import fwi
    torch = torch_cuda
    grid, geom, v, d = problem(torch, 75, 130, 6, 64, 9)
    opts = fwi.Options()
    pin = {"forward_variant": 0, "forward_chunk": 8, "backward_variant": 0, "backward_chunk": 8}
    out = []
    try:
        for first, second in ((0, 0), (0, 1), (1, 0), (1, 1)):
            ws = fwi.Workspace()
            fwi.autotune_reset()
            if first:
                fwi.autotune_set(grid, geom, opts, pin)
            fwi.forward(grid, geom, v, save=True, ws=ws)
            fwi.autotune_reset()
            if second:
                fwi.autotune_set(grid, geom, opts, pin)
            out.append(fwi.adjoint_apply(grid, geom, v, d, ws))
    finally:
        fwi.autotune_reset()
    for o in out[:-1]:
        assert rel(o, out[-1]) <= 1e-6


def test_crowded_tiles_take_the_streaming_adjoint(torch_cuda):
    """More receivers in a tile than a resident backward pass lists (a dense
    areal spread): the same gradient."""
    from paper_1406_1864_gb300 import fwi
    torch = torch_cuda
    zz, xx = np.meshgrid(np.arange(40), np.arange(60), indexing="ij")
    p = W.homogeneous(40, 60, nt=40, f0=25.0, sponge=6, src=[[20, 0, 30], [3, 0, 9]],
                      rec=np.stack([zz.ravel(), 0 * zz.ravel(), xx.ravel()], 1))
    grid, geom = fwi.from_problem(p)
    v = torch.as_tensor(p.v_init, device="cuda")
    d = torch.randn((2, 40, geom.nrec), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    opts = fwi.Options()
    a, b = both(fwi, grid, geom, opts, lambda: fwi.adjoint_gradient(grid, geom, v, d, opts))
    assert rel(a["grad"], b["grad"]) <= 1e-6


@pytest.mark.parametrize("hmax", [0, 3, 10, 12])
@pytest.mark.parametrize("nz,nx,ns,nt,P", [(37, 83, 3, 60, 7), (50, 130, 5, 40, 20), (8, 65, 1, 30, 1), (23, 64, 9, 70, 16)])
def test_offset_hessian_of_kept_levels(torch_cuda, nz, nx, ns, nt, P, hmax):
    """The offset-Hessian sums over the levels a resident pass keeps against
    those after each streaming step: widths around the 64-column tile, sponges
    narrower and wider than the 12 columns the sums read on each side, each
    compiled offset count, a last run of images that is not full. Both add the
    same FP32 products (at most 630 per point) in another order: 1e-5 is three
    times their random-walk rounding, 2^-24 sqrt(630) per side, in L2."""
    from paper_1406_1864_gb300 import fwi
    torch = torch_cuda
    grid, geom, v, d = problem(torch, nz, nx, ns, nt, P)
    opts = fwi.Options(hmax=hmax, precond="offset")
    a, b = both(fwi, grid, geom, opts, lambda: (fwi.adjoint_gradient(grid, geom, v, d, opts),
                                                fwi.offset_hessian_diag(grid, geom, v, opts)))
    for k in ("offh", "illum", "grad"):
        assert rel(a[0][k], b[0][k]) <= 1e-5, k
    assert rel(a[1], b[1]) <= 1e-5
    assert rel(a[0]["offh"][0], a[0]["illum"]) <= 1e-5
    # a workspace without room for the levels: the sums after each level
    small = torch.empty(fwi.workspace_bytes(grid, geom, opts, "gradient"), dtype=torch.uint8, device="cuda")
    assert small.numel() < fwi.preferred_workspace_bytes([grid], [geom], opts, "gradient")
    c = fwi.adjoint_gradient(grid, geom, v, d, opts, ws=small)
    assert rel(c["offh"], b[0]["offh"]) <= 1e-5 and rel(c["grad"], b[0]["grad"]) <= 1e-5
