"""Timing cases of the library's public entry points.

Each case is one call a user's program makes, at sizes taken from the named
workloads, the tests, the timing modules and the inversion experiment: data
modelling, the preconditioned gradient (small, inversion and benchmark size,
called directly, recorded as a graph, or batched over models), autograd with
snapshot checkpoints, Gauss-Newton products, extended imaging, the 3-D
gradient and the division by a preconditioner.

listed() gives the standing cases, draw(rng) further ones of the same ranges;
prepare() makes a case's inputs and keeps what such a program keeps (geometry,
workspace, recorded graph); run() makes the call; work() counts what the
method cannot do without; exact() evaluates the same quantities in FP64 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1406_1864_gb300 import autograd, fwi, workloads as W

KINDS = ("precondition", "forward", "gradient", "graph", "batch", "autograd", "hvp", "extended", "gradient3d")


def _case(kind, nz, nx, ns, nt, **kw):
    c = {"kind": kind, "nz": nz, "ny": 1, "nx": nx, "ns": ns, "nt": nt, "dx": 10.0, "dt": 8e-4, "f0": 8.0,
         "sponge": 20, "rec_step": 2, "misfit": "ols", "hmax": -1, "precond": "illum", "snap": "f32", "hext": 0}
    c.update(kw)
    return c


def listed():
    cases = [
        # M^-1 g of one outer iteration (PRCG, L-BFGS) at the inversion experiment's size: the smallest call
        ("precondition_offset_150x460", _case("precondition", 150, 460, 1, 2, hmax=10, precond="offset")),
        # modelling of a few shots on a small model (the two-layer workload)
        ("forward_100x200_4shots", _case("forward", 100, 200, 4, 1000, dt=1e-3, f0=10.0, rec_step=1)),
        # a small ragged model (no multiple of a tile or of 4), the size that checks and tutorials use
        ("gradient_37x83_3shots", _case("gradient", 37, 83, 3, 300, dt=1e-3, f0=10.0, sponge=7, rec_step=1)),
        # the two-layer workload with both of the paper's preconditioning ingredients
        ("gradient_100x200_4shots", _case("gradient", 100, 200, 4, 1000, dt=1e-3, f0=10.0, rec_step=1,
                                          misfit="integral", hmax=10, precond="offset")),
        # one gradient of the inversion experiment (every optimiser iteration calls this)
        ("gradient_150x460_80shots", _case("gradient", 150, 460, 80, 800, dx=20.0, dt=1.5e-3, f0=6.0, rec_step=1,
                                           misfit="integral")),
        # the benchmark's gradient (time levels cut), tuned and recorded as a graph as the benchmark does
        ("graph_300x1000_96shots", _case("graph", 300, 1000, 96, 500, misfit="integral", hmax=10, precond="offset")),
        # data modelling and line-search passes on the largest named 2-D workload
        ("forward_400x1200_64shots", _case("forward", 400, 1200, 64, 300)),
        # three independent models of uneven sizes in one call
        ("batch_3models_16shots", _case("batch", 200, 400, 16, 200)),
        # a torch loss on differentiable traces, sqrt(nt) snapshots
        ("autograd_400x1200_32shots", _case("autograd", 400, 1200, 32, 400)),
        # one Gauss-Newton Hessian-vector product of the inner CG
        ("hvp_300x1000_48shots", _case("hvp", 300, 1000, 48, 300)),
        # extended migration over subsurface offsets (Eq. 6)
        ("extended_300x1000_32shots", _case("extended", 300, 1000, 32, 200, hext=4)),
        # a 3-D gradient with snapshot checkpoints
        ("gradient3d_100x200x200_4shots", _case("gradient3d", 100, 200, 4, 60, ny=200, dx=12.5, dt=1e-3,
                                                rec_step=4)),
    ]
    return [dict(c, name=n) for n, c in cases]


# point-steps x passes of the largest listed case (the benchmark's gradient)
_MOST = 300 * 1000 * 96 * 500 * 3


def _passes(kind):
    return {"precondition": 0, "forward": 1, "autograd": 4, "hvp": 4, "extended": 5, "gradient3d": 8}.get(kind, 3)


def draw(rng):
    def span(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(KINDS)
    if kind == "precondition":
        return _case(kind, span(30, 500), span(60, 1500), 1, 2, hmax=rng.choice((0, 3, 10, 12)),
                     precond=rng.choice(("illum", "offset")))
    if kind == "gradient3d":
        nz, ny, nx, ns, nt = span(24, 100), span(30, 200), span(30, 200), rng.randint(1, 4), span(20, 60)
        return _case(kind, nz, nx, ns, nt, ny=ny, dx=12.5, dt=1e-3, rec_step=rng.choice((1, 2, 4)),
                     sponge=rng.choice((8, 10, 20)), hmax=rng.choice((-1, -1, 3)), snap=rng.choice(("f32", "bf16")))
    nz, nx, ns, nt = span(36, 400), span(80, 1200), span(1, 96), span(100, 1000)
    if kind == "batch":
        nz, nx, ns = min(nz, 200), min(nx, 600), min(ns, 32)
    points = nz * nx * (8 if kind == "batch" else 1)
    cap = 0.5 * _MOST / max(1, _passes(kind))
    while points * ns * nt > cap and (ns > 1 or nt > 100):
        ns, nt = max(1, (3 * ns) // 4), max(100, (3 * nt) // 4)
    full = kind in ("gradient", "graph", "batch")
    hmax = rng.choice((-1, 3, 10, 12)) if full else -1
    precond = rng.choice(("illum", "offset")) if hmax >= 0 else "illum"
    return _case(kind, nz, nx, ns, nt, sponge=rng.choice((20, 20, 10, 15)), rec_step=rng.choice((1, 2)),
                 misfit=rng.choice(("ols", "integral")) if full or kind == "hvp" else "ols", hmax=hmax,
                 precond=precond, snap=rng.choice(("f32", "bf16", "f16s")), hext=rng.choice((2, 4)) if
                 kind == "extended" else 0)


# ------------------------------------------------------------------ inputs

def _batch_sizes(case):
    nz, nx = case["nz"], case["nx"]
    return [(nz, nx), ((7 * nz) // 4, (9 * nx) // 4), ((5 * nz) // 2, (15 * nx) // 4)]


def _problems(case, seed):
    """The case's modelling problems (host arrays), one per model."""
    c = case
    if c["kind"] == "gradient3d":
        return [W.dipping3d(nz=c["nz"], ny=c["ny"], nx=c["nx"], dx=c["dx"], dt=c["dt"], nt=c["nt"], ns=c["ns"],
                            rec_step=c["rec_step"], f0=c["f0"], seed=seed, sponge=c["sponge"], smooth_m=60.0)]
    sizes = _batch_sizes(c) if c["kind"] == "batch" else [(c["nz"], c["nx"])]
    return [W.dipping(nz=nz, nx=nx, dx=c["dx"], dt=c["dt"], nt=c["nt"], ns=c["ns"], nrec=nx,
                      rec_step=c["rec_step"], f0=c["f0"], seed=seed + 1000 * k, sponge=c["sponge"])
            for k, (nz, nx) in enumerate(sizes)]


def _options(c):
    snapshot = c["kind"] in ("autograd", "gradient3d")
    return fwi.Options(misfit=c["misfit"], hmax=c["hmax"], precond=c["precond"],
                       ckpt="snapshot" if snapshot else "sponge", snap=c["snap"])


def _precondition_inputs(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = (c["nz"], c["nx"])
    grad = torch.randn(shape, device="cuda", generator=gen)
    planes = (c["hmax"] + 1,) if c["precond"] == "offset" else ()
    # positive, falling with depth by orders of magnitude, as an illumination does
    depth = torch.linspace(0.0, 9.0, shape[0], device="cuda")[:, None]
    scale = torch.exp(0.5 * torch.randn(planes + shape, device="cuda", generator=gen) - depth)
    return grad, scale.contiguous()


def _extended_source(c, p, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((p.nshots, p.nt, p.nrec), device="cuda", generator=gen)


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "precondition":
        grad, scale = _precondition_inputs(c, seed)
        return {"kind": c["kind"], "grid": fwi.Grid(c["nz"], c["nx"], c["dx"], c["dt"], c["nt"], c["sponge"]),
                "grad": grad, "scale": scale, "precond": c["precond"], "ws": fwi.Workspace()}
    probs = _problems(c, seed)
    gg = [fwi.from_problem(p) for p in probs]
    s = {"kind": c["kind"], "grids": [g for g, _ in gg], "geoms": [g for _, g in gg], "opts": _options(c),
         "v": [torch.as_tensor(p.v_init, device="cuda") for p in probs], "ws": fwi.Workspace()}
    if c["kind"] in ("gradient", "graph", "batch", "autograd", "gradient3d"):
        s["d_obs"] = [fwi.forward(g, ge, torch.as_tensor(p.v_true, device="cuda"))
                      for (g, ge), p in zip(gg, probs)]
    if c["kind"] == "hvp":
        s["dv"] = torch.as_tensor((probs[0].v_true - probs[0].v_init).astype(np.float32), device="cuda")
    if c["kind"] == "extended":
        s["adj"], s["hext"] = _extended_source(c, probs[0], seed), c["hext"]
    if c["kind"] == "graph":
        fwi.autotune(s["grids"][0], s["geoms"][0], s["v"][0], s["opts"], ws=s["ws"])
        s["graph"] = fwi.GradientGraph(s["grids"], s["geoms"], s["v"], s["d_obs"], s["opts"], ws=s["ws"])
    if c["kind"] == "autograd":
        s["v"][0].requires_grad_(True)
    return s


def run(s):
    kind = s["kind"]
    if kind == "precondition":
        return fwi.precondition(s["grid"], s["grad"], s["scale"], s["precond"], ws=s["ws"])
    grid, geom, v, ws = s["grids"][0], s["geoms"][0], s["v"][0], s["ws"]
    if kind == "forward":
        return fwi.forward(grid, geom, v, ws=ws)
    if kind in ("gradient", "gradient3d"):
        return fwi.adjoint_gradient(grid, geom, v, s["d_obs"][0], s["opts"], ws=ws)
    if kind == "graph":
        return s["graph"].run()
    if kind == "batch":
        return fwi.batch_gradient(s["grids"], s["geoms"], s["v"], s["d_obs"], s["opts"], ws=ws)
    if kind == "autograd":
        d = autograd.traces(v, grid, geom, s["opts"])
        loss = 0.5 * (d - s["d_obs"][0]).square().sum()
        (g,) = torch.autograd.grad(loss, v)
        return d.detach(), g
    if kind == "hvp":
        return fwi.gauss_newton_hvp(grid, geom, v, s["dv"], s["opts"], ws=ws)
    if kind == "extended":
        return fwi.extended_migration(grid, geom, v, s["adj"], s["hext"], ws=ws)
    raise ValueError(kind)


def work(case):
    """One pass: every input read once, every output written once; the
    arithmetic of the leapfrog (per padded point and level: the 8 z and 8 x
    pair sums and weights of the 2-D Laplacian and the update) of each
    propagated field, the imaging and the sums."""
    c = case
    h = c["hmax"] + 1
    if c["kind"] == "precondition":
        n = c["nz"] * c["nx"]
        planes = h if c["precond"] == "offset" else 1
        return {"bytes": 4.0 * n * (2 + planes), "flops": float(n * (planes + 2))}
    three = c["kind"] == "gradient3d"
    sizes = _batch_sizes(c) if c["kind"] == "batch" else [(c["nz"], c["nx"])]
    nbytes = flops = 0.0
    for nz, nx in sizes:
        ny, ns, nt = c["ny"], c["ns"], c["nt"]
        n = nz * ny * nx
        pad = (nz + 2 * c["sponge"]) * (ny + 2 * c["sponge"] if three else 1) * (nx + 2 * c["sponge"])
        per = -(-nx // c["rec_step"])
        nrec = per * -(-ny // c["rec_step"]) if three else per
        traces = 4.0 * ns * nt * nrec
        model = 4.0 * n
        step = 3 * 17 + 5 if three else 2 * 17 + 5
        levels = float(pad) * ns * nt
        phys = float(n) * ns * nt
        if c["kind"] == "forward":
            nbytes += model + traces
            flops += step * levels
        elif c["kind"] == "hvp":
            nbytes += 3 * model
            flops += (4 * step + 4) * levels
        elif c["kind"] == "extended":
            nbytes += traces + model * (2 + 2 * c["hext"])
            flops += (2 * step + 2 * (2 * c["hext"] + 1)) * levels
        else:
            nbytes += traces + model * (4 + max(0, h)) + (traces if c["kind"] == "autograd" else 0)
            flops += (2 * step + 2) * levels + (2 + 2 * max(0, h - 1)) * phys
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------- FP64 evaluation

class _Exact:
    """The discrete scheme of one model in FP64 torch on the padded grid:
    leapfrog with the sponge, its Born form and its adjoint."""

    W8 = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)

    def __init__(self, p):
        f = lambda x: float(np.float32(x))  # noqa: E731  (the call takes its scalars in FP32)
        self.p, self.nd, self.P = p, p.ndim, int(p.sponge)
        self.dx, self.dt, self.nt = f(p.dx), f(p.dt), int(p.nt)
        self.shape = p.shape
        self.pad = tuple(n + 2 * self.P for n in self.shape)
        v = torch.as_tensor(p.v_init, device="cuda").double()
        self.idx = [torch.arange(-self.P, n + self.P, device="cuda").clamp(0, n - 1) for n in self.shape]
        self.v = v
        self.vp = self.spread(v)
        self.c2 = (self.vp * self.dt / self.dx) ** 2
        etamax = 3.0 * f(p.vref) * math.log(1.0 / f(p.refl)) / (2.0 * self.P * self.dx)
        e = torch.zeros(self.pad, dtype=torch.float64, device="cuda")
        for a, n in enumerate(self.shape):
            k = torch.arange(n + 2 * self.P, device="cuda")
            d = torch.maximum(self.P - k, k - (self.P + n - 1)).clamp(min=0).double() / self.P
            e += (d * d).reshape([-1 if b == a else 1 for b in range(self.nd)])
        self.ed = etamax * self.dt * e
        self.ia = 1.0 / (1.0 + self.ed)
        self.kb = (1.0 - self.ed) * self.ia
        axes = (0, 2) if self.nd == 2 else (0, 1, 2)
        strides = [int(np.prod(self.pad[k + 1:])) for k in range(self.nd)]
        flat = lambda q: sum((q[..., a].astype(np.int64) + self.P) * s for a, s in zip(axes, strides))  # noqa: E731
        self.src = torch.as_tensor(flat(p.src), device="cuda")
        self.rec = torch.as_tensor(flat(p.rec), device="cuda")
        self.wav = torch.as_tensor(p.wavelet, device="cuda").double() * self.dx ** (2 - self.nd)
        self.inner = tuple(slice(self.P, self.P + n) for n in self.shape)

    def spread(self, m):
        """A model-shaped array continued into the sponge by its edge values."""
        for a, i in enumerate(self.idx):
            m = m.index_select(m.dim() - self.nd + a, i)
        return m

    def fold(self, g):
        """The transpose of spread."""
        for a, (i, n) in enumerate(zip(self.idx, self.shape)):
            d = g.dim() - self.nd + a
            out = torch.zeros(g.shape[:d] + (n,) + g.shape[d + 1:], dtype=g.dtype, device=g.device)
            g = out.index_add_(d, i, g)
        return g

    def field(self, g, extra=0):
        shape = (g,) + tuple(n + 8 for n in self.pad)
        return [torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(2 + extra)]

    def mid(self, u):
        return u[(slice(None),) + (slice(4, -4),) * self.nd]

    def lap(self, u):
        q = self.mid(u) * (self.nd * self.W8[0])
        for a in range(self.nd):
            for k in range(1, 5):
                for s in (-k, k):
                    sl = [slice(None)] + [slice(4, -4)] * self.nd
                    sl[1 + a] = slice(4 + s, s - 4 if s < 4 else None)
                    q.add_(u[tuple(sl)], alpha=self.W8[k])
        return q

    def step(self, u, prev, q, add=None):
        """prev <- the next level (in place)."""
        m, mp = self.mid(u), self.mid(prev)
        new = (m - mp).mul_(self.kb).add_(m)
        new += q * (self.c2 * self.ia)
        if add is not None:
            new += add * self.ia
        mp.copy_(new)

    def groups(self, per_shot_bytes):
        ns = self.p.nshots
        g = max(1, min(ns, int(5e10 / max(1.0, per_shot_bytes)), int(6e8 / (8 * np.prod(self.pad))) + 1))
        return [(a, min(ns, a + g)) for a in range(0, ns, g)]

    def forward(self, s0, s1, keep=False, hmax=None, dv=None):
        """Traces [g, nt, nrec] (Born traces with dv), the sums of u^2 and of
        the offset products, and every level's q = Lhat u + f delta."""
        g, cells = s1 - s0, int(np.prod(self.pad))
        (u, up), born = self.field(g), None
        if dv is not None:
            born = self.field(g)
            dc2 = self.spread(dv) * 2.0 * self.c2 / self.vp
        rec = self.rec[s0:s1]
        seis = torch.zeros((g, self.nt, rec.shape[1]), dtype=torch.float64, device="cuda")
        qs = torch.zeros((self.nt - 1, g) + self.pad, dtype=torch.float64, device="cuda") if keep else None
        sums = None if hmax is None else torch.zeros((hmax + 1,) + self.shape, dtype=torch.float64, device="cuda")
        rows = torch.arange(g, device="cuda")
        for n in range(self.nt):
            m = self.mid(u)
            obs = m if born is None else self.mid(born[0])
            if rec.shape[1]:
                seis[:, n] = obs.reshape(g, cells).gather(1, rec)
            if sums is not None:
                for h in range(hmax + 1):
                    z = torch.nn.functional.pad(m, (h, h)) if h > self.P else m
                    o = self.P + max(0, h - self.P)
                    nx = self.shape[-1]
                    mi = (slice(None),) + self.inner[:-1]
                    sums[h] += (z[mi + (slice(o + h, o + h + nx),)] * z[mi + (slice(o - h, o - h + nx),)]).sum(0)
            if n == self.nt - 1:
                break
            q = self.lap(u)
            q.view(g, cells)[rows, self.src[s0:s1]] += self.wav[s0:s1, n]
            if keep:
                qs[n] = q
            if born is not None:
                self.step(born[0], born[1], self.lap(born[0]), q * dc2)
                born.reverse()
            self.step(u, up, q)
            u, up = up, u
        return seis, sums, qs

    def adjoint(self, s0, s1, a, qs, hext=None):
        """The imaging sum of the adjoint source a [g, nt, nrec] against qs:
        the gradient, or with hext the extended image [2 hext + 1, ...]."""
        g, cells = s1 - s0, int(np.prod(self.pad))
        psi, nxt = self.field(g)
        rec = self.rec[s0:s1]
        offs = [0] if hext is None else range(-hext, hext + 1)
        acc = torch.zeros((len(offs),) + self.pad, dtype=torch.float64, device="cuda")
        nxp = self.pad[-1]
        for m in range(self.nt - 1, 0, -1):
            q = self.lap(psi)
            q.view(g, cells).scatter_add_(1, rec, a[:, m].contiguous())
            self.step(psi, nxt, q)
            psi, nxt = nxt, psi
            now = self.mid(psi)
            for k, h in enumerate(offs):  # psi(y) q(y + 2h)
                lo, hi = max(0, -2 * h), nxp - max(0, 2 * h)
                acc[k][..., lo:hi] += (now[..., lo:hi] * qs[m - 1][..., lo + 2 * h:hi + 2 * h]).sum(0)
        if hext is None:
            return self.fold(acc[0]) * (2.0 / self.v)
        image = []
        for k, h in enumerate(offs):  # at x = y + h
            w = torch.zeros(self.pad, dtype=torch.float64, device="cuda")
            lo, hi = max(0, -h), nxp - max(0, h)
            w[..., lo + h:hi + h] = (acc[k] / self.vp ** 2)[..., lo:hi]
            image.append(self.fold(w) * 2.0 * self.v)
        return torch.stack(image)

    def weighted(self, r, misfit):
        """(misfit, adjoint source) of residual traces."""
        if misfit == "ols":
            return 0.5 * (r * r).sum(), r
        y = self.dt * torch.cumsum(r, 1)
        return 0.5 * (y * y).sum(), self.dt * torch.flip(torch.cumsum(torch.flip(y, (1,)), 1), (1,))


def _preconditioned(grad, scale, eps=1e-3):
    if scale.dim() > grad.dim():
        scale = scale[0].abs() + 2.0 * scale[1:].abs().sum(0)
    return grad / (scale + eps * scale.max())


def _exact_gradient(c, p, d_obs):
    x = _Exact(p)
    per = 8.0 * np.prod(x.pad) * p.nt
    grad, sums, J = 0.0, 0.0, 0.0
    for a, b in x.groups(per):
        seis, sm, qs = x.forward(a, b, keep=True, hmax=max(0, c["hmax"]))
        j, adj = x.weighted(seis - d_obs[a:b].double(), c["misfit"])
        grad = grad + x.adjoint(a, b, adj, qs)
        sums, J = sums + sm, J + j
        del qs
    offh = sums * x.dt
    out = {"grad": grad, "misfit": J, "illum": offh[0],
           "grad_pre": _preconditioned(grad, offh if c["precond"] == "offset" else offh[0])}
    if c["hmax"] >= 0:
        out["offh"] = offh
    return out


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "precondition":
        grad, scale = _precondition_inputs(c, seed)
        return _preconditioned(grad.double(), scale.double())
    s = prepare(dict(c, kind="gradient") if c["kind"] == "graph" else c, seed)
    probs = _problems(c, seed)
    if c["kind"] in ("gradient", "graph", "batch", "gradient3d"):
        res = [_exact_gradient(c, p, d) for p, d in zip(probs, s["d_obs"])]
        return res if c["kind"] in ("graph", "batch") else res[0]
    p = probs[0]
    x = _Exact(p)
    per = 8.0 * np.prod(x.pad) * p.nt
    if c["kind"] == "forward":
        return torch.cat([x.forward(a, b)[0] for a, b in x.groups(0.0)])
    traces, total = [], 0.0
    for a, b in x.groups(per):
        if c["kind"] == "hvp":
            seis, _, qs = x.forward(a, b, keep=True, dv=s["dv"].double())
            total = total + x.adjoint(a, b, x.weighted(seis, c["misfit"])[1], qs)
        elif c["kind"] == "extended":
            _, _, qs = x.forward(a, b, keep=True)
            total = total + x.adjoint(a, b, s["adj"][a:b].double(), qs, hext=c["hext"])
        else:
            seis, _, qs = x.forward(a, b, keep=True)
            traces.append(seis)
            total = total + x.adjoint(a, b, seis - s["d_obs"][0][a:b].double(), qs)
        del qs
    return (torch.cat(traces), total) if c["kind"] == "autograd" else total
