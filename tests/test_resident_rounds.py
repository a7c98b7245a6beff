"""Several rounds of shots in the chip-resident 2-D time loops: a tile goes on to
its next shots with no barrier between tiles, so the packet buffers of the
exchange have to stay apart over a round's end too.

On the CPU: every order in which three neighbouring tiles can send, read and
step is followed with the library's choice of buffer (fwi_resident.h, compiled
here); none may leave a tile waiting for a packet that was overwritten. On the
GPU: passes of several rounds and tiles against the streaming steps."""
import ctypes

import numpy as np
import pytest

import native
from paper_1406_1864_gb300 import workloads as W

HELPER = """
#include "fwi_resident.h"
extern "C" int slot(int round, int nt, int v) { return fwi::res_slot(round, nt, v); }
extern "C" void plan(int nz, int nx, int P, int ns, int kind, int *out)
{
    fwi::Lay2D L{};
    L.nz = nz, L.nx = nx, L.P = P, L.nzp = nz + 2 * P, L.nxp = nx + 2 * P;
    const fwi::ResTile t = fwi::res_plan(L, ns, (fwi::ResKind)kind);
    out[0] = t.ok ? (t.per + t.s - 1) / t.s : 0;
    out[1] = t.ntx * t.ntz;
    out[2] = t.ok ? t.accs / t.sets : 0; // groups of warps
}
"""
KINDS = {"plain": 0, "illum": 1, "adjoint": 3}


@pytest.fixture(scope="module")
def helper(tmp_path_factory):
    return native.compile_helper(HELPER, tmp_path_factory.mktemp("resident"))


def stuck(slot, nt, rounds, tiles=3):
    """Whether some order of the tiles' actions leaves one waiting for ever.

    A tile's state: round, level v it has computed, levels sent, packets read
    (neighbour by neighbour, in order). The warps of a CTA as in the loops: level
    v + 1 is computed once level v's packets are read and level v - 1 is sent;
    level v is sent once computed; a tile reads level v's packets once it has
    computed level v - 1. Levels 1 .. nt - 2 are exchanged, levels 0 .. nt - 1
    computed."""
    nb = [[k for k in (t - 1, t + 1) if 0 <= k < tiles] for t in range(tiles)]
    last = nt - 2

    def moves(state):
        st, buf = state
        for t, (r, v, sent, read) in enumerate(st):
            n = len(nb[t])

            def to(**kw):
                new = dict(r=r, v=v, sent=sent, read=read)
                new.update(kw)
                return st[:t] + ((new["r"], new["v"], new["sent"], new["read"]),) + st[t + 1:]

            if r == rounds:
                continue
            if sent < min(v, last):  # the next level's packets, over what the buffer held
                b = list(buf)
                b[2 * t + slot(r, nt, sent + 1)] = (r, sent + 1)
                yield to(sent=sent + 1), tuple(b)
            lv = read // n + 1
            if lv <= last and v >= lv - 1 and buf[2 * nb[t][read % n] + slot(r, nt, lv)] == (r, lv):
                yield to(read=read + 1), buf
            if v < nt - 1 and read >= n * min(v, last) and sent >= min(v - 1, last):
                yield to(v=v + 1), buf
            if v == nt - 1 and sent == last and read == n * last:
                yield to(r=r + 1, v=0, sent=0, read=0), buf

    start = (((0, 0, 0, 0),) * tiles, (None,) * (2 * tiles))
    seen, todo = {start}, [start]
    while todo:
        s = todo.pop()
        nxt = list(moves(s))
        if not nxt and any(t[0] != rounds for t in s[0]):
            return True
        for m in nxt:
            if m not in seen:
                seen.add(m)
                todo.append(m)
    return False


@pytest.mark.parametrize("nt", [2, 3, 4, 5, 6, 7])
def test_no_order_of_the_tiles_loses_a_packet(helper, nt):
    assert not stuck(helper.slot, nt, rounds=3)


def test_the_levels_parity_would_lose_packets_where_nt_is_odd():
    """(the search finds the fault of buffers picked by the level alone)"""
    assert [stuck(lambda r, nt, v: v & 1, nt, rounds=3) for nt in (3, 4, 5, 6)] == [True, False, True, False]


# nz, nx, sponge, shots and the passes that are resident with several rounds and tiles
CASES = [(61, 100, 20, 64, ("adjoint",)), (50, 131, 5, 97, ("adjoint",)), (120, 131, 5, 97, ("plain", "illum")),
         (61, 494, 10, 97, ("plain", "illum")), (300, 1000, 20, 9, ("plain",))]


@pytest.mark.gpu
@pytest.mark.parametrize("nt", [24, 25, 3])
@pytest.mark.parametrize("nz,nx,P,ns,passes", CASES)
def test_several_rounds_match_the_streaming_steps(helper, nz, nx, P, ns, passes, nt):
    """Traces bit for bit, sums in another order (relative L2 1e-6, as between the
    tile variants)."""
    compare(helper, nz, nx, P, ns, passes, nt, 1, "u2")


# passes of two groups of warps: a last round of one shot (a group without one), sets without shots, odd counts
GROUPS = [(100, 494, 10, 61, ("plain",)), (37, 222, 20, 81, ("illum",)), (20, 131, 20, 77, ("adjoint",))]


@pytest.mark.gpu
@pytest.mark.parametrize("nt,illum", [(24, "u2"), (25, "utt2")])
@pytest.mark.parametrize("nz,nx,P,ns,passes", GROUPS)
def test_two_groups_of_warps_match_the_streaming_steps(helper, nz, nx, P, ns, passes, nt, illum):
    compare(helper, nz, nx, P, ns, passes, nt, 2, illum)


def compare(helper, nz, nx, P, ns, passes, nt, groups, illum):
    import torch
    from paper_1406_1864_gb300 import fwi
    rng = np.random.default_rng(nz + ns + nt)
    p = W.homogeneous(nz, nx, v=2500.0, dt=1e-3, nt=nt, f0=25.0, sponge=P,
                      src=np.stack([rng.integers(0, nz, ns), np.zeros(ns, int), rng.integers(0, nx, ns)], 1),
                      rec=np.stack([np.full(nx, 1), np.zeros(nx, int), np.arange(nx)], 1))
    p.wavelet[:] = rng.standard_normal(p.wavelet.shape).astype(np.float32)
    grid, geom = fwi.from_problem(p)
    v = torch.as_tensor((2500 + 300 * rng.random((nz, nx))).astype(np.float32), device="cuda")
    d = torch.as_tensor(rng.standard_normal((ns, nt, geom.nrec)).astype(np.float32), device="cuda")
    opts = fwi.Options(illum=illum, precond="none")
    for k in passes:
        o = (ctypes.c_int * 3)()
        helper.plan(nz, nx, P, ns, KINDS[k] + (k == "illum" and illum == "utt2"), o)
        assert o[0] > 1 and o[1] > 1 and o[2] >= groups

    def call():
        fwi.profile(True)
        try:
            t = fwi.forward(grid, geom, v)
            plain = fwi.last_phase_times()
            g = fwi.adjoint_gradient(grid, geom, v, d, opts)
            grad = fwi.last_phase_times()
        finally:
            fwi.profile(False)
        return (t, g), {"plain": plain["forward_launches"], "illum": grad["forward_launches"],
                        "adjoint": grad["adjoint_launches"]}

    fwi.autotune_reset()
    a, la = call()
    try:
        fwi.autotune_set(grid, geom, opts, {"forward_variant": 0, "forward_chunk": 8, "backward_variant": 0,
                                             "backward_chunk": 8})
        b, lb = call()
    finally:
        fwi.autotune_reset()
    assert all(la[k] == 1 for k in passes) and lb == {"plain": nt, "illum": nt, "adjoint": nt - 1}
    assert torch.equal(a[0], b[0])
    assert float((a[1]["grad"] - b[1]["grad"]).double().norm()) <= 1e-6 * float(b[1]["grad"].double().norm())
    assert float((a[1]["illum"] - b[1]["illum"]).double().norm()) <= 1e-6 * float(b[1]["illum"].double().norm())
