"""Choices by problem size where nothing was autotuned, against problems that were
measured both ways (152 SMs)."""
import ctypes

import pytest

import native

HELPER = """
#include "fwi_internal.h"
#include "fwi_resident.h"
namespace {
fwi::Lay2D layout(int nz, int nx, int P)
{
    fwi::Lay2D L{};
    L.nz = nz, L.nx = nx, L.P = P, L.nzp = nz + 2 * P, L.nxp = nx + 2 * P;
    return L;
}
}
extern "C" int backward_rows(int nz, int nx, int P, int ns)
{
    return fwi::make_tiling(layout(nz, nx, P), ns, fwi::STEP_BWD).tz;
}
// shots in flight, rows per thread, row groups, float4 columns, groups of warps
extern "C" void tiling(int nz, int nx, int P, int ns, int kind, int *out)
{
    const fwi::ResTile t = fwi::res_plan(layout(nz, nx, P), ns, (fwi::ResKind)kind);
    out[0] = t.s, out[1] = t.th / t.g, out[2] = t.g, out[3] = t.w4, out[4] = t.accs / t.sets;
}
// whether the resident loop is expected to be faster than the streaming steps
extern "C" int resident(int nz, int nx, int P, int ns, int kind, int steps, int band)
{
    const fwi::Lay2D L = layout(nz, nx, P), *l = &L;
    const fwi::ResTile t = fwi::res_plan(L, ns, (fwi::ResKind)kind);
    return t.ok && fwi::res_level_us(L, t, (fwi::ResKind)kind, band) <
                       fwi::step_level_us(1, &l, &ns, (fwi::StepKind)steps, band);
}
"""


@pytest.fixture(scope="module")
def helper(tmp_path_factory):
    return native.compile_helper(HELPER, tmp_path_factory.mktemp("choices"))


# nz, nx, sponge, shots, us per level of the backward step on 64 x 16 and 64 x 8 tiles:
# one round of CTAs or many, half blocks of shots left over, one to 92 shots
BACKWARD = [(150, 460, 20, 48, 34.1, 40.7), (94, 299, 20, 92, 31.5, 39.9), (95, 1039, 20, 27, 29.9, 36.7),
            (387, 136, 20, 54, 31.2, 37.1), (383, 202, 20, 45, 34.1, 38.4), (300, 1000, 20, 32, 60.2, 66.5),
            (314, 661, 15, 54, 66.0, 72.3), (300, 1000, 20, 48, 82.9, 92.1), (71, 333, 20, 90, 27.7, 38.3),
            (400, 1200, 20, 64, 150.3, 170.5), (400, 1200, 20, 2, 8.4, 11.7),
            (100, 200, 20, 64, 25.7, 22.7), (300, 1000, 20, 1, 5.6, 4.8), (300, 1000, 20, 2, 8.3, 7.4),
            (300, 1000, 20, 12, 29.7, 27.5), (37, 1109, 20, 19, 25.0, 22.1), (162, 867, 20, 7, 22.0, 17.9),
            (342, 107, 15, 42, 27.6, 24.5), (224, 947, 20, 8, 23.7, 20.5)]


@pytest.mark.parametrize("nz,nx,P,ns,us16,us8", BACKWARD)
def test_backward_tiles_are_the_faster_ones(helper, nz, nx, P, ns, us16, us8):
    assert helper.backward_rows(nz, nx, P, ns) == (16 if us16 < us8 else 8)


# nz, nx, sponge, shots, us per level of the streaming steps and of the resident loop
# (passes of a gradient keep or read the checkpoint), by pass: its resident kind, steps
# and whether it has the checkpoint
PASSES = {"plain": (0, 0, 0), "save": (0, 0, 1), "illum": (1, 0, 0), "gradient": (1, 0, 1), "adjoint": (3, 2, 1)}
LOOPS = [("plain", 400, 1200, 20, 32, 50.3, 57.5), ("plain", 250, 700, 20, 48, 34.7, 37.7),
         ("plain", 400, 1200, 20, 64, 88.1, 111.6), ("plain", 300, 1000, 20, 24, 28.2, 25.1),
         ("plain", 300, 1000, 20, 12, 17.4, 12.2), ("plain", 150, 460, 20, 80, 27.8, 19.8),
         ("plain", 100, 200, 20, 4, 6.1, 2.6), ("plain", 500, 1500, 20, 16, 39.8, 44.8),
         ("save", 400, 1200, 20, 8, 14.8, 19.7), ("save", 400, 1200, 20, 32, 57.2, 84.4),
         ("save", 300, 1001, 20, 48, 62.0, 80.5), ("save", 345, 446, 20, 39, 29.4, 36.2),
         ("save", 300, 1000, 20, 96, 111.1, 133.9), ("save", 200, 400, 20, 16, 12.9, 6.2),
         ("illum", 200, 400, 20, 16, 12.0, 6.4),
         ("gradient", 400, 1200, 20, 16, 29.9, 43.5), ("gradient", 400, 1200, 20, 8, 14.9, 20.5),
         ("gradient", 95, 1039, 20, 27, 20.3, 23.1), ("gradient", 158, 677, 20, 32, 23.3, 26.5),
         ("gradient", 300, 1000, 20, 6, 11.2, 7.8), ("gradient", 100, 200, 20, 64, 14.5, 8.8),
         ("adjoint", 100, 200, 20, 64, 22.4, 18.1), ("adjoint", 37, 1109, 20, 19, 22.1, 18.7),
         ("adjoint", 150, 460, 20, 12, 19.4, 12.1), ("adjoint", 100, 200, 20, 16, 17.8, 8.6),
         ("adjoint", 300, 1000, 20, 6, 16.7, 21.9), ("adjoint", 400, 1200, 20, 4, 13.3, 18.4),
         ("adjoint", 332, 898, 15, 3, 9.3, 10.5)]


@pytest.mark.parametrize("name,nz,nx,P,ns,steps,loop", LOOPS)
def test_the_faster_of_steps_and_resident_loop_is_taken(helper, name, nz, nx, P, ns, steps, loop):
    assert bool(helper.resident(nz, nx, P, ns, *PASSES[name])) == (loop < steps)


@pytest.mark.parametrize("kind,rows", [(0, (3, 4)), (1, (3, 4)), (2, (3, 4)), (3, (2, 3))])
def test_two_groups_of_warps_from_three_shots_in_flight(helper, kind, rows):
    """Where the tiling has a variant of two groups (6 warps each, these rows per
    thread), the choice between one and two is by the shots in flight, not by the
    rounding of equal costs."""
    seen = set()
    for nz, nx in ((37, 83), (37, 100), (60, 120), (100, 200), (120, 100), (150, 460), (200, 400), (300, 1000)):
        for P in (5, 20):
            for ns in (1, 2, 3, 4, 7, 12, 16, 32, 64, 97):
                o = (ctypes.c_int * 5)()
                helper.tiling(nz, nx, P, ns, kind, o)
                s, r, g, w4, groups = o
                two = s >= 3 and r in rows and g * w4 <= 6 * 32
                assert groups == (2 if two else 1), (nz, nx, P, ns, list(o))
                seen.add(two)
    assert seen == {True, False}
