"""Choices by problem size where nothing was autotuned, against problems that were
measured both ways (152 SMs)."""
import pytest

import native

HELPER = """
#include "fwi_internal.h"
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
