"""The tolerance of the resolve's division-free rounding (map_eps): it belongs to
the back-projection, so neither the view's size nor the forward map, which the
splat applies with divisions, has a part in it."""
import os
import shutil
import subprocess

import pytest

from paper_2007_00558_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "fvv_internal.h"
// W H Wv Hv z_min, then M8..M11 and N8..N11
int main(int, char** a)
{
    fvv::CamGeom g{};
    for (int i = 0; i < 4; ++i) g.M[8 + i] = std::strtof(a[6 + i], nullptr), g.N[8 + i] = std::strtof(a[10 + i], nullptr);
    std::printf("%.9g\n", double(fvv::map_eps(g, std::atoi(a[1]), std::atoi(a[2]), std::atoi(a[3]), std::atoi(a[4]),
                                              std::strtof(a[5], nullptr))));
}
"""


@pytest.fixture(scope="module")
def eps(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("eps")
    (d / "eps.cpp").write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(build.cuda_libdir()), "include")
    subprocess.check_call([gxx, "-std=c++17", "-O1", "-I", build.CSRC, "-I", build.INCLUDE, "-I", cuda, "-o",
                           str(d / "eps"), str(d / "eps.cpp")])
    return lambda *a: float(subprocess.check_output([str(d / "eps")] + ["%.9g" % x for x in a]))


PLAIN = (0.0, 0.0, 1.0, 0.0)
TINY = (0.0, 1e-23, 1.0, 0.0)                     # below 2^-70: the reciprocal may leave the normal numbers


@pytest.mark.parametrize("W,H,bits", [(320, 240, 9), (1280, 720, 11), (246, 154, 8)])
@pytest.mark.parametrize("Wv,Hv", [(64, 48), (1298, 697), (5000, 3000)])
def test_the_tolerance_is_that_of_the_camera(eps, W, H, bits, Wv, Hv):
    want = 2.0 ** (bits - 25) + 2.0 ** -20        # half a last place of a camera's pixel, and the fraction's error
    assert eps(W, H, Wv, Hv, 1.0, *PLAIN, *PLAIN) == pytest.approx(want, rel=1e-6)


def test_only_the_back_projection_can_take_every_point_to_the_division(eps):
    assert eps(1280, 720, 1280, 720, 0.0, *TINY, *PLAIN) < 1e-3
    assert eps(1280, 720, 1280, 720, 0.0, *PLAIN, *TINY) == float("inf")
    assert eps(1280, 720, 1280, 720, 1.0, *PLAIN, *TINY) < 1e-3          # z_min keeps Z off zero
    assert eps(1 << 21, 720, 1280, 720, 1.0, *PLAIN, *PLAIN) == float("inf")
