"""The division of a deterministic FP32 run over CTAs, which decides which lanes' currents are summed
before the fixed-point word, is the same on every device, and without one (where the division of the
other runs, which follows the device, is one CTA per tile)."""
import ctypes
import subprocess

import pytest

from paper_1909_09613_gb300 import _build

SOURCE = r"""
#include "pic_launch.h"
extern "C" unsigned ctas(int det, long long tiles, long long particles)
{
    static pic::RunDev rd;
    rd.det = det;
    rd.ntiles = tiles;
    rd.nsp = 1;
    rd.sp[0].n = particles;
    return pic::tile_ctas(rd);
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    src, so = str(d / "split.cu"), str(d / "split.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([_build._nvcc(), "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler",
                    "-fPIC", "-shared", "-I", _build.CSRC, "-I", _build.INCLUDE, src, "-o", so],
                   check=True, capture_output=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("tiles,particles,want", [
    (1, 1, 1), (8, 4096, 8 * 16), (64, 64 * 600, 64 * 4), (64, 64 * 8192, 304), (256, 1 << 20, 304),
    (304, 1 << 20, 304), (700, 1 << 21, 912), (4096, 1 << 26, 4096)])
def test_deterministic_division(host, tiles, particles, want):
    n = ctypes.c_longlong
    assert host.ctas(1, n(tiles), n(particles)) == want
