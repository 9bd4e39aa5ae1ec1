"""The rules that size the raster's work units (vs_units.h, host code without
CUDA): a launch has units for its warps, but not many more than they need, for
one large item as for many small ones, and no unit is coarser than was asked
for."""

import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_02482_gb300", "csrc")
SHIM = """
#include "vs_units.h"
extern "C" void raster(long long tris, int asked, int n, int warps, int* out) {
  const vsu::RasterUnits u = vsu::raster_units(tris, asked, n, warps);
  out[0] = u.tris;
  out[1] = u.lg;
}
extern "C" int shell(int unit, int tris, long long pixels, long long batch_tris, int n, int warps) {
  return vsu::shell_unit(unit, tris, pixels, batch_tris, n, warps);
}
"""
WARPS = 152 * 24


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("units")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    lib.raster.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    lib.shell.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    return lib


def units(lib, n, k, tris, pixels, asked=256):
    """(triangles per unit, lg, units of the launch) of n items of k shells."""
    out = (ctypes.c_int * 2)()
    lib.raster(n * k * tris, asked, n, WARPS, out)
    unit = lib.shell(out[0], tris, pixels, n * k * tris, n, WARPS)
    return unit, out[1], n * k * -(-tris // unit) << out[1]


@pytest.mark.parametrize("n,k,tris,side", [(64, 3, 1936, 64), (256, 3, 900, 32), (64, 5, 9800, 128), (16, 5, 19800, 32),
                                           (12, 5, 9800, 200)])
def test_many_small_items_share_the_warps(lib, n, k, tris, side):
    # every warp finds a unit, and the units' 5 ns stay below twice what one
    # each would cost, or the asked size is kept
    unit, _, total = units(lib, n, k, tris, side * side)
    assert total >= WARPS // 2
    assert unit == 256 or total <= 2 * WARPS * 1.05


@pytest.mark.parametrize("asked", [32, 256, 2048])
@pytest.mark.parametrize("n,k,tris,pixels", [(1, 1, 1, 1), (1, 16, (1 << 27) - 1, 1 << 28), (2, 1, 1, 1 << 28),
                                             (8, 9, 484, 1920 * 1080), (16, 5, 19800, 100000), (24, 7, 199396, 640000),
                                             (4, 9, 2000000, 3840 * 2160), (4096, 3, 20, 64)])
def test_units_are_powers_of_two_within_their_range(lib, n, k, tris, pixels, asked):
    unit, lg, total = units(lib, n, k, tris, pixels, asked)
    assert unit & (unit - 1) == 0 and 1 <= unit <= asked
    assert unit >= (8 if n > 1 else 1) and (lg == 0 or (n == 1 and unit == 1)) and 0 <= lg <= 6
    # no unit covers more pixels than the bound unless it is at its smallest
    assert unit <= 8 or unit * pixels <= 2048 * tris
    assert total < 1 << 31


def test_a_strip_with_few_triangles_keeps_several_units_per_warp(lib):
    unit, _, total = units(lib, 16, 5, 19800, 100 * 1000)
    assert unit == 64 and total > 4 * WARPS
