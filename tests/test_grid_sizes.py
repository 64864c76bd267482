"""The reduction workspace of a Lanczos run holds the partials of every kernel that reduces into it, on every lattice
that seedcg_create accepts (12 V < 2^31): its counters lie directly behind the partials.  The grids and the size are
host code (csrc/grids.h), compiled here with the host compiler."""
import ctypes
import os
import subprocess

import pytest

from paper_0901_3512_gb300.build import CSRC

WRAP = r'''
#include "grids.h"
using namespace seedcg;
extern "C" {
long partials(long n, int nrhs, int fp64) { return (long)lz_partial_doubles(n, nrhs, fp64 != 0); }
long site_grid(int sites) { return site_blocks_lz(sites); }
long half_grid(int vol) { return site_blocks(vol / 2); }
long tile_grid(int sites) { return fix_tiles(sites); }
long entry_grid(long n) { return entry_blocks(n, 1); }
long vec_grid(long n, int w) { return vec_blocks(n, w); }
long red_grid(long n) { return red_blocks(n); }
}
'''


@pytest.fixture(scope="module")
def grids(tmp_path_factory):
    d = tmp_path_factory.mktemp("grids")
    (d / "g.cpp").write_text(WRAP)
    so = str(d / "g.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(d / "g.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    for f in ("partials", "site_grid", "half_grid", "tile_grid", "entry_grid", "vec_grid", "red_grid"):
        getattr(lib, f).restype = ctypes.c_long
    lib.partials.argtypes = [ctypes.c_long, ctypes.c_int, ctypes.c_int]
    lib.entry_grid.argtypes = lib.red_grid.argtypes = [ctypes.c_long]
    lib.vec_grid.argtypes = [ctypes.c_long, ctypes.c_int]
    return lib


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (16, 16, 16, 32), (32, 32, 32, 64), (48, 48, 48, 64), (64, 64, 64, 128),
                                  (72, 72, 72, 96), (96, 96, 96, 192), (114, 114, 114, 120)])
@pytest.mark.parametrize("nrhs", [1, 2, 12, 256])
def test_partials_fit(grids, dims, nrhs):
    vol = dims[0] * dims[1] * dims[2] * dims[3]
    assert 12 * vol < 2 ** 31
    for sites in (vol, vol // 2):      # full lattices, and half vectors of the even-odd system
        n = 12 * sites
        rb = grids.red_grid(n)
        common = max(16 * rb, grids.vec_grid(n, 4), grids.vec_grid(n, 2), grids.vec_grid(n, 1))
        assert grids.partials(n, nrhs, 0) >= max(common, grids.site_grid(sites))
        assert grids.partials(n, nrhs, 1) >= max(common, grids.tile_grid(sites), grids.entry_grid(n))
    assert grids.partials(6 * vol, nrhs, 0) >= grids.half_grid(vol)
    assert grids.partials(12 * 16 ** 3 * 32, nrhs, 1) == max(4096, 1216 * (nrhs + 2)) * 64   # as it always was
