"""The rules that pick a 2-D lattice's step kernel and its rows per CTA (csrc/step_rules.h),
evaluated on the host: row blocks lie on the grid's y axis, at most 65535 of them, whatever
the lattice's height."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2409_02964_gb300", "csrc")
GRID_Y = 65535
SHIM = r"""
#include "step_rules.h"
extern "C" void rules(int nx, int ny, int gridx, int resident, int nsm, int kernel, int sbytes, int strip_rows,
                      int solid, int auto_kernel, int wall, int* out) {
    const lbmv::StepShape s{nx,         ny,         gridx,            resident, nsm, kernel, sbytes,
                            strip_rows, solid != 0, auto_kernel != 0, wall != 0};
    out[0] = lbmv::strip_height(s);
    const lbmv::TileShape t = lbmv::tile_shape(s);
    out[1] = sbytes == 8 ? lbmv::tile64_rows(s, out[0]) : t.rows;
    out[2] = t.big;
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "shim.cpp").write_text(SHIM)
    lib = str(d / "librules.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + CSRC, "-o", lib, str(d / "shim.cpp")],
                   check=True)
    fn = ctypes.CDLL(lib).rules

    def call(nx, ny, sbytes, solid=False, strip_rows=0, kernel=0, wall=False):
        k = kernel or (1 if sbytes == 8 else 5)
        cols, per_sm = (60, 8) if k == 5 else (124, 2)
        out = (ctypes.c_int * 3)()
        fn(nx, ny, -(-nx // cols), 152 * per_sm, 152, k, sbytes, strip_rows, int(solid), int(kernel == 0), int(wall),
           out)
        return tuple(out)

    return call


# the tile kernels' heights end at 8 * 65535 rows, march64_us's at 128 * 65535
HEIGHTS = [1, 3, 65535, 65536, 524279, 524280, 524281, 530000, 600000, 8388480, 8388481, 9700000, 2 ** 31 - 1]


@pytest.mark.parametrize("solid", [False, True])
@pytest.mark.parametrize("sbytes", [2, 4, 8])
@pytest.mark.parametrize("nx", [1, 7, 8, 16, 28, 84, 250])
def test_row_blocks_fit_the_grid(rules, nx, sbytes, solid):
    for ny in HEIGHTS:
        if nx * ny > 2 ** 31:
            continue
        rows, tile, _ = rules(nx, ny, sbytes, solid)
        assert 1 <= rows <= ny and -(-ny // rows) <= GRID_Y, (ny, rows)
        assert tile == 0 or -(-ny // tile) <= GRID_Y, (ny, tile)


@pytest.mark.parametrize("nx,sbytes,solid", [(28, 8, False), (7, 4, True), (7, 2, True)])
def test_tiles_up_to_the_last_height_that_fits(rules, nx, sbytes, solid):
    """Narrow lattices that tiles suit keep them up to 8 * 65535 rows and march beyond."""
    assert rules(nx, 8 * GRID_Y, sbytes, solid)[1] == 8
    assert rules(nx, 8 * GRID_Y + 1, sbytes, solid)[1] == 0


@pytest.mark.parametrize("nx,ny", [(80000, 100), (100000, 30), (100000, 600), (150000, 200), (300000, 100), (72961, 67),
                                   (4096, 4096), (1200, 900), (800, 800)])
def test_wide_lattices_do_not_leave_a_wave_to_a_few_strips(rules, nx, ny):
    """By whole waves of H + 6 rows the height is no worse than five waves of 16 rows and more."""
    cols, resident = -(-nx // 60), 152 * 8

    def row_times(H):
        return -(-(cols * -(-ny // H)) // resident) * (H + 6)

    generic = min(ny, max(16, -(-ny // max(1, -(-5 * resident // cols)))))
    assert row_times(rules(nx, ny, 4, kernel=5)[0]) <= row_times(generic)


@pytest.mark.parametrize("wall", [False, True])
@pytest.mark.parametrize("nx,ny,rows", [(30000, 5, 5), (36000, 8, 8), (60000, 20, 16)])
def test_low_wide_fp64_lattices_march(rules, nx, ny, rows, wall):
    assert rules(nx, ny, 8, wall=wall)[:2] == (rows, 0)
