"""Lattices with solid cells whose steps change between tiles and the marching kernel: beyond
3 M cells those with a force field, drag or a moving void fraction march. Both kernels give the
same populations, whichever ran before."""
import numpy as np
import pytest
from test_gpu_tile import _times_out

pytestmark = pytest.mark.gpu


def _lattice(P, nx, ny, storage, kernel=0):
    phi = np.full((ny, nx), 0.7, dtype=np.float32)
    phi += (0.2 * np.sin(np.arange(nx) / 50.0)).astype(np.float32)
    phi[40:60, 100:130] = 0.0
    lat = P.Lattice(nx, ny, 0.7, bc_y="bounceback", storage=storage, kernel=kernel)
    lat.set_solid_cells()
    lat.set_void_fraction(phi)
    lat.set_body_force(1e-6, 0.0)
    lat.init_fields(np.ones((ny, nx)), np.zeros((ny, nx)), np.zeros((ny, nx)))
    return lat, phi


@pytest.mark.parametrize("nx,tiles", [(2000, True), (2001, False)])
def test_fields_march_beyond_three_million_cells(nx, tiles):
    import paper_2409_02964_gb300 as P
    lat, _ = _lattice(P, nx, 1500, "fp32")
    lat.set_drag(1e-3, 0.05)
    assert _times_out(lat) is not tiles
    lat.close()


@pytest.mark.parametrize("storage", ["fp32", "bf16"])
def test_populations_do_not_depend_on_the_kernel(storage):
    import torch
    import paper_2409_02964_gb300 as P
    nx, ny = 2001, 1500
    fb = (1e-5 * np.random.default_rng(1).normal(size=(2, ny, nx))).astype(np.float32)
    got = []
    for kernel in (0, 5):
        lat, phi = _lattice(P, nx, ny, storage, kernel)
        lat.step(19)                                   # tiles (a replayed graph and a remainder)
        lat.set_body_force(1e-6, 0.0, fb)
        lat.step(3)                                    # marching
        lat.set_body_force(1e-6, 0.0)
        lat.set_void_fraction(phi, (phi * np.float32(0.999)).astype(np.float32))
        lat.step(2)                                    # marching, then tiles
        got.append(lat.get_populations())
        lat.sync()
        lat.close()
    assert bool(torch.isfinite(got[0]).all()) and torch.equal(got[0], got[1])
