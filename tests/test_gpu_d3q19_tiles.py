"""The marching kernels of the D3Q19 step at the edges of their work split: column tiles of
32 x 8 (FP32) and 32 x 4 (FP64) cells, chunks of 2 to 32 planes (test_gpu_d3q19.py covers
lattices inside one tile). Bounds as there: FP64 1e-13, FP32 2e-6 per step."""
import numpy as np
import pytest

from test_gpu_d3q19 import _case, _gpu, _params, _total_force

pytestmark = pytest.mark.gpu

SHAPES = [(32, 4, 1), (33, 9, 2), (31, 8, 40), (65, 17, 5), (64, 3, 33), (1, 1, 70)]


@pytest.mark.parametrize("storage", ["fp64", "fp32"])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("nx,ny,nz", SHAPES)
def test_populations_match_oracle_across_tiles(nx, ny, nz, walls, storage):
    import paper_2409_02964_gb300 as P
    from oracle import d3q19 as D
    c = _case(nx, ny, nz, seed=nx + 10 * ny + 100 * nz)
    lat = _gpu(P, nx, ny, nz, c, storage, walls)
    p = _params(nx, ny, nz, walls)
    f = D.init(p, c["rho"], c["u"], c["phi"], _total_force(c))
    f = D.step(p, f, c["phi"], c["phin"], _total_force(c))      # phi moves
    c2 = dict(c, phi=c["phin"], phin=None)
    f = D.step(p, f, c2["phi"], None, _total_force(c2))
    lat.step(2)
    g = lat.get_populations().cpu().numpy()
    assert np.abs(g - f).max() < (1e-13 if storage == "fp64" else 2 * 2e-6)
    lat.close()


@pytest.mark.parametrize("storage", ["fp64", "fp32"])
def test_rest_state_reads_back_exactly(storage):
    """Zero deviations (and a moving f_0) widen to the rest populations to the last bit."""
    import paper_2409_02964_gb300 as P
    nx, ny, nz = 35, 6, 5
    phi = np.full((nz, ny, nx), 0.75)
    lat = P.Lattice3D(nx, ny, nz, 0.8, storage=storage)
    lat.set_void_fraction(phi)
    lat.init_fields(np.ones(phi.shape), np.zeros((3,) + phi.shape))
    f = np.full((19, nz, ny, nx), 0.5 / 36)
    f[1:7] = 0.5 / 18
    f[0] = 0.75 - 2 * 0.5 / 3
    lat.set_populations(f)
    assert (lat.get_populations().cpu().numpy() == f).all()
    lat.close()
