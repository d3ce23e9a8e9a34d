"""FP64 lattices with solid cells: the strips of a lattice that leaves the kernel open (few
rows on small lattices) against those of one that asks for kernel 1 (16 rows and more). Both
put every cell through the same operations, so the populations are equal. Strips of one to a
few rows meet the y walls, the moving wall row and solid cells on their first and last rows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wall", ["periodic", "bounceback", "moving"])
@pytest.mark.parametrize("nx,ny", [(1, 4), (5, 3), (39, 17), (130, 90), (251, 163), (400, 300)])
def test_short_strips_equal_tall_ones(nx, ny, wall):
    import torch
    import paper_2409_02964_gb300 as P
    rng = np.random.default_rng(nx + ny)
    phi = rng.uniform(0.5, 1.0, size=(ny, nx))
    solid = rng.uniform(size=phi.shape) < 0.08
    solid[ny // 2, :nx // 2] = True
    if wall == "moving":
        solid[-3:] = False                      # as the moving wall asks: fluid below it
    phi[solid] = 0.0
    u = 0.01 * rng.normal(size=(2, ny, nx)) * ~solid
    got = []
    for kernel in (0, 1):
        lat = P.Lattice(nx, ny, 0.7, s_e=1.2, s_eps=1.2, s_q=1.2, bc_y="periodic" if wall == "periodic" else "bounceback",
                        storage="fp64", kernel=kernel)
        lat.set_solid_cells()
        if wall == "moving":
            lat.set_moving_wall(1e-3, 0.0)
        lat.set_void_fraction(phi)
        lat.set_body_force(1e-5, -2e-5)
        lat.init_fields(np.ones((ny, nx)), u[0], u[1])
        lat.step(9)
        got.append(lat.get_populations())
        lat.sync()
        lat.close()
    assert bool(torch.isfinite(got[0]).all()) and torch.equal(got[0], got[1])


@pytest.mark.parametrize("storage,nx,ny,tiles", [("fp32", 2250, 2000, True), ("fp32", 2251, 2000, False),
                                                 ("fp16", 2000, 2000, True), ("fp16", 2001, 2000, False)])
def test_large_lattices_with_solids_march(storage, nx, ny, tiles):
    """On both sides of the line between tiles and the marching kernel: which of them runs
    (only the marching kernel waits for staged rows, so only it can time out)."""
    import paper_2409_02964_gb300 as P
    phi = np.full((ny, nx), 0.7)
    phi[40:60, 100:130] = 0.0
    zero = np.zeros((ny, nx))
    lat = P.Lattice(nx, ny, 0.7, storage=storage)
    lat.set_solid_cells()
    lat.set_void_fraction(phi)
    lat.init_fields(np.ones((ny, nx)), zero, zero)
    lat.step(1)
    lat.sync()
    lat._L.lbm_vanse_set_row_wait_limit(lat._h, 0)
    lat.step(1)
    assert (lat._L.lbm_vanse_sync(lat._h) == -6) is not tiles     # LBM_ERR_TIMEOUT
    lat.close()
