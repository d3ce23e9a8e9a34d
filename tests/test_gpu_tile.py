"""The tile step kernel (vanse_tile.cuh, the automatic choice for small lattices and for
solid cells) against the one-warp marching kernel (kernel 5) from the same fields.

Both collide the stored deviations in FP32 with the same phase functions. Bounds (D =
max |f - f^rest|): each kernel stays within 8 * 2^-24 D per step of the oracle
(test_gpu_parity.py), so the two differ by at most 16 * 2^-24 D per step; FP16 / BF16 add
two spacings of the stored deviation per step, 2 * 2^-11 D and 2 * 2^-8 D."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ULP = {"fp32": 16 * 2.0 ** -24, "fp16": 16 * 2.0 ** -24 + 2 * 2.0 ** -11, "bf16": 16 * 2.0 ** -24 + 2 * 2.0 ** -8}
# tiles are 60 columns by 4 or 8 rows; ghost images wrap columns 0..2 and nx-3..nx-1
SIZES = [(1, 1), (2, 3), (3, 2), (60, 8), (61, 9), (57, 4), (121, 33), (250, 70), (500, 331)]


def _pair(P, nx, ny, wall, storage, extra, seed=7):
    rng = np.random.default_rng(seed)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    phi = f32(rng.uniform(0.5, 1.0, size=(ny, nx)))
    if extra == "solid":
        phi[rng.uniform(size=phi.shape) < 0.08] = 0.0
    fluid = phi > 0
    u = [f32(0.01 * rng.normal(size=(ny, nx))) * fluid for _ in range(2)]
    fb = f32(1e-5 * rng.normal(size=(2, ny, nx)))
    phin = np.where(fluid, f32(np.clip(phi + 0.005 * rng.normal(size=phi.shape), 0.4, 1.0)), 0.0)
    out = []
    for kernel in (0, 5):
        lat = P.Lattice(nx, ny, 0.7, s_e=1.2, s_eps=1.2, s_q=1.2, bc_y="bounceback" if wall else "periodic",
                        storage=storage, kernel=kernel)
        if extra == "solid":
            lat.set_solid_cells()
        if extra == "drag":
            lat.set_drag(1e-2, 0.1, 1e-3, 0.0)
        moving = extra in ("moving", "solid")
        lat.set_void_fraction(phi, phin if moving else None)
        lat.set_body_force(1e-5, -2e-5, fb if extra == "moving" else None)
        lat.init_fields(np.ones((ny, nx)), u[0], u[1])
        out.append(lat)
    return out, phin if moving else phi


@pytest.mark.parametrize("extra", ["plain", "moving", "drag", "solid"])
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("wall", [False, True])
def test_tile_kernel_matches_the_marching_kernel(wall, storage, extra):
    import paper_2409_02964_gb300 as P
    for nx, ny in SIZES:
        (tile, march), phi = _pair(P, nx, ny, wall, storage, extra)
        done = 0
        for n in (1, 2, 35):       # single steps, then a replayed graph and a remainder
            tile.step(n)
            march.step(n)
            done += n
            a = tile.get_populations().cpu().numpy()
            b = march.get_populations().cpu().numpy()
            rest = np.stack([phi - 5 * 0.5 / 9] + [np.full_like(phi, 0.5 / 9)] * 4 + [np.full_like(phi, 0.5 / 36)] * 4)
            D = np.abs(np.where(phi > 0, b - rest, 0.0)).max()
            assert np.isfinite(a).all()
            assert np.abs(a - b).max() <= done * ULP[storage] * D, (nx, ny, done)
        tile.sync()
        tile.close()
        march.close()


def _times_out(lat):
    """Whether the lattice's step waits for staged rows (the marching kernel does, tiles do not)."""
    lat.step(1)
    lat._L.lbm_vanse_set_row_wait_limit(lat._h, 0)
    lat.step(1)
    return lat._L.lbm_vanse_sync(lat._h) == -6     # LBM_ERR_TIMEOUT


@pytest.mark.parametrize("n,solid,tiles", [(64, False, True), (512, False, True), (1024, False, False), (1024, True, True)])
def test_small_lattices_and_solid_cells_run_as_tiles(n, solid, tiles):
    import paper_2409_02964_gb300 as P
    lat = P.Lattice(n, n, 0.7)
    if solid:
        lat.set_solid_cells()
    lat.set_void_fraction(np.full((n, n), 0.7))
    lat.init_fields(np.ones((n, n)), np.zeros((n, n)), np.zeros((n, n)))
    assert _times_out(lat) is not tiles
    lat.close()


@pytest.mark.parametrize("extra", ["plain", "moving", "drag"])
@pytest.mark.parametrize("wall", [False, True])
def test_fp64_tiles_match_the_marching_kernel(wall, extra):
    """Tiles of 28 columns by 1 to 8 rows against kernel 1: the same phases in FP64, each
    within 1e-12 D of the oracle over a few steps (test_gpu_parity.py)."""
    import paper_2409_02964_gb300 as P
    for nx, ny in [(1, 1), (2, 3), (28, 2), (29, 9), (57, 4), (121, 33), (250, 70), (400, 301)]:
        rng = np.random.default_rng(nx + ny)
        phi = rng.uniform(0.5, 1.0, size=(ny, nx))
        u = 0.01 * rng.normal(size=(2, ny, nx))
        fb = 1e-5 * rng.normal(size=(2, ny, nx))
        phin = np.clip(phi + 0.005 * rng.normal(size=phi.shape), 0.4, 1.0)
        out = []
        for kernel in (0, 1):
            lat = P.Lattice(nx, ny, 0.7, s_e=1.2, s_eps=1.2, s_q=1.2, bc_y="bounceback" if wall else "periodic",
                            storage="fp64", kernel=kernel)
            if extra == "drag":
                lat.set_drag(1e-2, 0.1, 1e-3, 0.0)
            lat.set_void_fraction(phi, phin if extra == "moving" else None)
            lat.set_body_force(1e-5, -2e-5, fb if extra == "moving" else None)
            lat.init_fields(np.ones((ny, nx)), u[0], u[1])
            lat.step(1)
            lat.step(36)
            out.append(lat.get_populations().cpu().numpy())
            lat.close()
        D = 0.05
        assert np.isfinite(out[0]).all() and np.abs(out[0] - out[1]).max() <= 2e-12 * D, (nx, ny)
