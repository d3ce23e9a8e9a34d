"""Strips of the one-warp kernel where force rows are staged as well: they take shared memory,
so fewer CTAs are resident (FP32: 7 per SM instead of 8), and heights picked for more would
leave a second wave nearly empty. Values do not depend on the height."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SMEM_SM, RESERVED, MAX_CTAS = 228 * 1024, 1024, 8     # bytes of an SM, of each CTA; CTAs by registers


@pytest.mark.parametrize("storage", ["fp32", "bf16"])
@pytest.mark.parametrize("nx,ny", [(1000, 700), (1200, 900)])
def test_one_wave_of_strips_with_and_without_a_force_field(storage, nx, ny):
    import torch
    import paper_2409_02964_gb300 as P
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(3)
    phi = rng.uniform(0.5, 1.0, size=(ny, nx)).astype(np.float32)
    phin = (phi * np.float32(0.999)).astype(np.float32)
    fb = (1e-5 * rng.normal(size=(2, ny, nx))).astype(np.float32)
    u = 0.01 * rng.normal(size=(2, ny, nx))
    got, shapes = [], []
    for strip_rows in (0, 16):
        lat = P.Lattice(nx, ny, 0.7, s_e=1.2, bc_y="bounceback", storage=storage, kernel=5, strip_rows=strip_rows)
        lat.set_void_fraction(phi, phin)
        lat.set_body_force(1e-6, 0.0, fb)
        lat.init_fields(np.ones((ny, nx)), u[0], u[1])
        for k in range(3):
            shapes.append((strip_rows, lat.launch_shape()))
            lat.step(1)
            if k == 1:
                lat.set_body_force(1e-6, 0.0)
        got.append(lat.get_populations())
        lat.sync()
        lat.close()
    assert torch.equal(got[0], got[1])
    smem = [s["smem_bytes"] for r, s in shapes if r == 0]
    assert smem[0] > smem[1] > smem[2]              # phi, phi(t+1) and force; phi and force; phi
    for rows, s in shapes:
        if rows == 0:
            resident = nsm * min(MAX_CTAS, SMEM_SM // (s["smem_bytes"] + RESERVED))
            assert s["grid_x"] * s["grid_y"] <= resident, s
        else:
            assert s["rows"] == 16
