"""A float32 body-force field equals the same field handed over as float64: FP32 lattices hold
it in float either way, FP64 ones widen it exactly. From the device and the host, from a
strided view (copied first), and refused with the wrong size."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("where", ["device", "host", "strided"])
def test_float_force_equals_double_force(where, storage):
    import torch
    import paper_2409_02964_gb300 as P
    nx, ny = 37, 21
    rng = np.random.default_rng(3)
    fb = (1e-4 * rng.normal(size=(2, ny, nx))).astype(np.float32)
    phi = rng.uniform(0.5, 1.0, size=(ny, nx)).astype(np.float32)
    if where == "strided":
        wide = torch.zeros((2, ny, 2 * nx), dtype=torch.float32, device="cuda")
        wide[:, :, ::2] = torch.from_numpy(fb).cuda()
        single = wide[:, :, ::2]
    else:
        single = torch.from_numpy(fb).cuda() if where == "device" else fb
    got = []
    for field in (single, fb.astype(np.float64)):
        lat = P.Lattice(nx, ny, 0.8, storage=storage)
        lat.set_void_fraction(phi)
        lat.set_body_force(0.0, 0.0, field)
        lat.init_fields(np.ones((ny, nx)), np.zeros((ny, nx)), np.zeros((ny, nx)))
        lat.step(3)
        got.append(lat.get_populations())
        with pytest.raises(ValueError):
            lat.set_body_force(0.0, 0.0, field[0])
        lat.close()
    assert bool(torch.isfinite(got[0]).all()) and torch.equal(got[0], got[1])
