"""Each instance of the tile step kernel against the one-warp marching kernel (kernel 5), bit
for bit: both put a cell through the same phase functions and round stored values by the same
random bits. The heights follow from the device's SM count, so that every class of the
dispatch (tile_shape in csrc/step_rules.h) is met: four rows a CTA in the small and in the
12-warp instance, eight rows."""
import pytest
from test_gpu_tile import _pair

pytestmark = pytest.mark.gpu

NX = 301      # six CTAs wide, the last one narrow


@pytest.mark.parametrize("extra", ["plain", "moving", "drag", "solid"])
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("wall", [False, True])
@pytest.mark.parametrize("per_sm,rows", [(1.5, 4), (2.5, 4), (3.5, 8)])
def test_instances_equal_the_marching_kernel(per_sm, rows, wall, storage, extra):
    import torch
    import paper_2409_02964_gb300 as P
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    ny = 4 * round(per_sm * nsm / 6) - 1
    ctas = 6 * -(-ny // 4)
    assert ctas <= 2 * nsm if per_sm == 1.5 else (2 * nsm < ctas <= 3 * nsm if rows == 4 else ctas > 3 * nsm)
    (tile, march), _ = _pair(P, NX, ny, wall, storage, extra)
    for n in (1, 2, 35):       # single steps, then a replayed graph and a remainder
        tile.step(n)
        march.step(n)
        a, b = tile.get_populations(), march.get_populations()
        assert bool(torch.isfinite(a).all()) and torch.equal(a, b)
    tile.sync()
    tile.close()
    march.close()


@pytest.mark.parametrize("extra", ["plain", "moving", "solid"])
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_edges_of_tiles_equal_the_marching_kernel(storage, extra):
    import torch
    import paper_2409_02964_gb300 as P
    for nx, ny in [(1, 1), (2, 3), (3, 2), (60, 8), (61, 9), (57, 4), (121, 33)]:
        for wall in (False, True):
            (tile, march), _ = _pair(P, nx, ny, wall, storage, extra, seed=nx + ny)
            for n in (1, 36):
                tile.step(n)
                march.step(n)
                assert torch.equal(tile.get_populations(), march.get_populations()), (nx, ny, wall)
            tile.close()
            march.close()
