"""The adjoint kernels where their row and memory rules change: lattices of one to three
rows or columns (both walls next to a cell, wraps onto itself) against the autograd oracle,
and whole segments on the device with the checkpoints on the host against everything on the
device. Bounds as in test_gpu_adjoint.py."""
import numpy as np
import pytest

from test_gpu_adjoint import _oracle, _phi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc_y", ["bounceback", "periodic"])
@pytest.mark.parametrize("nx,ny", [(3, 3), (5, 1), (7, 2), (1, 6), (2, 5), (67, 3)])
def test_thin_lattices_match_autograd_oracle(nx, ny, bc_y):
    import paper_2409_02964_gb300 as P
    ch = P.Channel(nx=nx, ny=ny, tau=0.7, s_q=1.3, bc_y=bc_y, gx=2e-5, gy=-5e-6, nsteps=9, avg_steps=4,
                   checkpoint_every=3)
    phi = _phi(nx, ny, nx + ny)
    J, g, _ = P.outlet_momentum(phi, ch)
    Jo, go = _oracle(ch, phi)
    assert abs(J - Jo) <= 1e-10 * max(abs(Jo), 1e-12)
    assert np.abs(g.cpu().numpy() - go).max() <= 1e-8 * np.abs(go).max()


def test_whole_segments_with_host_checkpoints():
    """512^2: 30 states take 566 MB (not kept whole), a segment of 10 does (189 MB)."""
    import paper_2409_02964_gb300 as P
    phi = _phi(512, 512, 3)
    base = dict(nx=512, ny=512, nsteps=30, avg_steps=7, checkpoint_every=10)
    J, g, st = P.outlet_momentum(phi, P.Channel(**base))
    Jd, gd, std = P.outlet_momentum(phi, P.Channel(**base, dense_segments=True))
    assert st["host_bytes"] == 3 * 9 * 512 * 512 * 8 and std["host_bytes"] == 0
    assert J == Jd and (g == gd).all()
