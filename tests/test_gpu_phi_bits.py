"""The void-fraction check at the edges of what it tells apart: values outside [0, 1] are
refused, and a value that is zero in the lattice's compute type (for FP32 arithmetic every
double up to 2^-150, which rounds to even) is reported by the next sync as a solid cell."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

T150 = 2.0 ** -150
ABOVE = np.nextafter(T150, 1.0)
TINY = 5e-324


@pytest.mark.parametrize("storage,value,verdict", [
    ("fp32", 1.0, "ok"), ("fp32", 2.0 ** -149, "ok"), ("fp32", ABOVE, "ok"), ("fp32", T150, "zero"),
    ("fp32", 1e-300, "zero"), ("fp32", TINY, "zero"), ("fp32", 0.0, "zero"), ("fp32", -0.0, "zero"),
    ("fp64", TINY, "ok"), ("fp64", T150, "ok"), ("fp64", 0.0, "zero"), ("fp64", -0.0, "zero"),
    ("fp32", np.nextafter(1.0, 2.0), "bad"), ("fp32", -TINY, "bad"), ("fp32", -1e-300, "bad"), ("fp32", np.inf, "bad"),
    ("fp32", -np.inf, "bad"), ("fp32", np.nan, "bad"), ("fp32", -np.nan, "bad"), ("fp64", -TINY, "bad"),
    ("fp64", np.nextafter(1.0, 2.0), "bad")])
@pytest.mark.parametrize("next_field", [False, True])
def test_edges_of_the_check(storage, value, verdict, next_field):
    import paper_2409_02964_gb300 as P
    from paper_2409_02964_gb300.lattice import LbmError
    lat = P.Lattice(33, 5, 0.7, storage=storage)
    good = np.full((5, 33), 0.7)
    phi = good.copy()
    phi[3, 17] = value
    args = (good, phi) if next_field else (phi,)
    if verdict == "bad":
        with pytest.raises(LbmError):
            lat.set_void_fraction(*args)
    else:
        lat.set_void_fraction(*args)
        if verdict == "zero":
            with pytest.raises(LbmError):
                lat.sync()
        else:
            lat.sync()
    lat.close()


@pytest.mark.parametrize("value,bad", [(1.0, False), (1e-45, False), (np.nextafter(np.float32(1), np.float32(2)), True),
                                       (-1e-45, True), (np.nan, True)])
def test_float_fields(value, bad):
    import paper_2409_02964_gb300 as P
    from paper_2409_02964_gb300.lattice import LbmError
    phi = np.full((5, 33), 0.7, dtype=np.float32)
    phi[0, 32] = value
    for storage in ("fp32", "fp64"):
        lat = P.Lattice(33, 5, 0.7, storage=storage)
        if bad:
            with pytest.raises(LbmError):
                lat.set_void_fraction(phi)
        else:
            lat.set_void_fraction(phi)
            lat.sync()
        lat.close()
