"""The batch kernel's work units: whatever their height, every cell goes through the same
FP32 operations, so the populations are the same bit for bit (FP16 / BF16 too: the rounding
bits depend on lattice, column, row and step). Sizes below the halo, around the 60-column
tile and with a last strip of few rows; heights of one row, of a few and beyond the lattice."""
import pytest

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 3, 5, 31, 59, 60, 61, 130, 251]


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_unit_heights_give_the_same_populations(storage):
    import torch
    import paper_2409_02964_gb300 as P
    lats = [(n, 0.6 + 0.05 * i, 0.1 + 0.01 * i, 500.0 + n, 0.3 / (n + 30)) for i, n in enumerate(SIZES)]
    want = None
    for rows in (0, 1, 7, 48, 400):
        b = P.Batch(lats, storage=storage, strip_rows=rows)
        b.init()
        b.step(3)           # single launches, then a replayed graph
        b.step(16)
        b.step_each(1)
        got = [b.populations(i) for i in range(len(lats))]
        b.close()
        assert all(bool(torch.isfinite(g).all()) for g in got)
        if want is None:
            want = got
        else:
            assert all(torch.equal(g, w) for g, w in zip(got, want)), rows
