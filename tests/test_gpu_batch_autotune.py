"""Autotuning never leaves a batch slower than it was: the height it had is timed too (a lone
48^2 lattice runs units of 12 rows; the best of the listed heights, 16, takes 1.16 times as
long). Margin: half of that."""
import pytest

pytestmark = pytest.mark.gpu


def test_a_faster_automatic_height_is_kept():
    import torch
    import paper_2409_02964_gb300 as P
    b = P.Batch([(48, 0.8, 0.2, 1000.0, 0.01)])

    def us_per_step():
        best = float("inf")
        for _ in range(20):
            a, e = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record(b.stream)
            b.step(64)
            e.record(b.stream)
            e.synchronize()
            best = min(best, a.elapsed_time(e) * 1e3 / 64)
        return best

    b.init()
    before = us_per_step()
    b.autotune(trial_steps=64)
    assert us_per_step() <= 1.08 * before
    b.close()
