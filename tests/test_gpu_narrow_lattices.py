"""Lattices of a few rows or columns: many steps in a call take no longer per step
than as many calls of one step each, which are launches of one step (before
the rule for two steps per launch looked at the shape: 30 % longer on the first of
these, 50 % on the last)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(110000, 8), (90000, 12), (30000, 24), (80, 50000), (30, 30000)])
def test_steps_together_are_no_slower(size):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1308_2071_gb300 import Cavity

    c = Cavity(*size, Ra=1e4, Da=1e-2, phi=0.6)
    n = 60  # (no graph: both sides are launched one by one)

    def us(calls):
        best = float("inf")
        for _ in range(6):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for k in calls:
                c.step(k)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3 / n)
        return best

    c.step(5)
    one, together = us([1] * n), us([n])
    c.close()
    assert together <= 1.08 * one, (one, together)
