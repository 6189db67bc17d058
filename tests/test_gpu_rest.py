"""A fluid at rest: max|u| and the residual are exactly 0 before the first step, in
every storage type."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f32t", "f64", "f16"])
@pytest.mark.parametrize("shape", [(8, 8), (65, 33), (300, 200)])
def test_nothing_moves_before_the_first_step(precision, shape):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1308_2071_gb300 import Cavity

    for kw in ({}, dict(phi_field=torch.full(shape[::-1], 0.4, device="cuda"))):
        c = Cavity(*shape, Ra=1e4, Da=1e-2, phi=0.6, precision=precision, **kw)
        for _ in range(2):  # without a velocity to compare with, and with one
            obs = c.observables(fields=True)
            assert obs["umax"] == 0.0 and obs["residual"] == 0.0
            assert not obs["ux"].any() and not obs["uy"].any()
        c.close()
