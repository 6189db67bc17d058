"""Batched sweep with two steps per launch (a schedule that lbm_batch_tune may
pick): every cavity evolves bit for bit as it does alone, whatever the number
of steps of a call, on odd and even widths, one strip and several, one segment
and several, and from either buffer."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CAVS = [dict(nx=37, ny=41, Ra=1e5, Da=1e-2, phi=0.6), dict(nx=64, ny=64, Ra=1e4, Da=1e-1, phi=0.3),
        dict(nx=190, ny=80, Ra=1e6, Da=1e-4, phi=0.9), dict(nx=193, ny=131, Ra=3e5, Da=3e-3, phi=0.45),
        dict(nx=8, ny=9, Ra=1e3, Da=1e-2, phi=0.5), dict(nx=401, ny=38, Ra=1e5, Da=1e-3, phi=0.5)]


@pytest.mark.parametrize("precision", ["f32", "f32t"])
def test_two_steps_per_launch_leave_the_same_bits(precision, tmp_path):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1308_2071_gb300 import Batch, Cavity

    # a cached plan names the schedule: tile width and height, blocks per SM, schedule (3 and more: in twos)
    cache = tmp_path / "tune.txt"
    probe = Batch(CAVS, precision=precision)
    probe.tune(str(cache))
    key = cache.read_text().split()[0]
    probe.close()
    for plan in ("256 1 0 3", "128 -2 0 4", "32 0 0 5"):
        cache.write_text(f"{key} {plan}\n")
        b = Batch(CAVS, precision=precision)
        b.tune(str(cache))
        for n in (1, 2, 3, 6, 25):
            b.step(n)
        assert b.status()[0] == 0 and b.query()["t"] == 37
        hot, _ = b.nusselt()
        for k, cv in enumerate(CAVS):
            c = Cavity(cv["nx"], cv["ny"], Ra=cv["Ra"], Da=cv["Da"], phi=cv["phi"], precision=precision)
            for _ in range(37):
                c.step(1)
            for x, y in zip(c.read_state(), b.read_state(k)):
                assert np.array_equal(x.cpu().numpy(), y.cpu().numpy()), (plan, k)
            assert abs(c.nusselt()[0] - hot[k]) <= 1e-12 * abs(hot[k])
            c.close()
        b.close()
