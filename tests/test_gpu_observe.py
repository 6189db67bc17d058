"""Observables against the fields that the same call returns, on lattices of one
block of nodes up to several nodes per thread, with ragged ends, with rows for
one Nusselt block and for several, and with a NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def hot_cold(T, L, dT):
    """Eq. 38 on a (ny, nx) temperature field, FP64."""
    w = np.ones(T.shape[0])
    w[0] = w[-1] = 0.5
    hot = -25 * T[:, 0] + 48 * T[:, 1] - 36 * T[:, 2] + 16 * T[:, 3] - 3 * T[:, 4]
    cold = 25 * T[:, -1] - 48 * T[:, -2] + 36 * T[:, -3] - 16 * T[:, -4] + 3 * T[:, -5]
    return [float(-(w * s).sum() * L / (12 * dT) / (T.shape[0] - 1)) for s in (hot, cold)]


@pytest.mark.parametrize("shape", [(8, 8), (31, 257), (300, 200), (1021, 611)])
def test_observables_agree_with_the_fields(shape):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1308_2071_gb300 import Cavity

    nx, ny = shape
    c = Cavity(nx, ny, Ra=1e5, Da=1e-2, phi=0.6, precision="f64")
    c.step(60)
    first = c.observables(fields=True)
    c.step(7)
    obs = c.observables(fields=True)
    again = c.observables()  # no step in between: the same sums, no residual
    old, new = ([o[k].cpu().numpy() for k in ("ux", "uy", "T", "p")] for o in (first, obs))
    # FP64 throughout; the sums differ from numpy's in their order (n 2^-53 of their size),
    # and a rounded T moves Eq. 38 by up to 128 L / 12 x 2^-53 = 1.2e-12 at the largest L here
    umax = np.hypot(new[0], new[1]).max()
    assert obs["umax"] == pytest.approx(umax, rel=1e-14)
    assert obs["residual"] == pytest.approx(np.hypot(new[0] - old[0], new[1] - old[1]).max() / umax, rel=1e-12)
    T = new[2]
    assert obs["heat"] == pytest.approx(T.sum(), rel=1e-10)
    for k, nu in zip(("nu_hot", "nu_cold"), hot_cold(T, nx - 1, T[ny // 2, 0] - T[ny // 2, -1])):
        assert obs[k] == pytest.approx(nu, rel=1e-10)
    assert [again[k] for k in ("nu_hot", "nu_cold", "umax", "mass", "heat")] == \
        [obs[k] for k in ("nu_hot", "nu_cold", "umax", "mass", "heat")] and again["residual"] == 0.0
    c.close()


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_a_nan_reaches_the_maximum(precision):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1308_2071_gb300 import Cavity

    c = Cavity(320, 40, Ra=1e5, Da=1e-2, phi=0.6, precision=precision)
    c.step(10)
    c.observables()
    blob = c.save()
    arr = np.frombuffer(blob, dtype=np.float32 if precision == "f32" else np.float64, count=2 * 40 * 320,
                        offset=40)
    arr.setflags(write=True)
    arr[40 * 320 + 7 * 320 + 20] = np.nan  # a moving population: the rest one has no part in the velocity
    c.load(blob)
    for _ in range(2):  # without a velocity to compare with, and with one
        obs = c.observables(check=False)
        assert np.isnan(obs["umax"]) and np.isnan(obs["mass"])
    c.close()
