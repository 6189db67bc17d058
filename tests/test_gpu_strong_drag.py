"""Velocities of nearly solid cells, where the drag takes almost all of v: the
fields, max|u| and the divergence flag after a few steps, against the oracle's
velocities of the library's own populations.

Tolerances, relative to the largest |u|.  u is v / (l0 + sqrt(l0^2 + l1 |v|)): the drag of
a cell takes about ten roundings (1 / phi^2 counts twice), the root, the reciprocal
(an ulp each) and the products as many: 24 eps.  v is summed from eight
deviations and the buoyancy, each sum rounded to the largest of them: 8 eps max|d| /
max|v|.  The oracle sums populations near 4/9 in FP64, 2^-53 apiece: 8 x 2^-53 /
max|v| more."""
import numpy as np
import pytest

from oracle import Oracle, derive

pytestmark = pytest.mark.gpu

W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]


def cavity(precision, phi, Da=1e-6):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1308_2071_gb300 import Cavity

    return Cavity(phi.shape[1], phi.shape[0], Ra=1e4, Da=Da, phi=0.6, precision=precision,
                  phi_field=torch.from_numpy(phi).cuda())


@pytest.mark.parametrize("part", ["all", "half"])
@pytest.mark.parametrize("solid", [1e-2, 5e-4, 1e-5, 1e-8])
@pytest.mark.parametrize("precision", ["f32", "f32t", "f64"])
def test_velocity_of_nearly_solid_cells(precision, solid, part):
    nx, ny = 37, 30
    phi = np.full((ny, nx), solid)
    if part == "half":
        phi[:, nx // 2:] = 0.6
    c = cavity(precision, phi)
    c.step(21)
    obs = c.observables(fields=True, check=False)
    f, g = (t.cpu().numpy() for t in c.read_state())
    c.close()
    assert obs["status"] == 0
    lat = derive(nx, ny, Ra=1e4, Da=1e-6, phi=0.6)
    o = Oracle(lat, phi_field=phi if precision == "f64" else phi.astype(np.float32).astype(np.float64))
    o.set_state(f, g)
    ux, uy = o.macros()[:2]
    u = np.hypot(ux, uy)
    j = np.hypot(f[1] - f[3] + f[5] - f[6] - f[7] + f[8], f[2] - f[4] + f[5] + f[6] - f[7] - f[8])
    vmax = j[1:-1, 1:-1].max()
    eps = 2.0 ** -53 if precision == "f64" else 2.0 ** -24
    rel = eps * (24 + 8 * np.abs(f - W).max() / vmax) + 8 * 2.0 ** -53 / vmax
    assert 0.0 < obs["umax"] and abs(obs["umax"] - u.max()) <= rel * u.max()
    for name, want in (("ux", ux), ("uy", uy)):
        assert np.abs(obs[name].cpu().numpy() - want)[1:-1, 1:-1].max() <= rel * u.max(), name


@pytest.mark.parametrize("solid", [1.2e-9, 9e-10, 6e-10])
@pytest.mark.parametrize("precision", ["f32", "f32t"])
def test_the_drag_stays_at_its_bound(precision, solid):
    # c_lin / 4 is 4e18 .. 1.5e19 here: from 6.5e18 on twice its square has no FP32 reciprocal, from
    # 1.3e19 on it overflows.  u is of the order of 1e-33
    c = cavity(precision, np.full((30, 37), solid))
    c.step(21)
    obs = c.observables(check=False)
    c.close()
    assert obs["status"] == 0 and 0.0 <= obs["umax"] < 1e-30


@pytest.mark.parametrize("least", [1e-8, 1e-6, 1e-4])
@pytest.mark.parametrize("precision", ["f32", "f32t"])
def test_max_speed_where_a_small_porosity_varies(precision, least):
    # by 5 % a row: v near the walls is 1e10 .. 1e2 times u.  Against the FP64 run; FP32's 21
    # steps and its drag (see above) take some hundred roundings of 6e-8, far below 1 %
    phi = np.geomspace(least, 4.8 * least, 30 * 37).reshape(30, 37)
    umax = {}
    for prec in ("f64", precision):
        c = cavity(prec, phi)
        c.step(21)
        umax[prec] = c.observables(check=False)["umax"]
        c.close()
    assert abs(umax[precision] - umax["f64"]) <= 1e-2 * umax["f64"]
