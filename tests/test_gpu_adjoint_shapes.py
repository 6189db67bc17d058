"""Gradient at the sizes where the reverse kernel's split can go wrong: the
smallest lattices (no or one interior column, rows and columns next to two
walls), odd and even widths (a thread takes two nodes), several blocks, the
cooled enclosure with a heat source, and recomputed segments shorter than asked
for.  Compared with central differences of the FP64 forward run."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (a few nodes across resolve, and stay stable at, a small Rayleigh number only)
TINY, SIDE, COOLED = dict(Ra=1e2, Da=1e-2), dict(Ra=1e5, Da=1e-2), dict(Ra=1e5, Da=1e-2, RaI=1e6, thermal_bc=1)


@pytest.mark.parametrize("nx,ny,kw", [(5, 5, TINY), (6, 8, TINY), (7, 5, TINY), (8, 9, TINY), (37, 23, SIDE),
                                      (130, 67, SIDE), (21, 24, COOLED)])
def test_gradient_matches_forward_differences(nx, ny, kw):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1308_2071_gb300 import Cavity

    steps = 200
    rng = np.random.default_rng(nx * ny)
    phi = 0.6 + 0.1 * rng.uniform(-1, 1, (ny, nx))

    def run(precision, p):
        return Cavity(nx, ny, phi=0.6, precision=precision, phi_field=torch.from_numpy(p).cuda(), **kw)

    def J(p):
        with run("f64", p) as c:
            c.step(steps)
            return c.nusselt()[0]

    dirs = [rng.uniform(-1, 1, phi.shape) for _ in range(2)]
    for x, y in ((0, 0), (1, 1), (nx - 1, ny // 2), (nx - 2, ny // 2), (nx - 3, 2), (nx // 2, ny - 1), (2, ny - 2)):
        v = np.zeros_like(phi)
        v[y, x] = 1.0
        dirs.append(v)

    def difference(v, h=1e-5):  # the third-order term taken out: directions over the whole field have a large one
        d1, d2 = ((J(phi + a * v) - J(phi - a * v)) / (2 * a) for a in (h, 2 * h))
        return (4 * d1 - d2) / 3

    fd = np.array([difference(v) for v in dirs])
    with run("f64", phi) as c:
        j, g = c.adjoint(steps, steps)
        few = c.adjoint(steps, 3)[1]
    assert torch.equal(g, few)
    g = g.cpu().numpy()
    ad = np.array([float((g * v).sum()) for v in dirs])
    # rounding of J, about 1e-14 of it, over 2 h
    assert np.abs(ad - fd).max() <= 1e-6 * np.abs(fd).max() + 1e-9 * abs(j), (ad, fd)
    for precision in ("f32", "f32t"):
        with run(precision, phi) as c:
            g32 = c.adjoint(steps, 50)[1].double().cpu().numpy()
        assert np.abs(g32 - g).max() <= 1e-3 * np.abs(g).max()
