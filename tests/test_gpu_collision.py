"""The rearranged collision (lbm_core.cuh) over the range of its drag solve: one
step of the lattice from the library's own state against the oracle, every
population, from nearly no permeability to none of the drag, with and without
the Forchheimer term, uniform and per-cell porosity, both collision
operators, wall temperatures and sources that move every constant.

Tolerances.  FP64: populations are at most 1 in magnitude (f_0 = 4/9, g_0 up to
0.9 here), the oracle and the library each round a few tens of operations of
that size, 1.1e-16 apiece: 5e-15.  FP32: stored deviations below 0.5 round to
3e-8, a step adds a few more roundings of that size: 2e-7.  The square root
and the reciprocal are the hardware's approximations refined to the last bit
or so: an error of 2^-20 left in them would show as 1e-6 of the drag."""
import numpy as np
import pytest

from oracle import Oracle, derive

pytestmark = pytest.mark.gpu

CASES = {
    "tight": dict(Ra=1e5, Da=1e-6, phi=0.4),
    "open": dict(Ra=1e4, Da=1e-1, phi=0.9),
    "no_darcy": dict(Ra=1e4, Da=float("inf"), phi=1.0, Pr=0.71),
    "no_forchheimer": dict(Ra=1e4, Da=1e-4, phi=0.5, forchheimer=0),
    "lbgk": dict(Ra=1e4, Da=1e-3, phi=0.6, collision=1),
    "source": dict(Ra=1e5, Da=1e-2, phi=0.4, Pr=0.7, RaI=1e6, Th=1.5, Tc=-0.25),
    "constants": dict(Ra=1e4, Da=1e-2, phi=0.6, sigma=1.3, varpi=-1.5, J=1.2),
    "field": dict(Ra=1e5, Da=1e-3, phi=0.6),
}


@pytest.mark.parametrize("precision,tol", [("f64", 5e-15), ("f32", 2e-7), ("f32t", 2e-7)])
@pytest.mark.parametrize("case", list(CASES))
def test_one_step_over_the_drag_range(case, precision, tol, nthreads):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1308_2071_gb300 import Cavity
    from paper_1308_2071_gb300.inputs import perturbed_porosity

    nx, ny = 21, 18
    kw = dict(CASES[case])
    phi = perturbed_porosity(ny, nx, phi_bar=0.6, amplitude=0.15, corr_len=3.0, seed=9) if case == "field" else None
    okw = {k: v for k, v in kw.items() if k not in ("forchheimer", "collision")}
    lat = derive(nx, ny, **okw)
    lat.forchheimer = kw.get("forchheimer", 1)
    if kw.get("collision"):
        tau, tau_t = 1 / lat.s[7], 1 / lat.zeta[1]
        for k in range(9):
            lat.s[k] = 1 / tau
        for k in range(5):
            lat.zeta[k] = 1 / tau_t
    if phi is not None:
        kw["phi_field"] = torch.from_numpy(phi).cuda()
    cav = Cavity(nx, ny, precision=precision, **kw)
    o = Oracle(lat, phi_field=phi) if phi is not None else Oracle(lat)
    for n in (1, 30, 300):
        cav.step(n - cav.query()[0])
        f, g = cav.read_state()
        o.set_state(f.cpu().numpy(), g.cpu().numpy())
        o.step(1, threads=nthreads)
        cav.step(1)
        f1, g1 = cav.read_state()
        fo, go = o.state()
        assert np.abs(f1.cpu().numpy() - fo).max() < tol and np.abs(g1.cpu().numpy() - go).max() < tol, n
    cav.close()
