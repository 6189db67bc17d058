"""The work that users of this library have it do, as cases that a program can
time and check: cavities advanced and observed, runs to steady state, Nusselt
series, porosity gradients, and parameter sweeps, through Cavity and Batch.

Sizes and physics are those of the repository's benchmark, tests and the
tables of the paper it follows (64^2 and 1024^2 .. 8192^2 porous cavities,
the 120^2 .. 250^2 lattices of the tables, the 256-cavity sweep, the 512^2
gradient), odd and ragged ones among them.

exact() restates the model (arXiv:1308.2071, Sections 2 to 4) in plain torch
in 64 bits, whole fields at a time, and shares nothing with the package.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

KINDS = ("step", "steady", "series", "adjoint", "batch")


def listed():
    return [
        # a monitoring loop on the smallest lattice of the tests and tables: few
        # steps, then every field is looked at; launches and latency count
        dict(name="monitor_64_f32", kind="step", precision="f32", nx=64, ny=64, Ra=1e4, Da=1e-2, phi=0.6, warm=200,
             steps=10, field=False),
        # the small porous cavity of the tests advanced in time (64^2, Ra 1e4)
        dict(name="run_64_f32", kind="step", precision="f32", nx=64, ny=64, Ra=1e4, Da=1e-2, phi=0.6, warm=200,
             steps=2000, field=False),
        # one row of Table 2: the loop to steady state on its 200^2 grid (capped)
        dict(name="steady_200_f32", kind="steady", precision="f32", nx=200, ny=200, Ra=1e5, Da=1e-4, phi=0.4,
             check_every=1000, steps=4000, field=False),
        # a mid-size lattice with odd, ragged sides and a measured porosity field
        dict(name="run_601x397_field_f32", kind="step", precision="f32", nx=601, ny=397, Ra=1e5, Da=1e-3, phi=0.55,
             warm=100, steps=300, field=True),
        # the precision study's lattice (1024^2, Ra 1e6, Da 1e-4)
        dict(name="run_1024_f32", kind="step", precision="f32", nx=1024, ny=1024, Ra=1e6, Da=1e-4, phi=0.4, warm=50,
             steps=200, field=False),
        # the throughput benchmark: 4096^2, lattice far larger than L2
        dict(name="run_4096_f32", kind="step", precision="f32", nx=4096, ny=4096, Ra=1e6, Da=1e-4, phi=0.4, warm=20,
             steps=100, field=False),
        # the heterogeneous case: 8192^2 with a log-normal permeability field
        dict(name="run_8192_field_f32", kind="step", precision="f32", nx=8192, ny=8192, Ra=1e5, Da=1e-4, phi=0.6,
             warm=5, steps=30, field=True),
        # FP16 flow storage on the precision study's lattice, once the flow has set
        # in (a fluid that has hardly moved is below what half precision resolves)
        dict(name="run_1024_f16", kind="step", precision="f16", nx=1024, ny=1024, Ra=1e6, Da=1e-4, phi=0.4,
             warm=1500, steps=200, field=False),
        # FP64: the wall Nusselt numbers of every step on a grid-refinement lattice
        dict(name="series_257_f64", kind="series", precision="f64", nx=257, ny=257, Ra=1e4, Da=1e-2, phi=0.6,
             warm=100, steps=200, field=False),
        # FP64 reference run of the precision study
        dict(name="run_1024_f64", kind="step", precision="f64", nx=1024, ny=1024, Ra=1e6, Da=1e-4, phi=0.4, warm=10,
             steps=50, field=False),
        # dNu/dphi of the gradient benchmark's lattice (512^2, a checkpoint every 100 steps)
        dict(name="adjoint_512_f32", kind="adjoint", precision="f32", nx=512, ny=512, Ra=1e5, Da=1e-2, phi=0.6,
             steps=600, ckpt=100, field=True),
        # the parameter sweep: 256 cavities of uneven size and parameters
        dict(name="sweep_256_f32", kind="batch", precision="f32", cavities=256, low=64, high=512, steps=20),
    ]


def _between(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def _drawn_physics(rng, nx):
    """Ra such that the viscous relaxation time of Eq. 37 (second occurrence)
    lies in 0.55 .. 1.5, where the lattice is stable, and Da, porosity."""
    tau = 0.5 + math.exp(rng.uniform(math.log(0.05), 0.0))
    Ra = min(1e6, max(1e3, 0.03 * (nx - 1.0) ** 2 / (tau - 0.5) ** 2))
    return dict(Ra=Ra, Da=10.0 ** rng.uniform(-4.0, -2.0), phi=rng.uniform(0.4, 0.7))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "steady", "series", "adjoint", "batch"))
    if kind == "batch":
        low = rng.randint(40, 96)
        return dict(kind="batch", precision="f32", cavities=_between(rng, 12, 220), low=low,
                    high=rng.randint(low + 20, 512), steps=rng.randint(5, 20))
    if kind == "adjoint":
        nx = _between(rng, 96, 500)
        ny = max(64, min(500, round(nx * rng.uniform(0.7, 1.4))))
        return dict(kind=kind, precision="f32", nx=nx, ny=ny, steps=rng.randint(150, 500), ckpt=rng.randint(30, 120),
                    field=True, **_drawn_physics(rng, nx))
    if kind == "steady":
        n = rng.randint(60, 260)
        check = rng.randint(200, 1000)
        return dict(kind=kind, precision="f32", nx=n, ny=n, check_every=check, steps=check * rng.randint(2, 4),
                    field=False, **_drawn_physics(rng, n))
    if kind == "series":
        n = rng.randint(48, 400)
        return dict(kind=kind, precision="f64", nx=n, ny=max(48, round(n * rng.uniform(0.7, 1.3))), warm=50,
                    steps=rng.randint(40, 200), field=False, **_drawn_physics(rng, n))
    precision = rng.choice(("f32", "f32", "f32", "f64", "f16"))
    if precision == "f16":
        nx, ny = rng.randint(256, 1100), rng.randint(256, 1100)
        return dict(kind=kind, precision=precision, nx=nx, ny=ny, warm=1500, steps=rng.randint(50, 400),
                    field=rng.random() < 0.4, **_drawn_physics(rng, nx))
    nx = _between(rng, 64, 1500 if precision == "f64" else 6000)
    ny = max(48, min(6000, round(nx * math.exp(rng.uniform(-0.5, 0.5)))))
    most = 1.5e9 if precision != "f64" else 5e7  # node updates of one pass
    field = rng.random() < 0.4
    steps = max(4, min(400 if field else 800, int(most * rng.uniform(0.3, 1.0) / (nx * ny))))
    return dict(kind=kind, precision=precision, nx=nx, ny=ny, warm=rng.randint(10, 40), steps=steps, field=field,
                **_drawn_physics(rng, nx))


# ---- inputs -----------------------------------------------------------------------------


def _physics(case, seed):
    """Ra, Da and the porosity of one input: those of the case, a little off, by the seed."""
    rng = np.random.default_rng(seed)
    a, b, c = rng.uniform(-1.0, 1.0, 3)
    return case["Ra"] * 1.1 ** a, case["Da"] * 1.1 ** b, case["phi"] + 0.02 * c


def _porosity(case, phi_bar, seed):
    """(ny, nx) float32 porosities on the GPU: a log-normal permeability with a
    Gaussian covariance, mapped through Ergun's K ~ phi^3 / (1 - phi)^2 and
    clipped to [0.3, 0.9]; the gradient's smooth perturbation for "adjoint"."""
    ny, nx = case["ny"], case["nx"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    noise = torch.randn((ny, nx), generator=gen, device="cuda", dtype=torch.float32)
    corr = max(4.0, min(32.0, nx / 16.0))
    ky = torch.fft.fftfreq(ny, device="cuda")[:, None]
    kx = torch.fft.rfftfreq(nx, device="cuda")[None, :]
    k2 = (2.0 * math.pi) ** 2 * (kx * kx + ky * ky)
    y = torch.fft.irfft2(torch.fft.rfft2(noise) * torch.exp(-0.25 * k2 * corr * corr), s=(ny, nx))
    y = (y - y.mean()) / y.std()
    if case["kind"] == "adjoint":
        return (phi_bar + 0.05 * torch.tanh(y)).contiguous()
    grid = np.linspace(0.05, 0.97, 1 << 12)
    g = 3.0 * np.log(grid) - 2.0 * np.log1p(-grid)
    target = 3.0 * math.log(phi_bar) - 2.0 * math.log1p(-phi_bar)
    at = np.interp(np.linspace(-7.0, 7.0, 1 << 12) + target, g, grid)
    table = torch.from_numpy(at).to("cuda", torch.float32)
    pos = ((y.clamp(-6.9, 6.9) + 7.0) * ((len(at) - 1) / 14.0))
    k = pos.floor().long().clamp(0, len(at) - 2)
    w = pos - k
    return (table[k] * (1.0 - w) + table[k + 1] * w).clamp(0.3, 0.9).contiguous()


def _sweep(case, seed):
    """The sweep's cavities: uneven squares, the same for every input, and Ra,
    Da and porosity over their ranges by the seed."""
    from paper_1308_2071_gb300.inputs import cavity_sweep

    sizes = cavity_sweep(case["cavities"], seed=2071, size_range=(case["low"], case["high"]))
    cavs = cavity_sweep(case["cavities"], seed=seed)
    return [dict(c, nx=s["nx"], ny=s["ny"]) for c, s in zip(cavs, sizes)]


def prepare(case, seed):
    from paper_1308_2071_gb300 import Batch, Cavity
    import paper_1308_2071_gb300 as package

    if case["kind"] == "batch":
        cavs = _sweep(case, seed)
        b = Batch(cavs, precision=case["precision"])
        # the plan that a program keeps: the tuned schedule, in the cache of this tree
        b.tune(os.path.join(os.path.dirname(package.__file__), "_build", "cases_tune.txt"))
        return dict(case=case, batch=b, shown=_shown(cavs))
    Ra, Da, phi = _physics(case, seed)
    kw = dict(phi_field=_porosity(case, phi, seed)) if case["field"] else {}
    cav = Cavity(case["nx"], case["ny"], Ra=Ra, Da=Da, phi=phi, precision=case["precision"], **kw)
    if case.get("warm"):
        cav.step(case["warm"])
    return dict(case=case, cavity=cav)


def _shown(cavs):
    """The cavities of a sweep whose whole state is looked at after a pass:
    the smallest, the largest and one between."""
    by = sorted(range(len(cavs)), key=lambda k: cavs[k]["nx"] * cavs[k]["ny"])
    return sorted({by[0], by[len(by) // 2], by[-1]})


# ---- one pass -----------------------------------------------------------------------------


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        b.step(case["steps"])
        hot, cold = b.nusselt()
        code, status = b.status()
        # FP32 lattices: what they hold is given in their own type
        shown = [tuple(t.to(torch.float32) for t in b.read_state(k)) for k in state["shown"]]
        return dict(hot=hot.astype(np.float32), cold=cold.astype(np.float32), code=code, status=status, states=shown)
    cav = state["cavity"]
    if case["kind"] == "step":
        cav.step(case["steps"])
        return cav.observables(fields=True)
    if case["kind"] == "series":
        nu = cav.step_nusselt(case["steps"])
        return dict(cav.observables(fields=True), series=nu)
    if case["kind"] == "steady":
        cav.reset()
        taken, change = cav.run_steady(tol=1e-12, check_every=case["check_every"], max_steps=case["steps"])
        return dict(cav.observables(fields=True), taken=taken, change=change)
    J, grad = cav.adjoint(case["steps"], case["ckpt"])
    return dict(J=J, grad=grad)


# ---- what a pass cannot do without ----------------------------------------------------------

# Operations on the nine flow and five thermal populations of one node in one
# step: sums, velocity, equilibria, relaxation and back-transform of Eq. 16-35.
_FLOPS = 250
_BYTES = {"f32": 57, "f16": 39, "f64": 112}  # of one node's populations as they are kept


def work(case):
    """A pass reads the lattice, and the porosity where there is one, and
    writes it and the fields once; between, each node is updated `steps`
    times, which needs no memory traffic by itself."""
    if case["kind"] == "batch":
        side = (case["low"] + case["high"]) / 2
        nodes = case["cavities"] * (side * side + (case["high"] - case["low"]) ** 2 / 12)
        return dict(bytes=2 * 57 * nodes, flops=_FLOPS * nodes * case["steps"])
    nodes = case["nx"] * case["ny"]
    real = 8 if case["precision"] == "f64" else 4
    given = real * nodes if case["field"] else 0
    if case["kind"] == "adjoint":
        # forward, and the reverse of every step at about twice its operations
        return dict(bytes=given + real * nodes, flops=3 * _FLOPS * nodes * case["steps"])
    return dict(bytes=2 * _BYTES[case["precision"]] * nodes + given + 4 * real * nodes,
                flops=_FLOPS * nodes * case["steps"])


# ---- the same in 64 bits ----------------------------------------------------------------------

_EX = [0, 1, 0, -1, 0, 1, -1, -1, 1]
_EY = [0, 0, 1, 0, -1, 1, 1, -1, -1]
_W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


class _Model:
    """The cavity of Section 4.1 in 64 bits: populations after streaming and
    before the wall rule, whole fields."""

    def __init__(self, nx, ny, Ra, Da, phi_bar, phi=None, device="cuda"):
        self.nx, self.ny, self.dev = nx, ny, device
        cs2, L, Ma = 1.0 / 3.0, float(nx - 1), 0.1
        self.L = L
        tau = 0.5 + Ma * L / math.sqrt(cs2) * math.sqrt(1.0 / Ra)
        tau_t = 0.5 + cs2 * (tau - 0.5) / 0.2
        self.nu = cs2 * (tau - 0.5)
        self.gbeta = Ma * Ma * cs2 / L
        self.s = [1.0, 1.1, 1.1, 1.0, 1.2, 1.0, 1.2, 1.0 / tau, 1.0 / tau]
        self.z = [1.0, 1.0 / tau_t, 1.0 / tau_t, 1.5, 1.5]
        K = Da * L * L
        if phi is None:
            self.phi = phi_bar
            self.lin = phi_bar * self.nu / K
            self.quad = phi_bar * 1.75 / math.sqrt(150.0 * phi_bar ** 3) / math.sqrt(K)
        else:
            self.phi = phi
            dp2 = 150.0 * K * (1.0 - phi_bar) ** 2 / phi_bar ** 3
            self.lin = 150.0 * self.nu / dp2 * (1.0 - phi) ** 2 / phi ** 2
            self.quad = 1.75 / math.sqrt(dp2) * (1.0 - phi) / phi ** 2
        self.wt = [0.6] + [0.1] * 4
        M = [[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1], _EX,
             [0, -2, 0, 2, 0, 1, -1, -1, 1], _EY, [0, 0, -2, 0, 2, 1, 1, -1, -1], [0, 1, -1, 1, -1, 0, 0, 0, 0],
             [0, 0, 0, 0, 0, 1, -1, 1, -1]]
        N = [[1] * 5, [0, 1, 0, -1, 0], [0, 0, 1, 0, -1], [-4, 1, 1, 1, 1], [0, 1, -1, 1, -1]]
        self.M, self.N = np.array(M, float), np.array(N, float)
        self.MI, self.NI = np.linalg.inv(self.M), np.linalg.inv(self.N)
        yb, xb, yf, xf = [], [], [], []
        for y in range(ny):
            for x in ((0, nx - 1) if 0 < y < ny - 1 else range(nx)):
                yb.append(y)
                xb.append(x)
                yf.append(min(max(y, 1), ny - 2))
                xf.append(min(max(x, 1), nx - 2))
        self.yb, self.xb, self.yf, self.xf = (torch.tensor(v, device=device) for v in (yb, xb, yf, xf))
        self.f = [torch.full((ny, nx), w, dtype=torch.float64, device=device) for w in _W]
        self.g = [torch.full((ny, nx), w * 0.5, dtype=torch.float64, device=device) for w in self.wt]

    def at(self, v, y, x):
        return v[y, x] if isinstance(v, torch.Tensor) else v

    def macros(self, f, g, phi, lin, quad):
        T = g[0] + g[1] + g[2] + g[3] + g[4]
        b = 0.5 * phi * self.gbeta * (T - 0.5)
        vx = (f[1] - f[3]) + (f[5] - f[6] - f[7] + f[8])
        vy = (f[2] - f[4]) + (f[5] + f[6] - f[7] - f[8]) + b
        l0 = 0.5 + 0.25 * lin
        v2 = vx * vx + vy * vy
        # |v| with the derivative 0 at v = 0
        vm = torch.where(v2 > 0, torch.sqrt(torch.where(v2 > 0, v2, torch.ones_like(v2))), torch.zeros_like(v2))
        den = l0 + torch.sqrt(l0 * l0 + 0.5 * quad * vm)
        ux, uy = vx / den, vy / den
        total = sum(f[1:])
        P = 0.6 * (total - 2.0 / 3.0 * (ux * ux + uy * uy) / phi)  # phi p, Eq. 23
        return ux, uy, P, T

    def feq(self, P, ux, uy, phi):
        out = []
        uu = ux * ux + uy * uy
        for i in range(9):
            eu = _EX[i] * ux + _EY[i] * uy
            s = _W[i] * (3.0 * eu + 4.5 * eu * eu / phi - 1.5 * uu / phi)
            out.append(3.0 * _W[i] * P + s if i else 1.0 - (5.0 / 3.0) * P + s)
        return out

    def geq(self, T, ux, uy):
        return [self.wt[j] * T * (1.0 + (_EX[j] * ux + _EY[j] * uy) / 0.2) for j in range(5)]

    def walls(self, f, g):
        """Populations and macroscopic values with the wall rule applied."""
        ux, uy, P, T = self.macros(f, g, self.phi, self.lin, self.quad)
        yb, xb, yf, xf = self.yb, self.xb, self.yf, self.xf
        uf, vf, Pf, Tf = (v[yf, xf] for v in (ux, uy, P, T))
        pf, pb = self.at(self.phi, yf, xf), self.at(self.phi, yb, xb)
        Pb = Pf / pf * pb
        Tb = torch.where(xb == 0, torch.ones_like(Tf), torch.where(xb == self.nx - 1, torch.zeros_like(Tf), Tf))
        zero = torch.zeros_like(Tf)
        f0, f1 = self.feq(Pb, zero, zero, pb), self.feq(Pf, uf, vf, pf)
        g0, g1 = self.geq(Tb, zero, zero), self.geq(Tf, uf, vf)
        put = lambda v, w: v.index_put((yb, xb), w)  # noqa: E731
        f = [put(f[i], f0[i] + f[i][yf, xf] - f1[i]) for i in range(9)]
        g = [put(g[j], g0[j] + g[j][yf, xf] - g1[j]) for j in range(5)]
        return f, g, put(ux, zero), put(uy, zero), put(P, Pb), put(T, Tb)

    def step(self, f, g):
        phi = self.phi
        f, g, ux, uy, P, T = self.walls(f, g)
        um = torch.where(ux * ux + uy * uy > 0, torch.sqrt(torch.where(ux * ux + uy * uy > 0, ux * ux + uy * uy,
                                                                       torch.ones_like(ux))), torch.zeros_like(ux))
        drag = self.lin + self.quad * um
        Fx, Fy = -drag * ux, -drag * uy + phi * self.gbeta * (T - 0.5)
        uu, uF = ux * ux + uy * uy, ux * Fx + uy * Fy
        # m_eq of Eq. 16 about the rest state, where P is 1/3, m_1 = -2 and m_2 = 1
        eq = [1.0, 6.0 * (P - 1.0 / 3.0) + 3.0 * uu / phi - 2.0, -9.0 * (P - 1.0 / 3.0) - 3.0 * uu / phi + 1.0, ux,
              -ux, uy, -uy, (ux * ux - uy * uy) / phi, ux * uy / phi]
        S = [None, 6.0 * uF / phi, -6.0 * uF / phi, Fx, -Fx, Fy, -Fy, 2.0 * (ux * Fx - uy * Fy) / phi,
             (ux * Fy + uy * Fx) / phi]
        post = []
        for k in range(9):
            m = sum(self.M[k][i] * f[i] for i in range(9) if self.M[k][i])
            d = self.s[k] * (eq[k] - m)
            if k:
                d = d + (1.0 - 0.5 * self.s[k]) * S[k]
            post.append(d)
        f = [f[i] + sum(self.MI[i][k] * post[k] for k in range(9) if abs(self.MI[i][k]) > 1e-14) for i in range(9)]
        del post, eq, S
        ne = [T, ux * T, uy * T, -2.0 * T, torch.zeros_like(T)]
        post = [self.z[k] * (ne[k] - sum(self.N[k][j] * g[j] for j in range(5) if self.N[k][j])) for k in range(5)]
        g = [g[j] + sum(self.NI[j][k] * post[k] for k in range(5) if abs(self.NI[j][k]) > 1e-14) for j in range(5)]
        shift = lambda v, i: torch.roll(v, (_EY[i], _EX[i]), (0, 1)) if i else v  # noqa: E731
        return [shift(f[i], i) for i in range(9)], [shift(g[j], j) for j in range(5)]

    def advance(self, n):
        with torch.no_grad():
            for _ in range(n):
                self.f, self.g = self.step(self.f, self.g)
        return self

    def nusselt(self, T):
        L = self.L
        c = (-25.0, 48.0, -36.0, 16.0, -3.0)
        left = sum(c[k] * T[:, k] for k in range(5)) / 12.0
        right = -sum(c[k] * T[:, -1 - k] for k in range(5)) / 12.0
        w = torch.ones_like(left)
        w[0] = w[-1] = 0.5
        return tuple((-L * d * w).sum() / (self.ny - 1) for d in (left, right))

    def observables(self):
        f, g, ux, uy, P, T = self.walls(self.f, self.g)
        hot, cold = self.nusselt(T)
        return dict(ux=ux, uy=uy, T=T, p=P / self.phi, t=None, nu_hot=float(hot), nu_cold=float(cold), residual=None,
                    umax=float(torch.sqrt(ux * ux + uy * uy).max()), mass=float(sum(v.sum() for v in f)),
                    heat=float(T.sum()), status=None)


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "batch":
        cavs = _sweep(case, seed)
        shown = _shown(cavs)
        states = []
        for k in shown:
            c = cavs[k]
            m = _Model(c["nx"], c["ny"], c["Ra"], c["Da"], c["phi"], device=device).advance(case["steps"])
            f, g = m.walls(m.f, m.g)[:2]
            states.append((torch.stack(f), torch.stack(g)))
        return dict(hot=None, cold=None, code=None, status=None, states=states)
    Ra, Da, phi = _physics(case, seed)
    field = _porosity(case, phi, seed).double() if case["field"] else None
    if case["kind"] == "adjoint":
        return _gradient(case, Ra, Da, phi, field, device)
    model = _Model(case["nx"], case["ny"], Ra, Da, phi, field, device=device)
    model.advance(case.get("warm", 0))
    if case["kind"] == "series":
        nu = []
        for _ in range(case["steps"]):
            model.advance(1)
            nu.append(torch.stack(model.nusselt(model.walls(model.f, model.g)[5])))
        return dict(model.observables(), series=torch.stack(nu))
    model.advance(case["steps"] if case["kind"] == "step" else -(-case["steps"] // case["check_every"]) *
                  (case["check_every"] + case["check_every"] % 2))
    if case["kind"] == "steady":
        return dict(model.observables(), taken=None, change=None)
    return model.observables()


def _gradient(case, Ra, Da, phi_bar, field, device):
    """J and dJ/dphi by reverse-mode differentiation of the restated steps, a
    few steps at a time from kept states."""
    phi = field.clone().requires_grad_(True)
    every, n = 20, case["steps"]
    kept = []
    with torch.no_grad():
        m = _Model(case["nx"], case["ny"], Ra, Da, phi_bar, field, device=device)
        for k in range(n):
            if k % every == 0:
                kept.append((m.f, m.g))
            m.f, m.g = m.step(m.f, m.g)
    f = [v.clone().requires_grad_(True) for v in m.f]
    g = [v.clone().requires_grad_(True) for v in m.g]
    m = _Model(case["nx"], case["ny"], Ra, Da, phi_bar, phi, device=device)
    J = m.nusselt(m.walls(f, g)[5])[0]
    grads = torch.autograd.grad(J, f + g + [phi], allow_unused=True)
    zero = torch.zeros_like(field)
    seeds = [zero if v is None else v for v in grads[:-1]]
    total = zero.clone() if grads[-1] is None else grads[-1].clone()
    for k in reversed(range(len(kept))):
        f = [v.clone().requires_grad_(True) for v in kept[k][0]]
        g = [v.clone().requires_grad_(True) for v in kept[k][1]]
        m = _Model(case["nx"], case["ny"], Ra, Da, phi_bar, phi, device=device)
        a, b = f, g
        for _ in range(min(every, n - k * every)):
            a, b = m.step(a, b)
        grads = torch.autograd.grad(a + b, f + g + [phi], grad_outputs=seeds, allow_unused=True)
        seeds = [zero if v is None else v for v in grads[:-1]]
        if grads[-1] is not None:
            total += grads[-1]
        kept[k] = None
    return dict(J=float(J.detach()), grad=total)
