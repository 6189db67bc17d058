"""Bounds-checked build of the library over the kernels that take several steps
per launch, which small lattices and untuned batches do not reach: tiles on
chip, two steps per launch just above the size that it starts at, on odd and even
widths and on the narrowest and lowest lattices that take it, and the two-step batch.  No access may
leave its plane (a read by a lane whose result is dropped would not show in any
bits)."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes as C
import json
import sys

sys.path.insert(0, sys.argv[1])
from paper_1308_2071_gb300 import _lib

lib = _lib.load(sys.argv[2])
import torch

from paper_1308_2071_gb300 import Batch, Cavity

torch.cuda.set_device(0)


def count():
    en, n = C.c_int(), C.c_long()
    _lib.check(lib.lbm_bounds_check(C.byref(en), C.byref(n)))
    return en.value, n.value


enabled, _ = count()
runs = []
tiles = [(8, 8), (9, 31), (33, 8), (64, 64), (121, 67), (200, 200), (8, 300), (300, 8)]
twos = [(901, 871), (1000, 790), (36, 25000), (37, 24001), (60000, 24), (80003, 20)]
for (nx, ny) in tiles + twos:
    for prec in ("f32", "f32t"):
        for kw in ({}, dict(adiabatic_order=2), dict(thermal_bc=1, RaI=1e4), "field"):
            phi = torch.full((ny, nx), 0.55, device="cuda") if kw == "field" else None
            c = Cavity(nx, ny, Ra=1e4, Da=1e-2, phi=0.6, precision=prec, phi_field=phi,
                       **({} if kw == "field" else kw))
            c.step(25)
            c.observables(fields=True, check=False)
            c.close()
            runs.append([nx, ny, prec, str(kw), count()[1]])
cavs = [dict(nx=n, ny=m, Ra=1e4, Da=1e-2, phi=0.6) for (n, m) in ((8, 9), (9, 8), (37, 41), (193, 131), (401, 38))]
for prec in ("f32", "f32t"):
    b = Batch(cavs, precision=prec)
    b.tune(sys.argv[3])
    key, *_ = open(sys.argv[3]).read().splitlines()[-1].split()
    b.close()
    with open(sys.argv[3], "w") as f:
        f.write(f"{key} 256 1 0 3\n")
    count()
    b = Batch(cavs, precision=prec)
    b.tune(sys.argv[3])
    b.step(25)
    b.nusselt()
    b.close()
    runs.append(["batch", prec, count()[1]])
print(json.dumps(dict(enabled=enabled, runs=runs)))
"""


def test_several_steps_per_launch_stay_in_their_planes(tmp_path):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1308_2071_gb300.build import build

    script = tmp_path / "child.py"
    script.write_text(CHILD)
    r = subprocess.run([sys.executable, str(script), ROOT, build(checked=True), str(tmp_path / "tune.txt")],
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["enabled"] == 1 and len(out["runs"]) == 14 * 2 * 4 + 2
    bad = [run for run in out["runs"] if run[-1] != 0]
    assert not bad, bad
