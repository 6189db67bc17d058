"""Graphs of the batched sweep: calls of the same numbers of steps instantiate none
once each number has been through both buffers, in either schedule and
whatever the parity that a call leaves; and runs long enough for graphs of
two-step launches leave the bits of cavities advanced alone.

The instantiations are counted in a child process, by a library in front of the
CUDA runtime that passes them on."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COUNTER = r"""
#include <dlfcn.h>
static int calls;
int graphs_instantiated(void) { return calls; }
int cudaGraphInstantiate(void** exec, void* graph, unsigned long long flags) {
    static int (*real)(void**, void*, unsigned long long);
    if (!real) {
        void* rt = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
        if (rt) real = (int (*)(void**, void*, unsigned long long))dlsym(rt, "cudaGraphInstantiate");
        if (!real) return 999;  /* cudaErrorUnknown */
    }
    ++calls;
    return real(exec, graph, flags);
}
"""

CHILD = r"""
import ctypes as C
import json
import sys

sys.path.insert(0, sys.argv[1])
import torch

from paper_1308_2071_gb300 import Batch

count = C.CDLL(sys.argv[2]).graphs_instantiated
cavs = [dict(nx=n, ny=m, Ra=1e4, Da=1e-2, phi=0.6) for (n, m) in ((37, 41), (40, 60), (64, 33))]
cache = sys.argv[3]
probe = Batch(cavs)
probe.tune(cache)
key = open(cache).read().split()[0]
probe.close()
out = []
for plan in ("128 2 0 0", "256 1 0 3"):
    with open(cache, "w") as f:
        f.write(f"{key} {plan}\n")
    for steps in (1, 2, 3, 4, 19, 20, 21, 64, 65, 66, 130):
        b = Batch(cavs)
        b.tune(cache)
        for _ in range(4):
            b.step(steps)
        before = count()
        for _ in range(6):
            b.step(steps)
        out.append([plan, steps, before, count() - before])
        assert b.status()[0] == 0 and b.query()["t"] == 10 * steps
        b.close()
print(json.dumps(out))
"""


def skip_without_gpu():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_no_graph_is_instantiated_twice(tmp_path):
    skip_without_gpu()
    src, so, child = tmp_path / "counter.c", tmp_path / "counter.so", tmp_path / "child.py"
    src.write_text(COUNTER)
    child.write_text(CHILD)
    subprocess.run(["gcc", "-O1", "-D_GNU_SOURCE", "-fPIC", "-shared", "-o", str(so), str(src), "-ldl"], check=True)
    r = subprocess.run([sys.executable, str(child), ROOT, str(so), str(tmp_path / "tune.txt")], capture_output=True,
                       text=True, timeout=600, env=dict(os.environ, LD_PRELOAD=str(so)))
    assert r.returncode == 0, r.stderr[-3000:]
    runs = json.loads(r.stdout.strip().splitlines()[-1])
    assert runs[0][2] > 0  # the counter is in front of the runtime
    again = [run for run in runs if run[3] != 0]
    assert not again, again


@pytest.mark.parametrize("precision", ["f32", "f32t"])
def test_graphs_of_two_step_launches_leave_the_same_bits(precision, tmp_path):
    skip_without_gpu()
    from paper_1308_2071_gb300 import Batch, Cavity

    cavs = [dict(nx=37, ny=41, Ra=1e5, Da=1e-2, phi=0.6), dict(nx=60, ny=9, Ra=1e4, Da=1e-1, phi=0.3)]
    cache = tmp_path / "tune.txt"
    probe = Batch(cavs, precision=precision)
    probe.tune(str(cache))
    key = cache.read_text().split()[0]
    probe.close()
    cache.write_text(f"{key} 256 1 0 3\n")
    b = Batch(cavs, precision=precision)
    b.tune(str(cache))
    total = 0
    for n in (64, 65, 66, 131, 1, 258):  # 0, 1, 1, 2, 0 and 4 graphs, from either parity
        b.step(n)
        total += n
    assert b.status()[0] == 0 and b.query()["t"] == total
    for k, cv in enumerate(cavs):
        c = Cavity(cv["nx"], cv["ny"], Ra=cv["Ra"], Da=cv["Da"], phi=cv["phi"], precision=precision)
        for _ in range(total):
            c.step(1)
        for x, y in zip(c.read_state(), b.read_state(k)):
            assert np.array_equal(x.cpu().numpy(), y.cpu().numpy()), k
        c.close()
    b.close()
