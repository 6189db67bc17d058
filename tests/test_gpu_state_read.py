"""A state read is bound by the 14 FP64 planes that it writes: no velocity is solved
for in a fluid node.  Against a copy of as many bytes on the same GPU, FP64 at
1024^2: 2.5 times the copy's time (uncoalesced shifts of the pull), 4.5 with the velocities."""
import pytest

pytestmark = pytest.mark.gpu


def ms(f, torch):
    best = float("inf")
    for _ in range(12):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def test_a_state_read_solves_for_no_velocity():
    import ctypes as C

    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1308_2071_gb300 import Cavity, _lib

    n = 1024
    c = Cavity(n, n, Ra=1e5, Da=1e-2, phi=0.6, precision="f64")
    c.step(3)
    f = torch.empty((9, n, n), dtype=torch.float64, device="cuda")
    g = torch.empty((5, n, n), dtype=torch.float64, device="cuda")
    src, dst = (torch.empty((14, n, n), dtype=torch.float64, device="cuda") for _ in range(2))
    read = ms(lambda: _lib.check(_lib.load().lbm_read_state(c.handle, C.c_void_p(f.data_ptr()),
                                                            C.c_void_p(g.data_ptr())), c.handle), torch)
    copy = ms(lambda: dst.copy_(src), torch)
    c.close()
    print(read, copy)
    assert read <= 3.4 * copy, (read, copy)
