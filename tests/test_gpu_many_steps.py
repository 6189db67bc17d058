"""Several steps per launch: lbm_step(n) runs all but its last step in launches
of several (tiles on chip on small lattices, two steps per launch on large
ones) and must leave the lattice that n calls of lbm_step(1) leave, bit for
bit, padding and frames included (every kernel runs the same explicit
operations per node).  Sizes at the edges of the tiles, strips and segments
(odd widths, whose right wall is alone in its pair of nodes; a strip or a
segment more or less), every wall variant."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SMALL = [(5, 5), (6, 11), (8, 8), (9, 8), (17, 13), (64, 64), (65, 33), (66, 9), (129, 41), (190, 12), (257, 70), (7, 900)]
# two steps per launch from 720,000 nodes: strips of up to 94 pairs, segments of up to 32 rows, wall tiles of 28 and 22 nodes
LARGE = [(1024, 832), (1025, 831), (901, 950), (2001, 437), (2003, 439), (8, 110000), (9, 95001), (110003, 8), (88300, 10),
         (1501, 1500), (848, 850), (851, 849), (7, 103001)]
MIDDLE = [(250, 249), (500, 451), (601, 397), (847, 849)]  # one step per launch
SIZES = SMALL + MIDDLE + LARGE


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _pair(nx, ny, **kw):
    from paper_1308_2071_gb300 import Cavity

    base = dict(Ra=1e4, Da=1e-2, phi=0.6, precision="f32")
    base.update(kw)
    return Cavity(nx, ny, **base), Cavity(nx, ny, **base)


def _same(a, b, n):
    for _ in range(n):
        a.step(1)
    b.step(n)
    assert a.query() == b.query()
    assert bytes(a.save()) == bytes(b.save())
    # and the lattice after it, from the other buffer
    a.step(1)
    b.step(1)
    assert bytes(a.save()) == bytes(b.save())
    a.close()
    b.close()


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("precision", ["f32", "f32t"])
def test_steps_in_twos_leave_the_same_bits(size, precision):
    a, b = _pair(*size, precision=precision)
    _same(a, b, 13)


# one step per launch: from 2^21 nodes rows of blocks take their own border nodes, if the y walls fit beside them
@pytest.mark.parametrize("size", [(2049, 1100), (1100, 2003), (300001, 8), (40, 60001), (2048, 1024)])
@pytest.mark.parametrize("block", [dict(block_x=32, block_y=1), dict(block_x=64, block_y=2), dict(block_x=8, block_y=2)])
def test_border_nodes_beside_their_rows(size, block):
    a, b = _pair(*size, **block)
    _same(a, b, 4)


@pytest.mark.parametrize("size", [(70, 50), (1040, 820)])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 7, 64, 65, 66, 131])
def test_every_count_of_steps(size, n):
    a, b = _pair(*size)
    _same(a, b, n)


@pytest.mark.parametrize("size", [(70, 50), (1040, 820)])
def test_the_steady_loop_takes_the_same_steps(size):
    # the loop's body runs its steps in an even number of launches, the last alone
    for every in (2, 4, 6, 20, 33):
        a, b = _pair(*size)
        n, _ = b.run_steady(tol=1e-30, check_every=every, max_steps=3 * every)
        assert n == 3 * (every + every % 2)
        _same_state = a.step(n).save()
        assert bytes(_same_state) == bytes(b.save()) and a.query() == b.query()
        a.close()
        b.close()


@pytest.mark.parametrize("size", [(9, 8), (64, 64), (129, 41), (1100, 795), (1101, 794)])
@pytest.mark.parametrize("kw", [dict(thermal_bc=1, Ra=0.0, phi=1.0, Pr=7.0, RaI=6.4e4, forchheimer=0),
                                dict(RaI=1e5, Pr=0.7, Th=1.5, Tc=-0.25), dict(Da=float("inf"), forchheimer=0),
                                dict(collision=1), dict(adiabatic_order=2), "field"])
def test_wall_and_parameter_variants(size, kw):
    import torch

    from paper_1308_2071_gb300.inputs import perturbed_porosity

    if kw == "field":
        phi = perturbed_porosity(size[1], size[0], phi_bar=0.6, amplitude=0.1, corr_len=6.0, seed=3)
        kw = dict(phi_field=torch.from_numpy(phi).cuda())
    a, b = _pair(*size, **kw)
    _same(a, b, 12)


@pytest.mark.parametrize("size", [(70, 50), (1040, 820)])
def test_divergence_between_two_steps_of_a_launch_is_flagged(size):
    # a NaN planted in the lattice spreads and raises the flag, also when the
    # first step that meets it is one whose lattice stays on chip
    from paper_1308_2071_gb300 import Cavity, _lib

    nx, ny = size
    pitch = -(-nx // 32) * 32
    c = Cavity(nx, ny, Ra=1e4, Da=1e-2, phi=0.6, precision="f32")
    c.step(5)
    blob = c.save()
    arr = np.frombuffer(blob, dtype=np.float32, count=14 * pitch * ny, offset=40)
    arr.setflags(write=True)
    arr[1 * pitch * ny + 25 * pitch + 33] = np.nan
    c.load(blob)
    c.step(9)
    assert c.query()[1] == _lib.LBM_ERR_DIVERGED
    c.close()


@pytest.mark.parametrize("nx,ny", [(127, 128), (257, 257), (260, 263), (333, 331), (903, 897)])
def test_fp64_default_shapes_leave_the_same_bits(nx, ny):
    """FP64 takes one or two nodes per thread by the size of the lattice; both on
    either side of each line give what one node per thread gives."""
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1308_2071_gb300 import Cavity

    got = []
    for shape in ({}, dict(block_x=64, block_y=1, nodes_per_thread=1)):
        with Cavity(nx, ny, Ra=1e5, Da=1e-2, phi=0.6, precision="f64", **shape) as c:
            c.step(12)
            got.append([a.cpu() for a in c.read_state()] + [c.nusselt()])
    assert all(torch.equal(a, b) for a, b in zip(got[0][:-1], got[1][:-1])) and got[0][-1] == got[1][-1]
