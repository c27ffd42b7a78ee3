"""Plain steps over blocks of consecutive nodes (rows off a multiple of 32)
against tiles of x-y planes.

A block of check_every = 1 runs its one step through the reducing kernel, which
keeps the tiles; longer ones run their plain steps over consecutive nodes.  Both
do the same operations on every node: equal bit for bit, tolerance zero.  The
lattices are too large for a resident launch, or of 16-bit storage with an odd
width, and end in the middle of a block.
"""
import pytest

torch = pytest.importorskip("torch")

from paper_2501_02161_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_02161_gb300 import build as B
    B.build()


LATTICES = {
    "bend_101x67x73": lambda: I.pipe_bend_3d(101, width=12, re=20.0, seed=2, ny=67, nz=73),
    "sink_129x96x81": lambda: I.heat_sink(129, 96, 81, re=20.0),
    "quarter_205x75x71": lambda: I.heat_sink_quarter(205, 75, 71),
    "bend2d_1301x701": lambda: I.pipe_bend_2d(1301, 701, width=40),
}


@pytest.mark.parametrize("storage", ["fp32", "fp16", "fp64"])
@pytest.mark.parametrize("name", LATTICES)
def test_consecutive_nodes_equal_tiles(name, storage):
    from paper_2501_02161_gb300.solver import Solver
    lat = LATTICES[name]()
    if storage == "fp16" and lat.stencil == I.D2Q9:
        pytest.skip("16-bit storage is built for D3Q19")
    got = []
    for check in (1, 5):
        s = Solver.from_lattice(lat, storage=storage)
        s.forward(tol=0, max_steps=10, check_every=check)
        s.adjoint(tol=0, max_steps=10, check_every=check)
        fs, gs = s.adjoint_fields()
        got.append([x for x in (*s.fields(), fs, gs, s.sensitivity()) if x is not None])
        s.close()
    for a, b in zip(*got):
        assert torch.isfinite(a).all()
        assert torch.equal(a, b)
