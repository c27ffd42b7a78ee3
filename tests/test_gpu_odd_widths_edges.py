"""Plain steps over blocks of consecutive nodes against tiles, at the smallest
lattices of each kind that take them (rows off a multiple of 32 and 50 000 nodes
in 64-bit arithmetic; 150 000 in the flow, 250 000 in the temperature and
1 200 000 in 2D otherwise), and just below.

A block of check_every = 1 runs its one step through the reducing kernel, which
keeps the tiles.  Both do the same operations on every node: equal bit for bit,
tolerance zero.
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


def bend(nx, ny, nz):
    return I.pipe_bend_3d(nx, width=6, re=10.0, seed=2, ny=ny, nz=nz)


CASES = {
    "flow_fp64_below": (lambda: bend(37, 37, 36), "fp64"),
    "flow_fp64": (lambda: bend(37, 37, 37), "fp64"),
    "flow_fp32_below": (lambda: bend(53, 53, 53), "fp32"),
    "flow_fp32": (lambda: bend(54, 53, 53), "fp32"),
    "flow_bf16": (lambda: bend(55, 53, 53), "bf16"),
    "heat_fp32_below": (lambda: I.heat_sink(90, 61, 45, re=10.0), "fp32"),
    "heat_fp32": (lambda: I.heat_sink(91, 61, 46, re=10.0), "fp32"),
    "heat_fp64": (lambda: I.heat_sink_quarter(75, 35, 20), "fp64"),
    "flow_2d_fp32": (lambda: I.pipe_bend_2d(1201, 1001, width=40), "fp32"),
    "flow_2d_fp64": (lambda: I.pipe_bend_2d(301, 171, width=21), "fp64"),
}


@pytest.mark.parametrize("name", CASES)
def test_consecutive_nodes_equal_tiles(name):
    from paper_2501_02161_gb300.solver import Solver
    make, storage = CASES[name]
    lat = make()
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
