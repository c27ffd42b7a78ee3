"""Resident launches (many steps in one launch, populations on the chip)
against a launch per step.

Both run the same operations on every node, so after the same number of steps
the fields, the objective, the adjoint populations and dJ/dgamma are equal bit
for bit: the tolerance is zero.  check_every decides the route: blocks of up to
six steps go a launch per step, longer ones resident.  The lattices cover one
box and many, sizes that leave cut boxes, axes of length 1 to 3 (a box that is
its own neighbour), symmetry planes, all faces and kinds of openings, every
storage, both gamma models, and step counts of both parities.
"""
import threading

import numpy as np
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


def periodic(nx, ny, nz, seed=3):
    """No walls at all: every population crosses the seams; one inlet node and
    one outlet node in the interior drive it."""
    rng = np.random.default_rng(seed)
    n = nx * ny * nz
    flags = np.zeros(n, np.uint8)
    bc = np.zeros((n, 4))
    flags[0] = I.make_flag(I.VEL, (0, 1, 0))
    bc[0, :3] = (0.01, 0.02, 0.0)
    if n > 1:
        flags[n - 1] = I.make_flag(I.PRES, (-1, 0, 0))
        bc[n - 1, 0] = 1.0
    return I.Lattice(f"periodic_{nx}x{ny}x{nz}", I.D3Q19, nx, ny, nz, flags, 0.4 + 0.6 * rng.random(n),
                     bc.ravel(), tau=0.9)


LATTICES = {
    "bend_12": lambda: I.pipe_bend_3d(12, width=4, re=10.0, seed=2),
    "bend_33x17x40_linear": lambda: I.pipe_bend_3d(33, width=4, re=10.0, seed=2, ny=17, nz=40,
                                                   gamma_model=I.GAMMA_LINEAR),
    "bend_64": lambda: I.pipe_bend_3d(64, width=16, re=20.0, seed=2),
    "six_port_a": lambda: I.six_port_box(thermal=True),
    "six_port_b": lambda: I.six_port_box(nx=23, ny=19, nz=31, swap=True, thermal=True),
    "sink_48x21x19": lambda: I.heat_sink(48, 21, 19, re=10.0),
    "sink_96x48x24": lambda: I.heat_sink(96, 48, 24, re=20.0),
    "quarter_45x24x13": lambda: I.heat_sink_quarter(45, 24, 13),
    "quarter_192x48x24": lambda: I.heat_sink_quarter(192, 48, 24),
    "periodic_1x1x1": lambda: periodic(1, 1, 1),
    "periodic_2x3x1": lambda: periodic(2, 3, 1),
    "periodic_37x2x3": lambda: periodic(37, 2, 3),
    "bend2d_64": lambda: I.pipe_bend_2d(64, 64, width=16),
    "bend2d_37x29": lambda: I.pipe_bend_2d(37, 29, width=7, gamma_value=0.8),
    "bend2d_300x211": lambda: I.pipe_bend_2d(300, 211, width=31),
}
CASES = [(n, s) for n in LATTICES for s in ("fp32", "fp64") if not (n in ("bend_64", "quarter_192x48x24") and s == "fp64")]
CASES += [(n, s) for n in ("bend_12", "bend_33x17x40_linear", "six_port_b") for s in ("fp16", "bf16")]


def solve(lat, storage, steps, check):
    from paper_2501_02161_gb300.solver import Solver
    s = Solver.from_lattice(lat, storage=storage)
    out = []
    rf = s.forward(tol=0, max_steps=steps, check_every=check)
    ra = s.adjoint(tol=0, max_steps=steps, check_every=check)
    rho, u, T = s.fields()
    fs, gs = s.adjoint_fields()
    out = [torch.tensor([rf.J, rf.I, ra.I], dtype=torch.float64), rho, u, fs, s.sensitivity()]
    out += [x for x in (T, gs) if x is not None]
    s.close()
    return [x.cpu() for x in out]


@pytest.mark.parametrize("name,storage", CASES, ids=lambda v: v)
def test_resident_steps_equal_single_steps(name, storage):
    lat = LATTICES[name]()
    for steps in (13, 50):
        ref = solve(lat, storage, steps, 5)
        got = solve(lat, storage, steps, steps)
        for a, b in zip(got, ref):
            assert torch.isfinite(b).all()
            assert torch.equal(a, b)


def test_threads_with_contexts_of_their_own():
    """One resident launch at a time: whoever finds the gate taken steps by
    launches, with the same results."""
    lats = [I.pipe_bend_3d(24, width=6, re=15.0, seed=k) for k in range(4)]
    ref = [solve(lat, "fp32", 400, 5) for lat in lats]
    got = [None] * 4

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(3):
                got[k] = solve(lats[k], "fp32", 400, 100)

    ts = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    # the fields and the adjoint; J and I are those of the last step in both
    for a, b in zip(got, ref):
        for x, y in zip(a, b):
            assert torch.equal(x, y)
