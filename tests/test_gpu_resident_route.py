"""Which route the steps of a solve take, and what happens when a resident
launch cannot be finished.

Results are the same bit for bit on every route, so the route itself is read
from the launch counter: a block of k steps with its finalize kernel is k + 1
launches, or 3 when its plain steps are one resident launch.
"""
import threading
import time

import pytest

torch = pytest.importorskip("torch")

from paper_2501_02161_gb300 import _capi as C
from paper_2501_02161_gb300 import inputs as I
from test_gpu_resident import CASES, LATTICES as LATTICES_OF_ALL_KINDS

pytestmark = pytest.mark.gpu

WAIT = 1 << 21  # polls of a wait, as the library has it by default


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_02161_gb300 import build as B
    B.build()


def solver(lat, storage="fp32"):
    from paper_2501_02161_gb300.solver import Solver
    return Solver.from_lattice(lat, storage=storage)


def set_resident(s, min_steps=0, wait_limit=WAIT, step_number=0):
    C.check(s.lib.lbm_set_resident(s._ctx, min_steps, wait_limit, step_number), "lbm_set_resident")


def solve(s, steps, check):
    rf = s.forward(tol=0, max_steps=steps, check_every=check)
    ra = s.adjoint(tol=0, max_steps=steps, check_every=check)
    fs, gs = s.adjoint_fields()
    out = [torch.tensor([rf.J, rf.I, ra.I], dtype=torch.float64), *s.fields(), fs, gs, s.sensitivity()]
    return [x.cpu() for x in out if x is not None]


def same(got, ref):
    for a, b in zip(got, ref):
        assert torch.isfinite(b).all()
        assert torch.equal(a, b)


LATTICES = {
    "bend_24": lambda: I.pipe_bend_3d(24, width=6, re=15.0, seed=1),
    "bend_32": lambda: I.pipe_bend_3d(32, width=8, re=15.0, seed=1),
    "bend_33": lambda: I.pipe_bend_3d(33, width=8, re=15.0, seed=1),
    "bend2d_64": lambda: I.pipe_bend_2d(64, 64, width=16),
    "quarter_45x24x13": lambda: I.heat_sink_quarter(45, 24, 13),
}


@pytest.mark.parametrize("storage", ["fp32", "fp64"])
@pytest.mark.parametrize("name", ["bend_24", "bend2d_64", "quarter_45x24x13"])
def test_a_wait_that_gives_up_is_made_good(name, storage):
    """With a limit of 0 polls a wait gives up at the first word that is not
    there yet; the kernel ends by itself, its block runs again a launch per
    step from the untouched input, and nothing of it is left in the results."""
    s = solver(LATTICES[name](), storage)
    ref = solve(s, 200, 5)
    set_resident(s, wait_limit=0)
    n = s.launches()
    same(solve(s, 200, 100), ref)
    phases = 4 if s.thermal else 2
    # every phase's two blocks a launch per step, and the launches that gave up beside them
    assert s.launches() - n > phases * 2 * 101 + 3
    s.close()


@pytest.mark.parametrize("start", [0xF0000000 - 70, 0xFFFFFFF0])
def test_step_numbers_start_again(start):
    """The words carry 32-bit step numbers: before they run out the inboxes are
    cleared and the count begins again."""
    s = solver(LATTICES["bend_24"]())
    ref = solve(s, 400, 5)
    set_resident(s, step_number=start)
    n = s.launches()
    same(solve(s, 400, 100), ref)
    # initial populations and four blocks per phase, and dJ/dgamma
    assert s.launches() - n == 2 * (1 + 4 * 3) + 1
    s.close()


def test_solves_beside_one_another_step_by_launches():
    """A resident launch would keep the other context's steps waiting for a
    whole block: while a second context is in a solve both go a launch per step."""
    s, other = solver(LATTICES["bend_24"]()), solver(I.pipe_bend_3d(64, width=16, re=20.0, seed=2))
    ref = solve(s, 400, 100)
    n = s.launches()
    same(solve(s, 400, 100), ref)
    assert s.launches() - n == 2 * (1 + 4 * 3) + 1  # alone: resident
    torch.cuda.synchronize()

    def long_solve():
        with torch.cuda.stream(torch.cuda.Stream()):
            other.forward(tol=0, max_steps=200000, check_every=500)

    t = threading.Thread(target=long_solve)
    began = other.launches()
    t.start()
    while other.launches() < began + 10:
        time.sleep(0.001)
    n = s.launches()
    with torch.cuda.stream(torch.cuda.Stream()):
        got = solve(s, 400, 100)
    n = s.launches() - n
    beside = t.is_alive()
    t.join()
    assert beside and n == 2 * (1 + 4 * 101) + 1
    same(got, ref)
    s.close()
    other.close()


def test_a_context_tries_again_after_a_wait_gave_up():
    """One stall does not turn a context slow for good; the third time it stays
    with a launch per step."""
    s = solver(LATTICES["bend_24"]())
    init, block, resident = 1, 101, 3

    def forward(blocks):
        n = s.launches()
        s.forward(tol=0, max_steps=100 * blocks, check_every=100)
        return s.launches() - n

    set_resident(s, wait_limit=0)
    assert forward(2) == init + 2 * (resident + block)
    assert forward(3) == init + (resident + block) + 2 * block
    assert forward(3) == init + 3 * block
    set_resident(s)
    assert forward(3) == init + 3 * resident
    s.close()


@pytest.mark.parametrize("storage", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [9, 400])
def test_timed_steps_advance_a_phase_as_a_solve_does(n, storage):
    """2 n steps (n rounded up to even) in either route."""
    for name in ("bend_24", "quarter_45x24x13"):
        s, ref = solver(LATTICES[name](), storage), solver(LATTICES[name](), storage)
        for x in (s, ref):
            x.forward(tol=0, max_steps=20, check_every=5)
            x.adjoint(tol=0, max_steps=20, check_every=5)
        steps = 2 * (n + n % 2)
        assert s.time_steps(0, n) > 0
        # the reducing step that ends a solve gives the fields
        s.forward(tol=0, max_steps=1, check_every=1, reset=False)
        ref.forward(tol=0, max_steps=steps, check_every=5, reset=False)
        ref.forward(tol=0, max_steps=1, check_every=1, reset=False)
        same(s.fields()[:2], ref.fields()[:2])
        s.close()
        ref.close()


@pytest.mark.parametrize("phase", [0, 1, 2, 3])
def test_timed_steps_that_gave_up_leave_nothing_to_read(phase):
    """Both buffers of the phase have been written: what builds on it is refused
    until it has been solved again, and then right."""
    s = solver(LATTICES["quarter_45x24x13"]())
    ref = solve(s, 40, 5)
    set_resident(s, wait_limit=0)
    with pytest.raises(C.LBMError):
        s.time_steps(phase, 400)
    set_resident(s)
    with pytest.raises(C.LBMError):
        s.sensitivity()
    with pytest.raises(C.LBMError):
        s.adjoint_fields()
    if phase < 2:
        with pytest.raises(C.LBMError):
            s.fields()
        s.forward(tol=0, max_steps=40, check_every=5, reset=False)
    s.adjoint(tol=0, max_steps=40, check_every=5, reset=phase < 2)
    fs, gs = s.adjoint_fields()
    same([x.cpu() for x in (*s.fields(), fs, gs, s.sensitivity())], ref[1:])
    s.close()


def test_timed_temperature_adjoint_leaves_the_coupling_its_values():
    """The coupling of the flow adjoint reads what a step of the temperature
    adjoint leaves at outflow nodes beside the populations."""
    s, ref = (solver(LATTICES["quarter_45x24x13"]()) for _ in range(2))
    for x in (s, ref):
        x.forward(tol=0, max_steps=40, check_every=5)
        x.adjoint(tol=0, max_steps=40, check_every=5)
    s.time_steps(3, 400)
    s.solve_phase(3, tol=0, max_steps=0, check_every=5, reset=False)  # the coupling alone
    ref.solve_phase(3, tol=0, max_steps=800, check_every=5, reset=False)
    for x in (s, ref):
        x.solve_phase(2, tol=0, max_steps=20, check_every=5, reset=False)
    same([*s.adjoint_fields(), s.sensitivity()], [*ref.adjoint_fields(), ref.sensitivity()])
    s.close()
    ref.close()


@pytest.mark.parametrize("name,storage,first", [
    ("bend_24", "fp32", {0: 36, 2: 36}),
    ("bend_32", "fp32", {0: 56, 2: 56}),
    ("bend_24", "fp64", {0: 6, 2: 6}),
    ("bend_32", "fp64", {0: 6, 2: 6}),
    ("bend2d_64", "fp32", {0: 56, 2: 56}),
    ("quarter_45x24x13", "fp32", {0: 36, 1: 36, 2: 36, 3: 36}),
    ("bend_33", "bf16", {0: 36, 2: 36}),
])
def test_short_blocks_keep_a_launch_per_step(name, storage, first):
    """The set-up of a resident launch takes 20 to 100 us: blocks with too few
    plain steps to make it good step by launches."""
    s = solver(LATTICES[name](), storage)
    s.forward(tol=0, max_steps=4, check_every=2)
    s.adjoint(tol=0, max_steps=4, check_every=2)
    for phase, steps in sorted(first.items(), key=lambda v: (0, 1, 3, 2).index(v[0])):
        for plain, launches in ((steps - 1, steps + 1), (steps, 3)):
            n = s.launches()
            s.solve_phase(phase, tol=0, max_steps=2 * (plain + 1), check_every=plain + 1, reset=False)
            # the temperature adjoint ends with the coupling
            assert s.launches() - n - (phase == 3) == 2 * launches
    s.close()


def test_short_16_bit_blocks_keep_the_paired_step():
    """The 16-bit forward step over pairs of nodes: the line lies with the box."""
    s = solver(LATTICES["bend_32"](), "fp16")
    s.forward(tol=0, max_steps=4, check_every=2)

    def per_block(plain):
        n = s.launches()
        s.solve_phase(0, tol=0, max_steps=plain + 1, check_every=plain + 1, reset=False)
        return s.launches() - n

    assert per_block(19) == 21
    assert per_block(60) == 3
    s.close()


@pytest.mark.parametrize("check", [2, 3, 4, 8, 15])
@pytest.mark.parametrize("storage", ["fp32", "fp64", "bf16"])
@pytest.mark.parametrize("name", ["bend_24", "quarter_45x24x13"])
def test_resident_launches_of_few_steps(name, storage, check):
    """One to fourteen steps in a launch, both parities."""
    s = solver(LATTICES[name](), storage)
    ref = solve(s, 60, 1)
    set_resident(s, min_steps=1)
    n = s.launches()
    same(solve(s, 60, check), ref)
    phases = 4 if s.thermal else 2
    # initial populations (the temperature's also collide), blocks, coupling, dJ/dgamma
    assert s.launches() - n == phases + 2 * (phases == 4) + phases * -(-60 // check) * 3 + 1
    s.close()


@pytest.mark.parametrize("name,storage", CASES, ids=lambda v: v)
def test_every_phase_with_a_cut_goes_resident(name, storage):
    """One box and many, cut boxes, axes of length 1 to 3, symmetry planes, all
    kinds of openings, every storage: the phases that fit on the chip, and only
    they, take 3 launches a block, and the results are those of single steps."""
    lat = LATTICES_OF_ALL_KINDS[name]()
    for steps in (13, 50):
        s = solver(lat, storage)
        ref = solve(s, steps, 1)
        set_resident(s, min_steps=1)
        n = s.launches()
        same(solve(s, steps, steps), ref)
        code = {"fp64": 0, "fp32": 1, "fp16": 2, "bf16": 3}[storage]
        fits = s.lib.lbm_resident_phases(lat.stencil, lat.nx, lat.ny, lat.nz, code, int(s.thermal))
        phases = (0, 1, 2, 3) if s.thermal else (0, 2)
        blocks = sum(3 if fits >> p & 1 else steps + 1 for p in phases)
        assert fits and s.launches() - n == len(phases) + 2 * s.thermal + blocks + 1
        s.close()


def test_contexts_of_different_sizes_in_turn():
    """Each size asks for its own shared memory; a captured launch of the larger
    one still runs resident after the smaller one's."""
    a, b = solver(I.pipe_bend_3d(64, width=16, re=20.0, seed=2)), solver(I.pipe_bend_3d(16, width=4, re=10.0, seed=2))
    for s in (a, b, a, b, a):
        n = s.launches()
        s.forward(tol=0, max_steps=400, check_every=100)
        assert s.launches() - n == 1 + 4 * 3
    a.close()
    b.close()


def test_a_solve_that_waits_for_its_stream_holds_up_no_other():
    """A context whose caller's stream is busy has not begun: another thread's
    solve comes and goes meanwhile."""
    s, other = solver(LATTICES["bend_24"]()), solver(LATTICES["bend_24"]())
    for x in (s, other):
        x.forward(tol=0, max_steps=100, check_every=100)
    torch.cuda.synchronize()

    def waits():
        with torch.cuda.stream(torch.cuda.Stream()):
            torch.cuda._sleep(2_000_000_000)  # about a second of one SM
            other.forward(tol=0, max_steps=100, check_every=100)

    t = threading.Thread(target=waits)
    t.start()
    time.sleep(0.2)
    with torch.cuda.stream(torch.cuda.Stream()):
        s.forward(tol=0, max_steps=100, check_every=100)
    meanwhile = t.is_alive()
    t.join()
    assert meanwhile
    s.close()
    other.close()
