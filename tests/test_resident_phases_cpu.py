"""Which phases of a lattice fit on the chip, and their exchange, on the CPU.

lbm_check_addressing counts the exchange of every (storage, phase) that has a
cut, none of one that has not: the expected phases are stated here (bits: flow,
temperature, flow adjoint, temperature adjoint), so that a phase that silently
loses its cut, and its check with it, is seen.
"""
import ctypes
import os
import subprocess
import sys

import pytest

from paper_2501_02161_gb300 import _capi as C


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_2501_02161_gb300 import build as B
    B.build()


# shape: phases of the flow alone, and with temperature, for FP64, FP32 and both 16-bit storages
PHASES_3D = {
    (12, 12, 12): ((5, 5, 5), (15, 15, 15)),
    (31, 23, 19): ((5, 5, 5), (15, 15, 15)),
    (48, 48, 48): ((5, 5, 5), (15, 15, 15)),
    (64, 64, 64): ((0, 5, 5), (10, 15, 15)),
    (97, 61, 43): ((0, 5, 5), (10, 11, 11)),  # the coupled adjoint's operands are too many
    (192, 48, 24): ((0, 5, 5), (10, 15, 15)),
    (72, 72, 72): ((0, 0, 1), (0, 10, 11)),
    (5, 200, 3): ((5, 5, 5), (15, 15, 15)),
    (256, 256, 256): ((0, 0, 0), (0, 0, 0)),
}
PHASES_2D = {(64, 64): 5, (300, 211): 5, (7, 500): 5, (512, 384): 5, (1000, 700): 0}


def exchange(stencil, shape):
    bad = ctypes.c_longlong(-1)
    C.check(C.lib().lbm_check_addressing(stencil, *shape, ctypes.byref(bad)), "lbm_check_addressing")
    return bad.value


@pytest.mark.parametrize("shape", PHASES_3D, ids=lambda s: "x".join(map(str, s)))
def test_3d_phases_and_their_words(shape):
    phases = C.lib().lbm_resident_phases
    for thermal in (0, 1):
        want = PHASES_3D[shape][thermal]
        assert [phases(1, *shape, storage, thermal) for storage in range(4)] == [*want, want[2]]
    if max(shape) < 256:
        assert exchange(1, shape) == 0
        assert exchange(2, shape) == 0


@pytest.mark.parametrize("shape", PHASES_2D, ids=lambda s: "x".join(map(str, s)))
def test_2d_phases_and_their_words(shape):
    phases = C.lib().lbm_resident_phases
    assert [phases(0, *shape, 1, storage, 0) for storage in range(2)] == [PHASES_2D[shape]] * 2
    assert exchange(0, (*shape, 1)) == 0


def test_lattices_that_are_refused_have_no_phases():
    phases = C.lib().lbm_resident_phases
    assert phases(0, 64, 64, 2, 1, 0) == phases(0, 64, 64, 1, 2, 0) == phases(0, 64, 64, 1, 1, 1) == 0
    assert phases(1, 0, 16, 16, 1, 0) == phases(1, 16, 16, 16, 4, 0) == phases(2, 16, 16, 16, 1, 0) == 0


def test_no_host_memory_is_an_error_not_an_abort():
    """The check's tables do not fit under the limit set here; the call reports it."""
    code = """
import ctypes, resource, sys
sys.path.insert(0, {root!r})
from paper_2501_02161_gb300 import _capi as C
L = C.lib()
vm = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (vm + (1 << 20), vm + (1 << 20)))
bad = ctypes.c_longlong(-1)
sys.exit(0 if L.lbm_check_addressing(1, 64, 64, 64, ctypes.byref(bad)) == C.LBM_ERR_OOM else 3)
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code.format(root=root)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
