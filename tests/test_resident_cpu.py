"""The exchange of resident launches, on the CPU: every population that leaves
a box is sent to the word its receiver reads, inside the inboxes and once, and
every word that is waited for is sent, under every set of symmetry planes."""
import ctypes

import pytest

from paper_2501_02161_gb300 import _capi as C


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_2501_02161_gb300 import build as B
    B.build()


def mismatches(stencil, nx, ny, nz):
    bad = ctypes.c_longlong(-1)
    C.check(C.lib().lbm_check_addressing(stencil, nx, ny, nz, ctypes.byref(bad)), "lbm_check_addressing")
    return bad.value


@pytest.mark.parametrize("shape", [(12, 12, 12), (16, 16, 16), (31, 23, 19), (97, 61, 43), (192, 48, 24), (1, 40, 2)])
@pytest.mark.parametrize("stencil", [1, 2], ids=["D3Q19", "D3Q7"])
def test_3d_words_reach_their_readers(stencil, shape):
    assert mismatches(stencil, *shape) == 0


@pytest.mark.parametrize("shape", [(64, 64), (300, 211), (8, 255), (600, 3), (2, 2)])
def test_2d_words_reach_their_readers(shape):
    assert mismatches(0, shape[0], shape[1], 1) == 0
