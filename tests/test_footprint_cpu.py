"""lbm_footprint_bytes is what lbm_create allocates: populations, fields and
per-block sums.  What resident launches exchange is not part of it, since the
contexts of a batch, which are admitted by it, never go resident."""
import pytest

from paper_2501_02161_gb300 import _capi as C


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_2501_02161_gb300 import build as B
    B.build()


@pytest.mark.parametrize("thermal", [0, 1])
@pytest.mark.parametrize("storage", [0, 1, 2, 3])
@pytest.mark.parametrize("shape", [(16, 16, 16), (64, 64, 64), (96, 48, 24), (97, 61, 43), (192, 96, 48), (320, 160, 80)])
def test_footprint_is_the_context_of_a_batch(shape, storage, thermal):
    nodes = shape[0] * shape[1] * shape[2]
    np_ = -(-nodes // 64) * 64
    pop, adj = {0: (8, 8), 1: (4, 4), 2: (2, 4), 3: (2, 4)}[storage]
    heat = aux = adj
    want = 2 * 19 * np_ * (pop + adj) + np_ * (1 + 10 * aux)  # flags; gamma, 4 bc, u, rho, dJ/dgamma
    if thermal:
        want += 2 * 7 * np_ * (heat + adj) + 13 * np_ * aux   # T, 7 collided, 3 coupling, sT, outflow
    got = C.lib().lbm_footprint_bytes(C.LBM_D3Q19, *shape, storage, thermal)
    # 64 bytes of results, and two sums of a block of at most 256 nodes, at least 32 of them in use
    assert want + 64 + 16 * nodes // 256 <= got <= want + 64 + 16 * nodes // 32
