"""Launch-shape entries on small volumes, on the CPU: an entry that sets any shape of the
adjoint keeps a small volume on the kernels it shapes, as the workspace they need shows."""
import pytest

import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import build as Bd


@pytest.fixture(autouse=True)
def clean_table():
    Bd.build()
    P.bsi_set_tile_configs([])
    yield
    P.bsi_set_tile_configs([])


@pytest.mark.parametrize("shape,spacing", [((64, 64, 64), (5, 5, 5)), ((40, 48, 50), (3, 4, 8)), ((128, 128, 128), (5, 5, 5))])
def test_adjoint_warps_keep_units_of_tile_planes(shape, spacing):
    def nbytes(**entry):
        P.bsi_set_tile_configs([entry] if entry else [])
        return P.bsi_adjoint_workspace_bytes(shape, spacing)

    tile_planes = max(nbytes(adj_zchunk=zc) for zc in range(3, 17))   # every length of a unit
    assert nbytes(adj_warps=2) == tile_planes
    assert nbytes(fwd_warps=2, fwd_strip_tiles=8) == nbytes() > tile_planes   # the forward's shapes leave the adjoint alone
