"""Which adjoint plan one volume takes, on the CPU, by the workspace it needs: units of
tile-planes where they are as short as cells' or fill the GPU better, cells' otherwise."""
import pytest

import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import build as Bd


@pytest.fixture(scope="module", autouse=True)
def lib():
    Bd.build()


def _tile_planes(shape, spacing):
    """A batch takes units of tile-planes only."""
    return P.bsi_batched_adjoint_workspace_bytes([shape] * 2, [spacing] * 2) // 2


@pytest.mark.parametrize("shape,spacing", [((3, 1, 882), (6, 2, 3)), ((2, 10, 2920), (7, 8, 1)), ((2, 2, 40), (5, 5, 5)),
                                           ((278, 195, 168), (6, 7, 4)), ((90, 92, 165), (3, 2, 8)),
                                           ((397, 215, 159), (14, 2, 8)), ((232, 148, 303), (7, 4, 8))])
def test_tile_planes(shape, spacing):
    assert P.bsi_adjoint_workspace_bytes(shape, spacing) == _tile_planes(shape, spacing)
    n, msg = P.bsi_selfcheck_ranges([shape], [spacing], "adjoint", cover=True)
    assert n == 0, msg


@pytest.mark.parametrize("shape,spacing", [((64, 64, 64), (5, 5, 5)), ((64, 64, 64), (3, 3, 3)), ((40, 1, 60), (5, 4, 3)),
                                           ((256, 256, 256), (8, 8, 8))])
def test_cells(shape, spacing):
    assert P.bsi_adjoint_workspace_bytes(shape, spacing) > _tile_planes(shape, spacing)
