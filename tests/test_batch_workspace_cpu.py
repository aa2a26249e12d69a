"""The adjoint's workspace, on the CPU: a batch needs the partial sums of units of
tile-planes only, a call of one volume also those of the plans it may take instead."""
import pytest

import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import build as Bd


@pytest.fixture(scope="module", autouse=True)
def lib():
    Bd.build()


def _tile_plane_bytes(shape, spacing):
    """The most over units of 3 to 16 tile-planes: (planes + 3) x 4 grid rows x 29 columns x 3 values each."""
    ncz, ncy, ncx = (-(-n // d) for n, d in zip(shape, spacing))
    units = lambda zc: -(-ncz // zc) * ncy * -(-(ncx + 3) // 29)
    floats = max(units(zc) * (zc + 3) * 4 * 29 * 3 for zc in range(3, 17))
    return 4 * (floats + 3 & ~3)


# (y-spacings outside 4..6: one tile-row per unit)
@pytest.mark.parametrize("shape,spacing", [((256, 256, 256), (12, 12, 12)), ((256, 256, 256), (64, 64, 64)), ((64, 64, 64), (8, 8, 8)),
                                           ((64, 65, 63), (3, 3, 3)), ((200, 200, 301), (7, 7, 7))])
def test_batch_workspace_is_that_of_its_units(shape, spacing):
    want = _tile_plane_bytes(shape, spacing)
    assert P.bsi_batched_adjoint_workspace_bytes([shape] * 2, [spacing] * 2) == 2 * want
    assert P.bsi_batched_adjoint_workspace_bytes([shape, (0, 3, 3)], [spacing, (2, 2, 2)]) == want
    one = P.bsi_adjoint_workspace_bytes(shape, spacing)
    assert P.bsi_batched_adjoint_workspace_bytes([shape], [spacing]) == one >= want
