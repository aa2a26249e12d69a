"""Small volumes of wide cells on the CPU: the forward's units may be parts of y-cells as
well as of z-cells; every row is written once and every access is in range."""
import pytest

import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import build as Bd


@pytest.fixture(scope="module", autouse=True)
def lib():
    Bd.build()


@pytest.mark.parametrize("shape,spacing", [((12, 61, 30), (57, 62, 43)), ((1, 64, 64), (64, 64, 64)), ((64, 64, 64), (12, 12, 12)), ((3, 7, 100), (4, 4, 9)),
                                           ((65, 33, 40), (24, 13, 24)), ((2, 90, 31), (20, 31, 10)), ((30, 30, 61), (16, 16, 8)), ((5, 17, 1000), (64, 5, 50))])
def test_parts_of_y_cells(shape, spacing):
    for op in ("forward", "adjoint"):
        n, msg = P.bsi_selfcheck_ranges([shape], [spacing], op, cover=True)
        assert n == 0, msg
