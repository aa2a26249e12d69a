"""The row-copy adjoint's staged rows on the CPU: a volume whose last x-tile is cut and
falls on the last lane of a strip of 32 tiles (widths just under 58, 87 and 116 tiles)
fills its staged row, so the zeros behind the row must end inside the row's slot."""
import ctypes

import pytest

import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import bsi as B
from paper_2004_05962_gb300 import build as Bd


@pytest.fixture(scope="module", autouse=True)
def lib():
    Bd.build()
    return B.library()


def _violations(shapes, spacings, grad):
    arr = B._instances(shapes, spacings)
    for i in range(len(shapes)):
        arr[i].grad_field = grad   # (only its alignment is looked at)
    msg = ctypes.create_string_buffer(256)
    n = B.library().bsi_selfcheck_ranges(arr, len(shapes), 2, 0, msg, 256)
    return n, msg.value.decode()


@pytest.mark.parametrize("grad", [256, 260], ids=["aligned", "unaligned"])
@pytest.mark.parametrize("dx", range(1, 9))
def test_zeros_after_a_staged_row_stay_in_its_slot(dx, grad):
    for k in (2, 3, 4):
        for c in range(dx):
            shape, spacing = (3, 3, 29 * k * dx - c), (3, 3, dx)
            n, msg = _violations([shape, shape], [spacing, spacing], grad)   # a batch: always units of tile-planes
            assert n == 0, (shape, spacing, msg)


@pytest.mark.parametrize("shape,spacing", [((300, 300, 347), (6, 6, 6)), ((300, 300, 405), (7, 7, 7)), ((300, 300, 463), (8, 8, 8)),
                                           ((300, 300, 289), (5, 5, 5))])
def test_single_volumes(shape, spacing):
    """Large enough for units of tile-planes in a call of one volume."""
    n, msg = P.bsi_selfcheck_ranges([shape], [spacing], "adjoint", cover=False)
    assert n == 0, msg
