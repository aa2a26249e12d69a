"""The host self-check over the units that calls of one volume launch: parts of
tile-planes in rows and in blocks, BF16's narrower strips, volumes alone in their launch."""
import pytest

import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import build as Bd


@pytest.fixture(scope="module", autouse=True)
def lib():
    Bd.build()


# few units: parts; rows on and off 16-byte boundaries; planes that do not divide into the parts
VOLUMES = [((65, 64, 64), (5, 5, 5)), ((14, 24, 240), (7, 4, 5)), ((64, 64, 64), (4, 4, 4)), ((30, 30, 128), (6, 6, 2)), ((9, 12, 200), (64, 2, 6)), ((1, 40, 32), (8, 8, 3)),
           ((10, 30, 116), (5, 6, 7)), ((12, 18, 252), (4, 6, 3)), ((13, 9, 41), (6, 3, 8)), ((5, 9, 64), (9, 4, 4))]


@pytest.mark.parametrize("op", ["forward", "forward_bf16", "scalar", "scalar_bf16", "resample", "resample_grad"])
def test_parts(op):
    for shape, spacing in VOLUMES:
        n, msg = P.bsi_selfcheck_ranges([shape], [spacing], op, cover=True)
        assert n == 0, (shape, spacing, msg)


@pytest.mark.parametrize("op", ["forward", "forward_bf16", "adjoint", "scalar", "resample_grad"])
def test_a_volume_alone_in_its_launch(op):
    """Two volumes whose kernels differ: each takes a launch of its own."""
    n, msg = P.bsi_selfcheck_ranges([(12, 20, 60), (9, 20, 60)], [(5, 5, 5), (3, 5, 13)], op, cover=True)
    assert n == 0, msg
