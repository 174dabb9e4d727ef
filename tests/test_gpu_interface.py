"""The reporting calls of the C interface: work split, probe and launch counter."""

import pytest

from paper_1807_11560_gb300 import Context

from helpers import ALPHA, S, SIGMA

pytestmark = pytest.mark.gpu


# (grid = band, plane parts per x1 column, quads per band item): the padded row pairs of
# the second axis (13 at band 16, 25 at 32) in items of at most 3 and 9; one plane item in 2D
@pytest.mark.parametrize("Ks,parts,quads", [((16, 16, 16), 5, 1), ((32, 32, 32), 3, 2), ((16, 16), 1, 1)])
def test_tiles_are_parts_and_quads(Ks, parts, quads):
    with Context(Ks, Ks, ALPHA, S, SIGMA, 1, precision="fp32") as ctx:
        assert ctx.tiles == (2, parts, quads)
