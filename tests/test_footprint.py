"""The device memory of an instance (gdg_footprint), which is what a server admits requests by, stays within what it was before
the stage kept boundary states, flux differences, indicator terms and its input by slots."""
import pytest

from paper_2402_04514_gb300 import assembly
from paper_2402_04514_gb300.gdg import footprint


@pytest.mark.parametrize("cells,degree,bytes_before", [
    ((200,), 1, 238080), ((8, 8), 1, 295168), ((64, 64), 1, 18381824), ((33, 47), 2, 26223616), ((48, 48), 3, 110229504),
    ((4, 4), 2, 502272), ((16, 16, 16), 1, 73294848), ((6, 6, 6), 2, 34524672), ((2, 2, 2), 1, 521728)])
def test_footprint_has_not_grown(cells, degree, bytes_before):
    P = {1: assembly.assemble_1d, 2: assembly.assemble_2d, 3: assembly.assemble_3d}[len(cells)](*cells, degree)
    assert footprint(P) <= bytes_before
