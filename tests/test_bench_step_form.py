"""The bench line's roofline bytes of the fine-level GMRES(3) step are the vector
passes of the kernels that run for the precision and the march option, not a
fixed fraction of a count made for others."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("precision,march,passes", [
    ("mixed", -1, 5), ("mixed", 1, 5), ("mixed-ff", -1, 5),   # x, b; x, b -> x'
    ("mixed", 0, 15),      # r 3, v1 2, v2 2, Gram sums of r, v1, v2 3, x + r, v1, v2 5
    ("fp64", 1, 16), ("fp64", -1, 28), ("fp64", 0, 28)])
def test_passes_of_a_step(precision, march, passes):
    sys.path.insert(0, ROOT)
    import bench
    n, form = bench.gmres_step_form(precision, march)
    assert n == passes
    assert ("march" in form) == (passes in (5, 16))
