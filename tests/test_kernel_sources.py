"""Rules of synchronisation that a passing run cannot show, read from the kernels' sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1811_11722_gb300", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("name", sorted(os.path.basename(p) for p in glob.glob(os.path.join(CSRC, "*.cu*"))))
def test_no_barrier_over_the_lanes_that_happen_to_be_there(name):
    """__activemask() gives the lanes that are converged, not those that have to take part."""
    assert "__activemask" not in source(name)
