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


@pytest.mark.parametrize("name,kernel,written_meanwhile", [("cv_device.cuh", "cv_fit_kernel", ["a"]),
                                                           ("cv.cu", "cv_adam_kernel", ["grad_part", "a", "m1", "m2"])])
def test_overlapped_kernels_load_what_the_one_before_writes_afresh(name, kernel, written_meanwhile):
    """A kernel that is resident while the one before it still writes may not declare that memory read-only for
    its lifetime, and reads it from L2 where the load stands: after griddepcontrol.wait, before it lets
    the next writer up."""
    text = source(name)
    head, body = re.search(kernel + r"\(([^)]*)\)\s*\{(.*?)\n\}\n", text, re.S).groups()
    params = [p.strip() for p in head.split(",")]
    for q in written_meanwhile:
        decl = next(p for p in params if re.search(r"\b%s$" % q, p))
        assert "const" not in decl and "__restrict__" not in decl, decl
        loads = [m.start() for m in re.finditer(r"ld_fresh4?\(%s\b" % q, body)]
        assert loads and min(loads) > body.index("grid_wait()")
        assert not re.search(r"(?<![\w.])%s\[[^\]]*\](?!\s*=[^=])" % q, body), "a plain load of %s" % q
    if kernel == "cv_fit_kernel":  # the next Adam step writes a
        assert body.index("grid_launch_next()") > body.rindex("ld_fresh4(a")
