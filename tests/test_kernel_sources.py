"""Promises that kernel signatures make to the compiler, read from the sources
(CPU only)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2406_18356_gb300", "csrc")


def _parameters(source, function):
    """The parameter list of a function's definition, one string each."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, source)).read())
    at = re.search(rf"\b{function}\s*\(([^{{;]*?)\)\s*\{{", text)
    assert at, function
    return [" ".join(p.split()) for p in at.group(1).split(",")]


# degridding takes vis_out == vis_obs (rows_apart in mstep.cu), and a pointer
# that is __restrict__ may be read through the non-coherent path
@pytest.mark.parametrize("function", ["degrid_item", "degrid_kernel"])
def test_degridding_promises_no_distinct_rows(function):
    params = _parameters("grid_kernels.cu", function)
    for name in ("obs", "out"):
        (decl,) = [p for p in params if re.search(rf"\b{name}$", p)]
        assert "__restrict__" not in decl, decl
