"""The kernels of a time step run while their predecessor still writes: what they read
has to stay behind their wait. A pointer to const with __restrict__ lets the compiler
take what it points to as unchanging over the whole kernel, and load ahead of the wait.
So no device function has one, and no kernel that waits."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1907_00080_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))


def functions(text):
    """the function definitions of a source: from a line at the margin to the next
    brace that closes at the margin"""
    text = re.sub(r"//[^\n]*", "", text)
    return re.findall(r"^(?:template|static|__global__|__device__|inline)[^\n;]*\n(?:[^\n]*\n)*?}", text, re.M)


def test_functions_are_found():
    found = [f for s in SOURCES for f in functions(open(s).read())]
    for name in ("lb_tile", "load_pack", "stage_rows", "k_settle_batch", "k_hydro", "advance_unit", "forces_unit"):
        assert any(re.search(r"\b%s\(" % name, f.split("{")[0]) for f in found), name


@pytest.mark.parametrize("source", SOURCES, ids=os.path.basename)
def test_no_invariant_pointers_behind_a_wait(source):
    for f in functions(open(source).read()):
        kernel, waits = "__global__" in f.split("{")[0], "dep_wait(" in f
        if kernel and not waits:
            continue  # launched by itself
        assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", f), f.split("{")[0]
