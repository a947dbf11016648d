"""Kernels that start while their predecessor runs (launch_chained) read what it writes by
ordinary loads: no __ldg and no const __restrict__ pointer, whose loads may take the
read-only path, which is defined only for memory that nobody writes while the kernel lives.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2506_07430_gb300", "csrc")


def _function(name, source):
    """The text of function `name` in csrc/`source`: its parameters and its body."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, source)).read())
    start = re.search(r"\b%s\([^;{]*\{" % name, text)
    assert start, name
    depth, end = 0, start.end() - 1
    while True:
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        end += 1
        if depth == 0:
            return text[start.start():end]


@pytest.mark.parametrize("source,name,written", [
    ("sigma_rows.cu", "rows_d_items", ["x"]),
    ("sigma_rows.cu", "sigma_rows_cta", ["x", "xr", "y"]),
    ("recursion.cu", "cheb_update_cta", ["s", "c", "prev"]),
    ("recursion.cu", "k_cheb_update", ["s", "c", "prev"]),
    ("sigma_tc.cu", "row_scale", ["rowmax", "amax"]),
    ("sigma_tc.cu", "k_rowpass", ["rscale"]),
])
def test_predecessor_output_is_read_by_ordinary_loads(source, name, written):
    text = _function(name, source)
    for w in written:
        assert not re.search(r"__ldg\(\s*&?\(?\s*(p\.|m\.)?%s\b" % w, text), (name, w)
        assert not re.search(r"__restrict__\s+%s\b" % w, text), (name, w)
