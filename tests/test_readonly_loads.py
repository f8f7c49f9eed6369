"""Read-only loads (ld.global.nc) require data that no kernel writes while the
reading kernel runs.  The k-means kernels start as programmatic dependents,
before the kernel in front of them has ended, so of their buffers only the
caller's tokens may be read that way."""
import os
import re

import paper_2609_26425_gb300 as qwm

CSRC = os.path.join(os.path.dirname(os.path.abspath(qwm.__file__)), "csrc")


def test_fit_reads_only_the_tokens_through_the_readonly_path():
    with open(os.path.join(CSRC, "fit.cu")) as f:
        src = f.read()
    loads = re.findall(r"__ldg\(reinterpret_cast<[^>]*>\((.*?)\)", src)
    assert loads and src.count("__ldg(") == len(loads) and "global.nc" not in src
    for arg in loads:
        assert arg == "x" or arg.startswith("a.x "), arg
