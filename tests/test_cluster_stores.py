"""A CTA's shared memory may be written by another CTA of its cluster only once it has started: the order of barrier and store in the
source of the kernels that do so (a violation is a race that a GPU run need not show)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_27527_b200", "csrc")


def functions(name):
    """Bodies of the functions of a source file (from a definition at the start of a line to the closing brace there)."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    return re.findall(r"^[A-Za-z_][^;{}]*\)\s*\{\n.*?^\}", text, re.M | re.S)


def test_maxima_wait_for_the_cluster_before_they_write_into_it():
    (write,) = [f for f in functions("nvfp4_device.cuh") if " cells_write(" in f.split("{")[0]]
    before = write.split("st.shared::cluster")[0]
    assert "barrier.cluster.wait" in before
    callers = [f for name in sorted(os.listdir(CSRC)) if name.endswith(".cu") for f in functions(name) if "cells_write<" in f]
    assert len(callers) == 2
    for f in callers:
        assert "__global__" in f.split("{")[0] and f.split("{", 1)[1].lstrip().startswith("cells_begin();")
