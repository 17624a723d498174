"""Rules of the kernels that no run shows reliably when they are broken: checked on the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_05454_b200", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cuh", ".cu"))))
def test_read_only_loads_are_of_data_that_no_kernel_of_a_step_writes(name):
    """A kernel of a step may be resident while its predecessors still write.  A read-only load has no order against those
    writes, not even behind the wait, so it is for weights and tables: the rotary table (c4), the normalisation's gains (gr) and the embedding's rows (src)."""
    for m in re.finditer(r"__ldg\(\s*([A-Za-z_][\w.>-]*)", _source(name)):
        assert m.group(1) in ("c4", "gr", "src"), f"{name}: __ldg of {m.group(1)}"


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cuh", ".cu"))))
def test_no_kernel_declares_data_of_the_step_read_only(name):
    """const T* __restrict__ lets the compiler choose the same read-only load by itself: for weights (embed, g, W0, W1) and for the
    lengths that the host copies before a plain launch (P, G)."""
    for m in re.finditer(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", _source(name)):
        assert m.group(1) in ("embed", "g", "W0", "W1", "P", "G"), f"{name}: {m.group(1)}"
