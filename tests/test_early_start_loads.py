"""Kernels that start while the launch before still writes the placement
(programmatic dependent launches) must read it by ordinary loads: non-coherent
ones (__ldg, or a const __restrict__ pointer) ask for data that does not change
while the kernel runs. Checked on the source: a stale line would show on a GPU
by chance only."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1606_02162_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_positions_are_not_read_through_the_non_coherent_path():
    early = 0
    for name in ("layout.cu", "blocked.cu", "force.cuh"):
        src = _source(name)
        early += src.count("pdl_wait();")
        assert not re.search(r"__ldg\(\s*pos\b", src), name
        # a view of the launch's placement declared inside a kernel or helper
        assert not re.search(r"const P2\s*\*\s*__restrict__\s+pos\b", src), name
    assert early > 0
