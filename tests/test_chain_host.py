"""Sources of the kernels launched as programmatic dependents (no GPU).  Such a kernel is resident while
the launch before it still writes levels, sources or the right-hand side, so it may neither read them
through the read-only path nor through pointers declared unaliased: the compiler need not keep
those accesses behind the wait for the predecessor."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_17057_gb300", "csrc")


def code(name):
    with open(os.path.join(CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", fh.read(), flags=re.S))


CHAINED = sorted(f for f in os.listdir(CSRC)
                 if f.endswith((".cu", ".cuh")) and re.search(r"\b(chain_wait|launch_chained)\b", code(f)))


def test_the_list_holds_every_marching_kernel():
    assert {"k_direct.cuh", "k_march2d.cuh", "k_march3d.cuh", "k_march2d_tb.cu", "k_march2d_tb_nse.cu"} <= set(CHAINED)


@pytest.mark.parametrize("name", CHAINED)
def test_no_read_only_or_unaliased_access(name):
    found = re.findall(r"__ldg|ld\.global\.nc|__restrict(?:__)?\b|\brestrict\b", code(name))
    assert not found, (name, found)
