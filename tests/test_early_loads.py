"""Kernels that may start before the kernels ahead of them have ended read what those wrote through loads that stay behind the wait
(load_behind_wait in csrc/async.cuh).  The compiler may move __ldcg and __ldcs across it; __ldg and a plain read through a const
__restrict__ pointer promise data that nobody writes while the kernel exists.  No result shows that, so the sources are looked at."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_11357_b200", "csrc")


@pytest.mark.parametrize("name", ["repack.cu", "gemv.cu", "gemm.cu"])
def test_loads_of_earlier_kernels_results_stay_behind_the_wait(name):
    code = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    assert "grid_dependency_wait()" in code
    assert re.findall(r"\b__ld(?:g|cg|cs|ca)\s*\(", code) == []
    # the packed weights alone are read ahead of the wait and are nobody's result there
    assert [p for p in re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", code) if p != "blob"] == []
