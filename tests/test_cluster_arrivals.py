"""An arrival on another CTA's mbarrier names the cluster as its scope: without a scope it is one for the arriving CTA, and nothing then orders
what that CTA put into tensor memory before the MMAs of the CTA that waits.  No result shows that, so the sources are looked at."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_11357_b200", "csrc")


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_remote_arrivals_name_their_scope(name):
    code = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    remote = [i for i in re.findall(r"\bmbarrier\.arrive[.\w:]*", code) if ".shared::cluster" in i]
    assert all(re.match(r"mbarrier\.arrive(\.expect_tx)?\.(relaxed|release)\.cluster\.", i) for i in remote)
    assert remote or name != "async.cuh"
