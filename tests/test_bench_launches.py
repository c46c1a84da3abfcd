"""bench.py's count of its own kernels against the launch list of its timed window."""
import os
import re

import bench

LIST = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "profiles", "launches_c4_bench.md")


def test_step_kernels_counts_the_launch_list():
    """Steps 91 to 110, with sweeps of both kinds at 100 and 110 and an exchange at 100."""
    text = open(LIST).read()
    assert "20 steps from step 91" in text
    own = sum(int(n) for n in re.findall(r"^cph::.*?\s(\d+)\s+[\d.]+\s+[\d.]+%$", text, re.M))
    assert own == 194
    assert sum(bench.step_kernels(t) for t in range(91, 111)) == own
    assert [bench.step_kernels(t) for t in (0, 91, 100, 110)] == [9, 9, 17, 15]
    assert bench.step_kernels(91, any_ordered=True) == 12
