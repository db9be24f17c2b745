"""The CPU side of bench.py."""
import pytest

import bench
from paper_2411_17178_b200 import workloads as wl


@pytest.mark.parametrize("workload", [wl.WORKLOADS[1], wl.small_workload((1, 2, 3, 4, 6), index=91)], ids=["layers", "sampled-rows"])
def test_the_oracle_is_timed_however_short_the_budget(workload):
    """Making the inputs is not on the clock, and at least one layer or one batch of rows is run."""
    flop, seconds, _ = bench.oracle_sample(workload, 0.0)
    assert flop > 0 and seconds > 0
