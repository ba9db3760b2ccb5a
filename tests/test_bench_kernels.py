"""bench.py attributes a counter of tfkt_step_profiled to the kernel that ran."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


@pytest.mark.parametrize("path,first,second", [
    ("fused", ("fused_kernel", 10 * (2 * 1000 + 2 * 60)), ("fixup_kernel", None)),
    ("split", ("collide_kernel", 10 * (2 * 1000 + 60)), ("moments_kernel", 10 * (1000 + 60)))])
def test_kernel_and_bytes_behind_a_counter(path, first, second):
    m = bench.launch_models(path, 10, 1000, 60)
    assert m["fused"] == first and m["fixup"] == second


def test_two_pass_counters():
    m = bench.launch_models("two_pass", 10, 1000, 60)
    assert m["moments"] == ("moments_kernel", 10600) and m["step"] == ("collide_kernel", 20600)
