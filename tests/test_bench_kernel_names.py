"""The benchmark line names the FP64 kernel that ran: the default multiply, which the library
reports as the packed kernel, runs on the digit kernel."""
import importlib
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("number,forced,autotune,want", [
    (3, None, False, "dg"), (3, 3, False, "pk12"), (3, None, True, "dg or pk12"),
    (5, None, False, "g8"), (0, 0, False, "t16b2"), (-1, None, False, None)])
def test_kernel_that_ran(number, forced, autotune, want):
    sys.path.insert(0, ROOT)
    bench = importlib.import_module("bench")
    assert bench.fp64_kernel_run(number, forced, autotune) == want


def test_traffic_of_either_kernel_is_its_own():
    sys.path.insert(0, ROOT)
    bench = importlib.import_module("bench")
    a, b = (bench.MEASURED_TRAFFIC[(k, "water2048")] for k in ("dg", "pk12"))
    assert a["bytes"] != b["bytes"]
    for entry in (a, b):
        assert all(bench.kernel_source_sha(src, sec) is not None for src, sec, _ in entry["sections"])
    # an edit of one kernel does not concern the other's capture
    assert a["sections"][0][1] != b["sections"][0][1]
    assert bench.measured_traffic("dg or pk12", "water2048") is None
