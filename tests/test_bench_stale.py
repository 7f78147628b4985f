"""The benchmark attaches no ncu counter of an earlier version of a kernel to its times."""
import types

import pytest

import bench


@pytest.mark.parametrize("kernel", sorted(bench._FP64_PIPE_BUSY))
def test_no_counter_of_a_changed_kernel_is_reported(monkeypatch, kernel):
    args = types.SimpleNamespace(workload="large_4000", steps=20, warmup=5)
    monkeypatch.setattr(bench, "_COUNTERS_STALE", {"fp64": set(), "fp32mix": set()})
    assert bench._fp64_pipe_busy(kernel) == bench._FP64_PIPE_BUSY[kernel]
    assert bench._traffic(kernel, "fp64", args)[0] is not None
    monkeypatch.setattr(bench, "_COUNTERS_STALE", {"fp64": {kernel}, "fp32mix": set()})
    assert bench._fp64_pipe_busy(kernel) is None
    assert bench._traffic(kernel, "fp64", args) == (None, "counters stale")


def test_every_reported_pipe_share_goes_through_the_check():
    src = open(bench.__file__).read()
    assert src.count("_FP64_PIPE_BUSY") == 2          # the table and the function that looks into it
