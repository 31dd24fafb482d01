"""bench.py's account of a step: the kernel that ran, its steps per launch, and the bytes it moves."""
import pytest

import bench


class _Cavity:
    """mclbm_step_launches of a cavity on the step-by-step, grid-resident or cluster-resident kernel."""

    def __init__(self, kind):
        self.kind = kind

    def step_launches(self, n):
        if self.kind == "tma":
            return bench.step_launches(n)
        whole, left = divmod(n, 16384)
        if self.kind == "cluster":
            return whole + (left > 0)
        return whole + (left > 1) + left % 2


def _line(kind, n, step_time=2.8e-6, state=14.2e6):
    return bench.step_roofline(_Cavity(kind), n, step_time, state, 6763.6, "measured", 0.5, 2)


def test_one_launch_per_step_is_measured_against_memory():
    r = _line("tma", 1000, step_time=40e-6, state=226e6)
    assert (r["bound"], r["kernel"], r["steps_per_launch"]) == ("hbm", "step_pair_tma_kernel", 1)
    assert r["traffic"] == 0.5 and r["nodes_per_thread"] == 2
    assert r["achieved"] == pytest.approx(226e6 / 40e-6 / 1e9)
    assert r["frac"] == pytest.approx(r["achieved"] / 6763.6)


@pytest.mark.parametrize("kind,kernel,n,per", [
    ("grid", "step_resident_kernel", 1000, 1000), ("grid", "step_resident_kernel", 1001, 1000),
    ("grid", "step_resident_kernel", 40000, 16384), ("cluster", "step_cluster_kernel", 1001, 1001),
    ("cluster", "step_cluster_kernel", 40000, 16384)])
def test_a_resident_kernel_moves_the_state_once_per_launch(kind, kernel, n, per):
    r = _line(kind, n)
    assert (r["bound"], r["kernel"], r["steps_per_launch"]) == ("latency", kernel, per)
    assert r["traffic"] is None and r["nodes_per_thread"] == 1
    assert r["launch_us"] == pytest.approx(2.8 * per)
    assert r["bytes_per_launch"] == 14.2e6
    assert r["achieved"] == pytest.approx(14.2e6 / (2.8e-6 * per) / 1e9)


def test_reduction_launches():
    assert bench.reduction_launches(256) == 5 and bench.reduction_launches(257) == 6
