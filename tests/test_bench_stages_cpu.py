"""The benchmark's counts of a stage's work, on the CPU: whatever launches a step is made of, they add up to its contractions."""
import pytest

import bench
from paper_2502_16927_b200 import workloads as wl

DENSE = ["gemm_descend", "gemm_ascend", "gemm_dy_lo", "gemm_dw_up", "gemm_dw2", "gemm_dw1", "gemm_dx", "gemm_dw_down"]
APART = ["gemm_expert1", "gemm_expert2", "gemm_dz", "gemm_dxg"]
PAIRS = ["fused_expert_mlp", "fused_expert_mlp_bwd"]


@pytest.mark.parametrize("name,calls", [
    ("medium", dict.fromkeys(DENSE + APART, 10)), ("medium", dict.fromkeys(DENSE + PAIRS, 10)),
    ("tiny", {"gemm_batch": 30, "gemm_ascend": 10, "fused_expert_mlp": 10, "fused_expert_mlp_bwd": 10}),
    ("tiny", {"gemm_batch": 40, "gemm_ascend": 10, "gemm_expert1": 10, "gemm_expert2": 10, "gemm_dz": 10})])
def test_stages_of_a_step_add_up(name, calls):
    w = wl.WORKLOADS[name]
    b = 2 if w.dtype == wl.DTYPE_BF16 else 4
    flops, size = bench.stage_work(w, b, calls, 10, True)
    assert sum(flops[n] * c / 10 for n, c in calls.items()) == pytest.approx(3.0 * bench.forward_flops(w), rel=1e-12)
    assert all(size[n] > 0 for n in calls)


def test_bytes_of_both_contractions_in_one_launch():
    for name in ("tiny", "medium", "decode"):
        w = wl.WORKLOADS[name]
        b = 2 if w.dtype == wl.DTYPE_BF16 else 4
        rows_and_weights = (2.0 * w.N * w.r + 2.0 * w.E * w.h * w.r) * b
        middle = w.N * w.h * (b + (1 if b == 2 else b))               # a and sigma', or dz and sigma'
        calls = {"fused_expert_mlp": 1, "fused_expert_mlp_bwd": 1}
        assert bench.stage_work(w, b, calls, 1, True)[1]["fused_expert_mlp"] == rows_and_weights + middle
        assert bench.stage_work(w, b, calls, 1, True)[1]["fused_expert_mlp_bwd"] == rows_and_weights + middle
        assert bench.stage_work(w, b, calls, 1, False)[1]["fused_expert_mlp"] == rows_and_weights
