"""bench.py: bytes and names of the kernels of a step by precision (the names
are those of nlc_timing_name)."""
import os
import re

import pytest

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
STEP = {"fp32": ["fused_lb", "fused_be"], "fp64": ["stress", "lb", "predict", "correct"],
        "fp32_qf64": ["stress", "lb", "predict", "correct"]}


@pytest.mark.parametrize("precision", STEP)
def test_kernels_of_a_step(precision):
    with open(os.path.join(ROOT, "paper_1907_13415_gb300", "csrc", "nlc_api.cu")) as f:
        names = re.search(r"names\[nlc::KID_COUNT\] = \{(.*?)\}", f.read(), re.S).group(1)
    step, kernels = bench.alg_bytes(precision)
    assert list(kernels) == STEP[precision]
    assert all(f'"{k}"' in names for k in kernels)
    _, gw, qw, _ = bench.PRECISIONS[precision]
    # Q is read by two kernels
    assert sum(kernels.values()) == step + 5 * qw
    assert bench.step_label(kernels) == "step (" + " + ".join(STEP[precision]) + ")"
