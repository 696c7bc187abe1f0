"""Passes hold as many operations as their kernels do (host-only): narrow groups are not
cut short by the coefficients of 4-qubit layers, gate lists not by layers they do not have."""
import pytest

import workloads as W
from paper_2202_07017_gb300 import C64, C128, sv_fusion_plan, sv_fusion_plan_reverse


@pytest.mark.parametrize("k", [2, 3])
def test_small_states_forward(k):
    """Every qubit of n = 10 is staged, so a second pass is a matter of capacity alone."""
    c, theta = W.hea(10, 4, 5), None
    c, theta = c
    assert sv_fusion_plan(c, theta, C64, k)[2] == 1
    assert sv_fusion_plan(W.qft(10), None, C64, k)[2] == 1


@pytest.mark.parametrize("dtype,k", [(C64, 2), (C64, 3), (C128, 2), (C128, 3), (C128, 4)])
def test_gate_lists_in_reverse(dtype, k):
    """70 rotations, their gradients and 63 CZs: below every limit of two passes."""
    c, theta = W.hea(10, 7, 6)
    assert sv_fusion_plan_reverse(c, theta, dtype, k)[1] <= 2
