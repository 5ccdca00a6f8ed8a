"""Strength thresholds that are no positive number: a coupling is weak when a < theta max,
which no coupling is against a NaN or a negative bound, so the hierarchy is that of the
threshold 0, in the oracle and on the device.
"""
import numpy as np
import pytest

from test_gpu_amg_setup import compare_hierarchies, options_case, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("theta", [float("nan"), -float("nan"), -0.5, -float("inf")])
def test_no_bound_keeps_every_coupling(torch_cuda, theta):
    assert compare_hierarchies(options_case(4, theta), 5.0) == compare_hierarchies(options_case(4, 0.0), 5.0)
