"""Rows of the SES interior whose chord FP32 cannot express: R^2 overflows (an atom that covers the grid from 3e19 A
away), or 1 / spacing does (a grid of subnormal spacing).  The exact test decides every point, as the oracle does."""
import numpy as np
import pytest

import oracle
from test_gpu_ses import gpu_ses

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("radius,inside", [(3.3e19, True), (2.7e19, False)])
def test_overflowing_radius(axis, radius, inside):
    x = np.array([[0.0, 0.0, 0.0, radius], [3.0, 4.0, 5.0, 1.5]], np.float32)
    x[0, axis] = 3e19
    origin, dims = np.zeros(3, np.float32), np.array((37, 11, 9), np.int32)
    ref = oracle.ses(x, origin, np.float32(0.7), dims, probe=0.0)
    got = gpu_ses(x, origin, 0.7, dims, 0.0)
    assert (ref.sas.mean() == 1.0) if inside else (0.0 < ref.sas.mean() < 1.0)
    np.testing.assert_array_equal(got["sas"], ref.sas)


def test_subnormal_spacing():
    x = np.array([[0.0, 0.0, 0.0, 1.5]], np.float32)
    origin, dims = np.zeros(3, np.float32), np.array((37, 5, 4), np.int32)
    ref = oracle.ses(x, origin, np.float32(1e-39), dims, probe=0.0)
    got = gpu_ses(x, origin, np.float32(1e-39), dims, 0.0)
    assert ref.sas.mean() == 1.0
    np.testing.assert_array_equal(got["sas"], ref.sas)
