"""Mixed-radix FFT passes at lengths whose schedules hold the radices that the
list of test_gpu_mixed_radix leaves out: ends of 4 and 6, and in float-float a
first radix of 10 and a middle one of 4."""
import pytest

import test_gpu_mixed_radix as base
from test_gpu_mixed_radix import B  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu
MORE_LENGTHS = [16, 24, 36, 84, 100]


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n", MORE_LENGTHS)
def test_axis_length(B, n, axis):  # noqa: F811
    base.test_axis_length(B, n, axis)
