"""FP32-basis projection over the vector counts at which its warp sums change shape.

The last group of a CTA holds 1 to 8 vectors, summed across the warp 4, 8 or 16 values at
a time, and the last CTA sums the partials two or four columns at a time over one to
several rounds of CTAs.  Check and bound are those of test_gpu_gram_schmidt_f32.py.
"""
import pytest

import test_gpu_gram_schmidt_f32 as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 4098, 700002])
@pytest.mark.parametrize("nvec", [1, 2, 3, 4, 5, 7, 8, 9, 12, 16, 17, 30, 64])
@pytest.mark.parametrize("mode", [0, 1])
def test_projection_group_sizes(n, nvec, mode):
    T.test_projection_error_bound(n, nvec, mode)
