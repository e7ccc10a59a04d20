"""Virtual images whose rows are no whole quads: the producers load single pixels, before or after they wait for the stage (before where
every stage has a producer group of its own).  Both forms for at most 64 filters, stacked taps or not, and more filters alone and in
clusters; one item per block and several, channels and columns that leave remainders.  Integers: equal to the definition bit for bit."""
import numpy as np
import pytest

from test_gpu_padded import _run as run_padded
from test_gpu_strided import _reference, _run as run_strided
from workloads import small_integers

pytestmark = pytest.mark.gpu

CASES = [
    # N, C, H, W, K, R, S, padding, stride
    (3, 64, 13, 15, 64, 3, 3, 1, 1), (2, 64, 55, 55, 64, 3, 3, 1, 1), (16, 61, 55, 55, 33, 3, 3, 1, 1), (4, 48, 21, 23, 40, 3, 3, 1, 1),
    (3, 64, 31, 33, 48, 5, 5, 2, 1), (3, 64, 61, 63, 48, 5, 5, 2, 1), (40, 48, 13, 15, 17, 5, 5, 2, 1),           # stacked taps
    (2, 70, 13, 15, 130, 3, 3, 1, 1), (9, 70, 41, 43, 130, 3, 3, 1, 1),                                           # a cluster; more than 64 filters
    (2, 40, 21, 23, 70, 3, 3, 1, 2), (5, 24, 20, 22, 50, 3, 3, 0, 3), (8, 40, 61, 63, 64, 3, 3, 1, 2), (3, 33, 15, 17, 64, 3, 3, 1, 2),
]


@pytest.mark.parametrize("case", CASES)
def test_single_pixels_exact_on_integers(oracle, case):
    N, C, H, W, K, R, S, pad, stride = case
    x, w = small_integers((N, C, H, W), 1951), small_integers((K, C, R, S), 1952)
    if stride == 1:
        y_ref, _ = oracle.conv2d_oracle(np.pad(x, ((0, 0), (0, 0), (pad, pad), (pad, pad))), w)
        y = run_padded(x, w, pad, pad, 2)
    else:
        y_ref, _ = _reference(oracle, x, w, pad, pad, stride)
        y = run_strided(x, w, pad, pad, stride, 2)[0]
    np.testing.assert_array_equal(y.astype(np.float64), y_ref)
