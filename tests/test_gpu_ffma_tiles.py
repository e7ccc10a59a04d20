"""fp32 general kernel: every segment length (adjacent outputs of a thread) and the planner's choice give the same bits and
match the oracle within the fp32 bound; the launcher picks the length, the filter groups and the block size by an estimate."""
import numpy as np
import pytest

from helpers import FFMA_TOL, assert_parity, run_library
from workloads import uniform

pytestmark = pytest.mark.gpu
ALGO_FFMA = 1

# N, C, H, W, K, R, S: output maps of 30 and 26 columns (five segments of 6; four of 7), 54 wide, 12 x 12 (two of 6), a ragged
# filter count, a map wide enough for column strips, one row of channels left over
SHAPES = [
    (2, 12, 32, 32, 70, 3, 3),
    (2, 6, 32, 32, 64, 7, 7),
    (1, 10, 20, 56, 24, 3, 3),
    (3, 20, 14, 14, 130, 3, 3),
    (2, 9, 17, 70, 40, 5, 5),
    (2, 16, 9, 31, 64, 1, 1),
    (1, 9, 10, 150, 20, 3, 3),
]


@pytest.mark.parametrize("dims", SHAPES)
def test_ffma_segment_lengths_agree(oracle, dims, monkeypatch):
    N, C, H, W, K, R, S = dims
    x, w = uniform((N, C, H, W), 1201), uniform((K, C, R, S), 1202)
    y_ref, yabs = oracle.conv2d_oracle(x, w)
    y0 = run_library(x, w, entry="general", algo=ALGO_FFMA)
    assert_parity(y0, y_ref, yabs, FFMA_TOL, f"fp32, planner's segments {dims}")
    for length in (6, 7, 8):
        monkeypatch.setenv("CONV2D_B200_FFMA_SEGMENT", str(length))
        np.testing.assert_array_equal(run_library(x, w, entry="general", algo=ALGO_FFMA), y0, err_msg=f"segments of {length} {dims}")
