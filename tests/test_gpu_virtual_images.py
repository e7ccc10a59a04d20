"""Padding and strides computed on virtual images by the tensor-core kernel: rows whose zeros are shared with the next row,
quads and single pixels, every phase of a stride, few channels (phases as staged channels), resident and streamed filters,
stacked taps, split contraction.  Integer inputs are exact in TF32: the result has to equal the oracle's bit for bit."""
import numpy as np
import pytest

from test_gpu_padded import _run as run_padded
from test_gpu_strided import _reference, _run as run_strided
from workloads import small_integers, uniform
from helpers import TF32_TOL, assert_parity

pytestmark = pytest.mark.gpu

PADDED = [
    # N, C, H, W, K, R, S, pad_h, pad_w
    (3, 17, 12, 16, 20, 3, 3, 1, 1), (2, 16, 9, 15, 64, 3, 3, 1, 1), (2, 33, 7, 6, 130, 3, 3, 1, 1),
    (1, 20, 13, 20, 70, 5, 5, 2, 2), (2, 64, 8, 12, 40, 5, 5, 2, 2), (2, 40, 7, 8, 64, 7, 7, 3, 3),     # stacked taps
    (1, 16, 6, 8, 24, 3, 3, 4, 5), (1, 8, 4, 4, 9, 2, 2, 3, 7), (2, 5, 8, 12, 10, 4, 2, 0, 1),          # more zeros than the filter needs
    (32, 256, 7, 7, 256, 3, 3, 1, 1),                                                                   # split contraction
    (1, 16, 40, 200, 16, 7, 7, 3, 3), (4, 2, 30, 44, 8, 3, 3, 1, 1),
]
STRIDED = [
    # N, C, H, W, K, R, S, pad_h, pad_w, stride
    (2, 16, 14, 16, 24, 3, 3, 1, 1, 2), (1, 40, 15, 13, 130, 5, 5, 2, 2, 2), (2, 20, 17, 19, 66, 7, 7, 3, 3, 3),
    (1, 33, 16, 20, 64, 3, 3, 1, 1, 4), (2, 3, 31, 30, 64, 7, 7, 3, 3, 2), (1, 4, 21, 24, 16, 3, 3, 1, 1, 3),
    (2, 1, 40, 36, 5, 5, 5, 2, 2, 4), (1, 64, 9, 9, 32, 1, 1, 0, 0, 3), (1, 18, 12, 14, 12, 2, 5, 0, 2, 4),
    (16, 256, 14, 14, 256, 3, 3, 1, 1, 2), (2, 24, 33, 8, 100, 3, 1, 1, 0, 2), (1, 16, 20, 20, 8, 3, 3, 0, 0, 8),
    (1, 9, 64, 70, 12, 5, 3, 2, 1, 5),
    (32, 16, 56, 56, 20, 3, 3, 1, 1, 2),     # rows of 30 columns instead of 32: fewer, smaller items
]


@pytest.mark.parametrize("case", PADDED)
def test_padded_exact_on_integers(oracle, monkeypatch, case):
    N, C, H, W, K, R, S, ph, pw = case
    x, w = small_integers((N, C, H, W), 1601), small_integers((K, C, R, S), 1602)
    y_ref, _ = oracle.conv2d_oracle(np.pad(x, ((0, 0), (0, 0), (ph, ph), (pw, pw))), w)
    for mode in ("2", "0"):                      # on virtual images; as patches of the image (or extended)
        monkeypatch.setenv("CONV2D_B200_TF32_VIRT", mode)
        np.testing.assert_array_equal(run_padded(x, w, ph, pw, 2).astype(np.float64), y_ref)


@pytest.mark.parametrize("case", [
    (5, 80, 65, 33, 48, 3, 3, 1, 1),         # a contraction that only virtual images would split
    (21, 16, 37, 184, 4, 7, 7, 3, 3),        # a clear difference of the estimates: a long halo
    (2, 272, 51, 247, 11, 3, 3, 1, 1),       # ... rows staged pixel by pixel
])
def test_padded_layers_left_to_patches(oracle, case):
    N, C, H, W, K, R, S, ph, pw = case
    x, w = small_integers((N, C, H, W), 1607), small_integers((K, C, R, S), 1608)
    y_ref, _ = oracle.conv2d_oracle(np.pad(x, ((0, 0), (0, 0), (ph, ph), (pw, pw))), w)
    np.testing.assert_array_equal(run_padded(x, w, ph, pw, 2).astype(np.float64), y_ref)


@pytest.mark.parametrize("case", STRIDED)
def test_strided_exact_on_integers(oracle, case):
    N, C, H, W, K, R, S, ph, pw, st = case
    x, w = small_integers((N, C, H, W), 1603), small_integers((K, C, R, S), 1604)
    y_ref, _ = _reference(oracle, x, w, ph, pw, st)
    y, ws = run_strided(x, w, ph, pw, st, 2)
    np.testing.assert_array_equal(y.astype(np.float64), y_ref)
    np.testing.assert_array_equal(run_strided(x, w, ph, pw, st, 2, flags=1, ws=ws)[0], y)       # filters re-ordered before
    x, w = uniform((N, C, H, W), 1605), uniform((K, C, R, S), 1606)
    y_ref, yabs = _reference(oracle, x, w, ph, pw, st)
    assert_parity(run_strided(x, w, ph, pw, st, 2)[0], y_ref, yabs, TF32_TOL, f"strided {case}")
