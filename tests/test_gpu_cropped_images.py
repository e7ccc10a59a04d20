"""Items of the tensor-core kernel that leave out an image's last R - 1 rows, whose windows wrap: equal parts of one image.  Remainders of 16 columns, odd image counts, planes that are no whole
quads, stacked taps, split contraction, 16-bit operands, virtual images.  Integer inputs: equal to the oracle bit for bit."""
import numpy as np
import pytest

from helpers import run_library
from test_gpu_padded import _run as run_padded
from test_gpu_strided import _reference, _run as run_strided
from workloads import small_integers

pytestmark = pytest.mark.gpu

CASES = [
    # N, C, H, W, K, R, S
    (32, 256, 14, 14, 256, 3, 3), (3, 128, 32, 32, 70, 7, 7), (5, 33, 13, 15, 130, 3, 3), (1, 48, 9, 31, 96, 2, 5),
    (7, 100, 11, 9, 65, 5, 3), (4, 160, 16, 16, 64, 3, 3), (3, 64, 40, 36, 33, 7, 7),           # (the last two: stacked taps)
    (2, 130, 8, 30, 129, 8, 2), (150, 32, 7, 7, 200, 3, 3), (2, 64, 24, 24, 80, 3, 3),
]


@pytest.mark.parametrize("case", CASES)
def test_cropped_items_exact_on_integers(oracle, monkeypatch, case):
    N, C, H, W, K, R, S = case
    monkeypatch.setenv("CONV2D_B200_TF32_CROP", "2")
    monkeypatch.setenv("CONV2D_B200_TF32_RESIDENT", "0")
    x, w = small_integers((N, C, H, W), 1701), small_integers((K, C, R, S), 1702)
    y_ref, _ = oracle.conv2d_oracle(x, w)
    for entry, algo in (("general", 2), ("bf16", 3)):
        np.testing.assert_array_equal(run_library(x, w, entry=entry, algo=algo).astype(np.float64), y_ref)


def test_cropped_items_on_virtual_images(oracle, monkeypatch):
    monkeypatch.setenv("CONV2D_B200_TF32_CROP", "2")
    monkeypatch.setenv("CONV2D_B200_TF32_RESIDENT", "0")
    for N, C, H, W, K, R, S, pad in ((3, 70, 12, 16, 130, 5, 5, 2), (5, 64, 7, 7, 96, 3, 3, 1)):
        x, w = small_integers((N, C, H, W), 1703), small_integers((K, C, R, S), 1704)
        y_ref, _ = oracle.conv2d_oracle(np.pad(x, ((0, 0), (0, 0), (pad, pad), (pad, pad))), w)
        np.testing.assert_array_equal(run_padded(x, w, pad, pad, 2).astype(np.float64), y_ref)
    for N, C, H, W, K, R, S, pad, st in ((3, 40, 15, 13, 130, 5, 5, 2, 2), (5, 64, 16, 16, 80, 3, 3, 1, 2), (3, 24, 20, 22, 70, 7, 7, 0, 3)):
        x, w = small_integers((N, C, H, W), 1705), small_integers((K, C, R, S), 1706)
        y_ref, _ = _reference(oracle, x, w, pad, pad, st)
        np.testing.assert_array_equal(run_strided(x, w, pad, pad, st, 2)[0].astype(np.float64), y_ref)


@pytest.mark.parametrize("case", [
    # at most 64 filters, no split: stores of quads, of pairs and of single pixels; blocks of 32 columns whose number is odd, the last one half full;
    # more items than SMs
    (80, 64, 16, 16, 64, 5, 5), (75, 64, 14, 14, 33, 5, 5), (80, 64, 15, 17, 64, 5, 5), (160, 64, 14, 16, 20, 5, 5), (160, 48, 14, 14, 64, 3, 3), (150, 40, 10, 18, 61, 3, 3),
])
def test_cropped_items_of_few_filters_exact_on_integers(oracle, monkeypatch, case):
    import paper_1705_10591_b200 as lib
    N, C, H, W, K, R, S = case
    monkeypatch.setenv("CONV2D_B200_TF32_CROP", "2")
    monkeypatch.setenv("CONV2D_B200_TF32_RESIDENT", "0")
    x, w = small_integers((N, C, H, W), 1707), small_integers((K, C, R, S), 1708)
    y_ref, _ = oracle.conv2d_oracle(x, w)
    for entry, algo in (("general", 2), ("bf16", 3)):
        plan = lib.conv2d_fwd_plan_describe(N, C, H, W, K, R, S, algo)
        assert plan["crop"] == 1 and plan["ksplit"] == 1
        np.testing.assert_array_equal(run_library(x, w, entry=entry, algo=algo).astype(np.float64), y_ref)
