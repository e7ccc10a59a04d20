"""fp32 general kernel, split into segments of output rows numbered through the batch: blocks that cross images, rows of any
alignment (a staged row then starts 0 to 3 floats into its place), column strips of wide maps, filter counts that fill no
group, channel counts that fill no channel block, tensors whose last 16-byte piece is short.  Integer inputs: every sum is
exact, so the result has to equal the oracle's bit for bit."""
import numpy as np
import pytest

from helpers import run_library
from workloads import small_integers

pytestmark = pytest.mark.gpu
ALGO_FFMA = 1

# N, C, H, W, K, R, S
SHAPES = [(3, 9, 8 + h, 13 + w, 11, 3, 3) for h in range(2) for w in range(4)]
SHAPES += [
    (40, 3, 4, 5, 9, 3, 3), (70, 2, 3, 3, 17, 3, 3),                  # blocks over many images, one output per image
    (1, 17, 11, 131, 20, 3, 3), (2, 5, 6, 260, 8, 5, 5), (1, 4, 9, 333, 3, 7, 7),     # column strips
    (2, 33, 7, 9, 130, 1, 1), (1, 7, 5, 6, 1, 2, 2), (2, 10, 12, 11, 40, 4, 4), (1, 3, 15, 15, 65, 7, 7),
    (1, 1, 5, 5, 8, 5, 5), (5, 13, 1, 31, 16, 1, 1), (90, 2, 7, 8, 3, 7, 7), (100, 3, 5, 5, 8, 5, 5),
]


@pytest.mark.parametrize("length", [None, "8", "7", "6"])      # chosen by the launcher; forced
@pytest.mark.parametrize("dims", SHAPES)
def test_exact_on_integers(oracle, monkeypatch, dims, length):
    N, C, H, W, K, R, S = dims
    if length is not None:
        monkeypatch.setenv("CONV2D_B200_FFMA_SEGMENT", length)
    x, w = small_integers((N, C, H, W), 1501), small_integers((K, C, R, S), 1502)
    y_ref, _ = oracle.conv2d_oracle(x, w)
    np.testing.assert_array_equal(run_library(x, w, entry="general", algo=ALGO_FFMA).astype(np.float64), y_ref)


def test_non_finite_pixels_stay_in_their_windows(oracle):
    """What lies beside a row or behind the tensor in shared memory must not reach an output."""
    x, w = small_integers((2, 9, 10, 15), 1503), np.abs(small_integers((12, 9, 3, 3), 1504)) + 1
    clean = run_library(x, w, entry="general", algo=ALGO_FFMA)
    x[0, 8, 9, 14], x[1, 0, 0, 0] = np.nan, np.inf
    y = run_library(x, w, entry="general", algo=ALGO_FFMA)
    hit = np.zeros((2, 8, 13), bool)
    hit[0, 7, 12] = hit[1, 0, 0] = True
    assert np.isnan(y[0][:, hit[0]]).all() and np.isposinf(y[1][:, hit[1]]).all()
    for n in range(2):
        np.testing.assert_array_equal(y[n][:, ~hit[n]], clean[n][:, ~hit[n]])


@pytest.mark.parametrize("dims", [
    (36, 480, 11, 11, 7), (9, 80, 21, 21, 16), (3, 33, 19, 18, 9),      # one or two groups: a part of the threads only copies
    (2, 16, 31, 62, 384), (5, 5, 20, 47, 55), (1, 1, 3, 3, 1),           # one channel block
])
def test_pointwise_splits_exact_on_integers(oracle, dims):
    N, C, H, W, K = dims
    x, w = small_integers((N, C, H, W), 1505), small_integers((K, C, 1, 1), 1506)
    y_ref, _ = oracle.conv2d_oracle(x, w)
    np.testing.assert_array_equal(run_library(x, w, entry="general", algo=ALGO_FFMA).astype(np.float64), y_ref)
