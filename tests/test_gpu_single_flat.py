"""One input channel, rows of any alignment (the kernel that stores aligned quads of the output tensor): every residue of
Q and of P*Q modulo four, filters that are not square, one map up to several map blocks, one and two column tiles, one
output row or column.  Integer inputs: every sum is exact, so the result has to equal the oracle's bit for bit."""
import numpy as np
import pytest

from helpers import run_library
from workloads import small_integers

pytestmark = pytest.mark.gpu

# N, H, W, K, R, S
SHAPES = [(2, 20 + p, 30 + q, k, 3, 3) for p in range(4) for q in range(4) for k in (1, 6)]
SHAPES += [
    (1, 9, 1030, 5, 3, 3), (2, 6, 1029, 17, 3, 3), (1, 7, 2063, 3, 1, 1),     # two and three column tiles
    (1, 13, 50, 33, 5, 5), (3, 11, 47, 9, 5, 5), (1, 17, 29, 18, 7, 7), (2, 8, 11, 64, 7, 7),
    (1, 12, 45, 7, 1, 2), (1, 12, 45, 7, 2, 1), (2, 15, 33, 10, 5, 3), (1, 15, 41, 4, 3, 4), (1, 19, 40, 21, 7, 5),
    (1, 30, 23, 3, 9, 6), (1, 40, 37, 2, 30, 7),                              # filter heights without an instance of their own
    (1, 3, 3, 5, 3, 3), (1, 5, 7, 2, 5, 2), (1, 3, 40, 300, 3, 3), (16, 5, 6, 1, 1, 1),
]


@pytest.mark.parametrize("turn", [0, 1])      # maps in classes of equal alignment / quads turned at the store
@pytest.mark.parametrize("dims", SHAPES)
def test_exact_on_integers(oracle, monkeypatch, dims, turn):
    N, H, W, K, R, S = dims
    monkeypatch.setenv("CONV2D_B200_SC_FLAT", "1")
    monkeypatch.setenv("CONV2D_B200_SC_TURN", str(turn))
    x, w = small_integers((N, 1, H, W), 1401), small_integers((K, 1, R, S), 1402)
    y_ref, _ = oracle.conv2d_oracle(x, w)
    np.testing.assert_array_equal(run_library(x, w, entry="single").astype(np.float64), y_ref)


def test_non_finite_pixels_stay_in_their_windows(oracle, monkeypatch):
    """An infinity and a NaN reach the outputs whose windows hold them and no others."""
    monkeypatch.setenv("CONV2D_B200_SC_FLAT", "1")
    x, w = small_integers((1, 1, 21, 39), 1403), np.abs(small_integers((6, 1, 3, 3), 1404)) + 1
    clean = run_library(x, w, entry="single")
    x[0, 0, 4, 17], x[0, 0, 15, 38] = np.inf, np.nan
    y = run_library(x, w, entry="single")
    hit = np.zeros((19, 37), bool)
    hit[2:5, 15:18] = True
    assert np.isposinf(y[0][:, hit]).all()
    nan = np.zeros_like(hit)
    nan[13:16, 36:37] = True
    assert np.isnan(y[0][:, nan]).all()
    np.testing.assert_array_equal(y[0][:, ~(hit | nan)], clean[0][:, ~(hit | nan)])
