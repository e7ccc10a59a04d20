"""conv2d_fwd_host on calls large enough to be copied in groups of images: groups that do not divide the batch, every kernel
the entry reaches, pageable and page-locked buffers, two threads with streams of their own.  Integer inputs: exact."""
import threading

import numpy as np
import pytest

from test_gpu_host_entry import ALGO_AUTO, ALGO_FFMA, ALGO_TF32, _host_call
from workloads import small_integers

pytestmark = pytest.mark.gpu

CASES = [
    # x shape, w shape, algo, workspace
    ((7, 16, 120, 124), (24, 16, 3, 3), ALGO_TF32, "query"),         # five groups, the last one smaller
    ((7, 16, 120, 124), (24, 16, 3, 3), ALGO_FFMA, "none"),
    ((3, 15, 121, 123), (21, 15, 2, 2), ALGO_AUTO, "query"),         # images of odd size: groups that keep the buffers aligned
    ((5, 1, 400, 403), (8, 1, 3, 3), ALGO_AUTO, "none"),             # one channel
    ((9, 128, 40, 40), (128, 128, 1, 1), ALGO_AUTO, "query"),        # the 1 x 1 kernel
]


@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("case", CASES)
def test_exact_on_integers(oracle, case, pinned):
    xs, ws, algo, workspace = case
    x, w = small_integers(xs, 1701), small_integers(ws, 1702)
    y_ref, _ = oracle.conv2d_oracle(x, w)
    np.testing.assert_array_equal(_host_call(x, w, algo, pinned, workspace).astype(np.float64), y_ref)


def test_two_threads(oracle):
    import torch
    xs, ws, algo, workspace = CASES[0]
    inputs = [(small_integers(xs, 1703 + i), small_integers(ws, 1705 + i)) for i in range(2)]
    results = [None, None]

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(3):
                results[i] = _host_call(*inputs[i], algo, True, workspace)
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(2):
        y_ref, _ = oracle.conv2d_oracle(*inputs[i])
        np.testing.assert_array_equal(results[i].astype(np.float64), y_ref)
