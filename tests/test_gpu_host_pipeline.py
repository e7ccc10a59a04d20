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


def test_a_batch_the_single_channel_entry_refuses_is_not_accepted_in_groups():
    import paper_1705_10591_b200 as lib
    x, w = np.zeros((70000, 1, 8, 8), np.float32), np.zeros((1, 1, 3, 3), np.float32)
    with pytest.raises(lib.Conv2dError) as e:
        _host_call(x, w, ALGO_AUTO, False, "none")
    assert e.value.status == 5                      # CONV2D_ERR_UNSUPPORTED


def test_a_call_on_a_captured_stream_leaves_the_other_calls_alone(oracle):
    """The call waits for its stream, so it fails under capture; until that capture ends, a call of another thread on a
    stream of its own must neither fail nor be drawn into it."""
    import torch
    import paper_1705_10591_b200 as lib
    rt = pytest.importorskip("cuda.bindings.runtime")
    xs, ws, algo, workspace = CASES[1]
    x, w = small_integers(xs, 1707), small_integers(ws, 1708)
    y_ref, _ = oracle.conv2d_oracle(x, w)
    N, C, H, W = xs
    xh, wh = torch.from_numpy(x).pin_memory(), torch.from_numpy(w).pin_memory()
    yh = torch.zeros(y_ref.shape).pin_memory()
    xd, wd, yd = (torch.empty(t.shape, device="cuda:0") for t in (xh, wh, yh))
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    outcome = {}

    def captured():
        (err,) = rt.cudaStreamBeginCapture(stream.cuda_stream, rt.cudaStreamCaptureMode.cudaStreamCaptureModeRelaxed)
        outcome["begin"] = int(err)
        try:
            lib.conv2d_fwd_host(xh.data_ptr(), wh.data_ptr(), yh.data_ptr(), xd.data_ptr(), wd.data_ptr(), yd.data_ptr(),
                                N, C, H, W, ws[0], ws[2], ws[3], algo, 0, 0, stream.cuda_stream)
        except lib.Conv2dError as e:
            outcome["captured"] = e.status

    def free():
        with torch.cuda.stream(torch.cuda.Stream()):
            outcome["free"] = _host_call(x, w, algo, True, workspace)
    for part in (captured, free):                   # (threads: a runtime error stays with the thread that met it)
        thread = threading.Thread(target=part)
        thread.start()
        thread.join()
    rt.cudaStreamEndCapture(stream.cuda_stream)
    assert outcome["begin"] == 0 and outcome["captured"] == 7                    # CONV2D_ERR_CUDA
    np.testing.assert_array_equal(outcome["free"].astype(np.float64), y_ref)


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


def test_time_out_of_an_early_group_reaches_its_own_call(oracle, monkeypatch):
    """Host-side injection: the 37th filter copy of a block is armed but never issued, and the wait bound is short.  With
    items of 64 pixels and one tap a copy, only blocks that get a second item come that far: those of the groups of two
    images, not those of the last group of one.  Another thread asks for the device's status all the while: the time-out
    belongs to the host call and must not reach that thread."""
    import torch
    import paper_1705_10591_b200 as lib
    N, C, H, W, K = 9, 64, 96, 96, 128
    x, w = small_integers((N, C, H, W), 1711), small_integers((K, C, 3, 3), 1712)
    y_ref, _ = oracle.conv2d_oracle(x, w)
    xh, wh = torch.from_numpy(x).pin_memory(), torch.from_numpy(w).pin_memory()
    yh = torch.zeros((N, K, H - 2, W - 2)).pin_memory()
    xd, wd, yd = (torch.empty(t.shape, device="cuda:0") for t in (xh, wh, yh))
    nbytes = lib.conv2d_fwd_workspace_size(N, C, H, W, K, 3, 3, ALGO_TF32)
    ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda:0")

    def call():
        lib.conv2d_fwd_host(xh.data_ptr(), wh.data_ptr(), yh.data_ptr(), xd.data_ptr(), wd.data_ptr(), yd.data_ptr(),
                            N, C, H, W, K, 3, 3, ALGO_TF32, ws.data_ptr(), nbytes, torch.cuda.current_stream().cuda_stream)
    monkeypatch.setenv("CONV2D_B200_TF32_TILE_PX", "64")
    monkeypatch.setenv("CONV2D_B200_TF32_STAGE_KB", "8")
    call()
    np.testing.assert_array_equal(yh.numpy().astype(np.float64), y_ref)
    stop, stolen, asked = threading.Event(), [], []

    def ask():
        stream = torch.cuda.Stream()
        while not stop.is_set():
            try:
                lib.conv2d_get_status(0, stream.cuda_stream)
                asked.append(1)
            except lib.Conv2dError as e:
                stolen.append(e.status)
    thread = threading.Thread(target=ask)
    thread.start()
    monkeypatch.setenv("CONV2D_B200_TF32_MAX_POLLS", "20000")
    monkeypatch.setenv("CONV2D_B200_TF32_TEST_DROP_STAGE", "36")
    reported, shown = [], []
    for _ in range(5):
        yh.zero_()
        try:
            call()
            reported.append(0)
        except lib.Conv2dError as e:
            reported.append(e.status)
        shown.append(int(ws[:4].sum()))
    monkeypatch.delenv("CONV2D_B200_TF32_MAX_POLLS")
    monkeypatch.delenv("CONV2D_B200_TF32_TEST_DROP_STAGE")
    stop.set()
    thread.join()
    np.testing.assert_array_equal(yh.numpy()[-1].astype(np.float64), y_ref[-1])       # (the last group did not time out)
    assert asked and not stolen
    assert reported == [8] * 5                      # CONV2D_ERR_DEVICE_TIMEOUT
    assert all(shown)                               # and the status block shows it
    call()
    lib.conv2d_get_status(ws.data_ptr(), 0)
    np.testing.assert_array_equal(yh.numpy().astype(np.float64), y_ref)
