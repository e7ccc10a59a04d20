"""A call whose kernels cannot be launched says so and leaves nothing behind: the next valid call of the same thread succeeds."""
import numpy as np
import pytest

from workloads import small_integers

pytestmark = pytest.mark.gpu


def test_calls_on_a_broken_capture_leave_later_calls_alone(oracle):
    import torch
    import paper_1705_10591_b200 as lib
    from cuda.bindings import runtime as rt

    N, C, H, K = 2, 16, 20, 16
    x, x1 = small_integers((N, C, H, H), 1901), small_integers((N, 1, H, H), 1902)
    w, w1, w2 = small_integers((K, C, 3, 3), 1903), small_integers((K, 1, 3, 3), 1904), small_integers((K, C, 2, 2), 1905)
    xp, wp = small_integers((N, 512, H, H), 1906), small_integers((K, 512, 1, 1), 1907)
    dev = {k: torch.from_numpy(v).cuda() for k, v in dict(x=x, x1=x1, w=w, w1=w1, w2=w2, xp=xp, wp=wp).items()}
    y = torch.empty((N, K, H, H), device="cuda")
    ws = torch.zeros(1 << 22, dtype=torch.uint8, device="cuda")
    p = {k: v.data_ptr() for k, v in dev.items()}
    args = (ws.data_ptr(), ws.numel(), 0)
    # every way of launching: one channel, re-ordered filters, an extended image, a rewritten stride, rounded filters, fp32
    calls = {
        "single": (lambda s: lib.conv2d_fwd_single_channel(p["x1"], p["w1"], y.data_ptr(), N, H, H, K, 3, 3, 0, 0, 0, s),
                   lambda: oracle.conv2d_oracle(x1, w1)[0]),
        "tf32": (lambda s: lib.conv2d_fwd_general(p["x"], p["w"], y.data_ptr(), N, C, H, H, K, 3, 3, lib.ALGO_TF32, *args, s),
                 lambda: oracle.conv2d_oracle(x, w)[0]),
        "padded": (lambda s: lib.conv2d_fwd_general_padded(p["x"], p["w"], y.data_ptr(), N, C, H, H, K, 3, 3, 1, 1, lib.ALGO_FFMA, *args, s),
                   lambda: oracle.conv2d_oracle(np.pad(x, ((0, 0), (0, 0), (1, 1), (1, 1))), w)[0]),
        "strided": (lambda s: lib.conv2d_fwd_general_strided(p["x"], p["w2"], y.data_ptr(), N, C, H, H, K, 2, 2, 0, 0, 2, lib.ALGO_FFMA, *args, s),
                    lambda: oracle.conv2d_oracle(x, w2)[0][:, :, ::2, ::2]),
        "pointwise": (lambda s: lib.conv2d_fwd_general(p["xp"], p["wp"], y.data_ptr(), N, 512, H, H, K, 1, 1, lib.ALGO_TF32, *args, s),
                      lambda: oracle.conv2d_oracle(xp, wp)[0]),
        "fp32": (lambda s: lib.conv2d_fwd_general(p["x"], p["w"], y.data_ptr(), N, C, H, H, K, 3, 3, lib.ALGO_FFMA, 0, 0, 0, s),
                 lambda: oracle.conv2d_oracle(x, w)[0]),
    }
    torch.cuda.synchronize()
    for broken in calls:
        stream = torch.cuda.Stream()
        (err,) = rt.cudaStreamBeginCapture(stream.cuda_stream, rt.cudaStreamCaptureMode.cudaStreamCaptureModeRelaxed)
        assert int(err) == 0
        with pytest.raises(lib.Conv2dError) as e:
            lib.conv2d_get_status(0, stream.cuda_stream)             # (waiting for a captured stream breaks the capture)
        assert e.value.status == 7                                   # CONV2D_ERR_CUDA
        with pytest.raises(lib.Conv2dError) as e:
            calls[broken][0](stream.cuda_stream)
        assert e.value.status == 7
        rt.cudaStreamEndCapture(stream.cuda_stream)
        for name, (call, reference) in calls.items():
            call(0)                                                  # raises if it met the error of the call before
            lib.conv2d_get_status(0, 0)
            r = reference()
            got = y.flatten()[:r.size].cpu().numpy().reshape(r.shape)
            np.testing.assert_array_equal(got.astype(np.float64), r, err_msg=f"{name} after {broken}")
