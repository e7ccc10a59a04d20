"""Calls whose input is the output of the call before, with no synchronisation between them: one channel, tensor cores with filters
re-ordered by the call, zero padding in the fp32 algorithm, a stride rewritten first.  Every kernel may be launched while the one
before it ends and has to wait for its results.  Integers: equal to the definition in 64 bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_chained_calls_wait_for_each_other(oracle):
    import torch
    import paper_1705_10591_b200 as lib
    from workloads import small_integers

    N, H, K = 2, 40, 16
    stream = torch.cuda.current_stream().cuda_stream
    ws = [np.sign(small_integers(shape, 1800 + i)) for i, shape in enumerate(((K, 1, 3, 3), (K, K, 3, 3), (K, K, 3, 3), (K, K, 2, 2)))]
    wd = [torch.from_numpy(w.astype(np.float32)).cuda() for w in ws]
    sizes = (lib.conv2d_fwd_workspace_size(N, K, H - 2, H - 2, K, 3, 3, lib.ALGO_TF32),
             lib.conv2d_fwd_padded_workspace_size(N, K, H - 4, H - 4, K, 3, 3, 1, 1, lib.ALGO_FFMA),
             lib.conv2d_fwd_strided_workspace_size(N, K, H - 4, H - 4, K, 2, 2, 0, 0, 2, lib.ALGO_FFMA))
    scratch = [torch.empty(max(size, 16), dtype=torch.uint8, device="cuda") for size in sizes]
    xs = [small_integers((N, 1, H, H), 1810 + i) for i in range(6)]
    xd = [torch.from_numpy(x.astype(np.float32)).cuda() for x in xs]
    a = torch.empty((N, K, H - 2, H - 2), device="cuda")
    b = torch.empty((N, K, H - 4, H - 4), device="cuda")
    c = torch.empty((N, K, H - 4, H - 4), device="cuda")
    out = [torch.full((N, K, H // 2 - 2, H // 2 - 2), float("nan"), device="cuda") for _ in xs]
    torch.cuda.synchronize()
    for _ in range(5):                           # (the next chain overwrites the buffers between the calls)
        for x, y in zip(xd, out):
            lib.conv2d_fwd_single_channel(x.data_ptr(), wd[0].data_ptr(), a.data_ptr(), N, H, H, K, 3, 3, 0, 0, 0, stream)
            lib.conv2d_fwd_general(a.data_ptr(), wd[1].data_ptr(), b.data_ptr(), N, K, H - 2, H - 2, K, 3, 3, lib.ALGO_TF32,
                                   scratch[0].data_ptr(), sizes[0], 0, stream)
            lib.conv2d_fwd_general_padded(b.data_ptr(), wd[2].data_ptr(), c.data_ptr(), N, K, H - 4, H - 4, K, 3, 3, 1, 1, lib.ALGO_FFMA,
                                          scratch[1].data_ptr(), sizes[1], 0, stream)
            lib.conv2d_fwd_general_strided(c.data_ptr(), wd[3].data_ptr(), y.data_ptr(), N, K, H - 4, H - 4, K, 2, 2, 0, 0, 2, lib.ALGO_FFMA,
                                           scratch[2].data_ptr(), sizes[2], 0, stream)
    torch.cuda.synchronize()
    for x, y in zip(xs, out):
        r, _ = oracle.conv2d_oracle(x.astype(np.float32), ws[0].astype(np.float32))
        r, _ = oracle.conv2d_oracle(r.astype(np.float32), ws[1].astype(np.float32))
        r, _ = oracle.conv2d_oracle(np.pad(r.astype(np.float32), ((0, 0), (0, 0), (1, 1), (1, 1))), ws[2].astype(np.float32))
        r, total = oracle.conv2d_oracle(r.astype(np.float32), ws[3].astype(np.float32))
        assert total.max() < 2 ** 24             # every partial sum is exact
        np.testing.assert_array_equal(y.cpu().numpy().astype(np.float64), r[:, :, ::2, ::2])
