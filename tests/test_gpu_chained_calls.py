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


def _layer(kind, x, y, seed):
    """A call that reads the whole of x and writes y (flat buffers are reinterpreted), as a function of a stream."""
    import torch
    import paper_1705_10591_b200 as lib
    from workloads import small_integers

    N, C, H, W = x.shape
    K, (R, S) = (40, (3, 3)) if kind != "pointwise" and kind != "rounded" else (48, (1, 1))
    if kind == "rows" or kind == "flat":                    # every plane an image of one channel
        N, C, K, (R, S) = N * C, 1, 2, ((5, 5) if kind == "rows" else (3, 3))
    w = torch.from_numpy(np.sign(small_integers((K, C, R, S), seed)).astype(np.float32)).cuda()
    algo = lib.ALGO_FFMA if kind in ("padded_fp32", "rewritten") else lib.ALGO_TF32
    sizes = {"padded_fp32": lambda: lib.conv2d_fwd_padded_workspace_size(N, C, H, W, K, R, S, 1, 1, algo),
             "packed_same": lambda: lib.conv2d_fwd_padded_workspace_size(N, C, H, W, K, R, S, 1, 1, algo),
             "rewritten": lambda: lib.conv2d_fwd_strided_workspace_size(N, C, H, W, K, R, S, 0, 0, 2, algo)}
    size = max(16, sizes.get(kind, lambda: lib.conv2d_fwd_workspace_size(N, C, H, W, K, R, S, algo) if C > 1 else 0)())
    ws = torch.zeros(size, dtype=torch.uint8, device="cuda")
    a = (x.data_ptr(), w.data_ptr(), y.data_ptr(), N, C, H, W, K, R, S)

    def call(stream, flags=0):
        if kind in ("rows", "flat"):
            lib.conv2d_fwd_single_channel(*a[:4], H, W, K, R, S, 0, 0, 0, stream)
        elif kind in ("padded_fp32", "packed_same"):
            lib.conv2d_fwd_general_padded(*a, 1, 1, algo, ws.data_ptr(), size, flags, stream)
        elif kind == "rewritten":
            lib.conv2d_fwd_general_strided(*a, 0, 0, 2, algo, ws.data_ptr(), size, flags, stream)
        else:
            lib.conv2d_fwd_general(*a, algo, ws.data_ptr(), size, flags, stream)
    call.keep = (w, ws)
    if kind.startswith("packed"):
        call(0)                                             # leaves the filters in the workspace
        return lambda stream, call=call: call(stream, lib.FLAG_WEIGHTS_PACKED)
    return call


FOLLOWERS = ["padded_fp32", "rewritten", "reordered", "packed", "packed_same", "pointwise", "rounded", "flat", "rows"]


@pytest.mark.parametrize("first,shape", [
    ("packed_same", (24, 64, 56, 56)), ("packed", (8, 64, 14, 14)),      # several rounds of items; a cluster of two blocks
    ("pointwise", (24, 64, 56, 56)),                                     # triggers early with nothing packed
    ("rounded", (8, 320, 28, 28)),
])
def test_calls_after_one_that_triggers_early_wait_for_it(first, shape):
    """The first call lets the next kernel on the stream be placed while it runs; whatever follows reads its output, and the first
    call of the next round overwrites what that one read.  Equal to the same calls with a synchronisation after each."""
    import torch
    from workloads import small_integers

    xs = [torch.from_numpy(small_integers(shape, 1821 + i).astype(np.float32)).cuda() for i in range(3)]
    x = torch.empty_like(xs[0])
    K, out = (48, shape[2:]) if first in ("pointwise", "rounded") else (40, shape[2:] if first == "packed_same" else tuple(v - 2 for v in shape[2:]))
    mid = torch.empty((shape[0], K) + tuple(out), device="cuda")
    last = torch.empty(shape[0] * 96 * shape[2] * shape[3], device="cuda")
    producer = _layer(first, x, mid, 1831)
    for kind in FOLLOWERS:
        follower = _layer(kind, mid, last, 1832)
        stream = torch.cuda.current_stream().cuda_stream
        results = []
        for synchronised in (True, False):
            got = []
            torch.cuda.synchronize()
            for _ in range(2):
                for v in xs:
                    x.copy_(v)
                    last.zero_()
                    producer(stream)
                    if synchronised:
                        torch.cuda.synchronize()
                    follower(stream)
                    if synchronised:
                        torch.cuda.synchronize()
                    producer(stream)                        # (writes what the call before reads)
                    got.append((mid.clone(), last.clone()))
            torch.cuda.synchronize()
            results.append(got)
        for a, b in zip(*results):
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]), (first, kind)


@pytest.mark.parametrize("layer", [(24, 64, 56, 56, 64, 3, 3), (8, 128, 14, 14, 160, 3, 3), (8, 512, 28, 28, 96, 1, 1)])
def test_filters_packed_anew_while_a_packed_call_runs(layer):
    """Other filters are re-ordered into the workspace of a call that still reads it, and used; no synchronisation between."""
    import torch
    import paper_1705_10591_b200 as lib
    from workloads import small_integers

    N, C, H, W, K, R, S = layer
    x = torch.from_numpy(small_integers((N, C, H, W), 1841).astype(np.float32)).cuda()
    ws = [torch.from_numpy(small_integers((K, C, R, S), 1842 + i).astype(np.float32)).cuda() for i in range(3)]
    size = lib.conv2d_fwd_workspace_size(N, C, H, W, K, R, S, lib.ALGO_TF32)
    scratch = torch.zeros(size, dtype=torch.uint8, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream

    def run(w, y, flags):
        lib.conv2d_fwd_general(x.data_ptr(), w.data_ptr(), y.data_ptr(), N, C, H, W, K, R, S, lib.ALGO_TF32,
                               scratch.data_ptr(), size, flags, stream)
    ys = [[torch.empty((N, K, H - R + 1, W - S + 1), device="cuda") for _ in range(3)] for _ in ws]
    expect = []
    for w in ws:
        y = torch.empty_like(ys[0][0])
        run(w, y, 0)
        torch.cuda.synchronize()
        expect.append(y)
    for _ in range(3):
        for w, outs in zip(ws, ys):
            for i, y in enumerate(outs):
                run(w, y, lib.FLAG_WEIGHTS_PACKED if i else 0)
    torch.cuda.synchronize()
    for y_ref, outs in zip(expect, ys):
        for y in outs:
            assert torch.equal(y, y_ref)
