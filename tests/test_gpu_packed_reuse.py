"""Filters packed by one call serve calls with other numbers and sizes of images and other paddings: the re-ordered filters depend on
the layer (filters and their sizes, algorithm) alone, although the kernel that reads them is chosen by the image, too."""
import numpy as np
import pytest

# K, C, R, S; then N, H, W, padding: around every line of the rule for compact stacked taps (quads of pixels, patches, room for the bank
# beside the stages), one round of items and several
LAYERS = [
    ((64, 64, 3, 3), [(2, 56, 56, 1), (2, 55, 55, 1), (1, 124, 128, 0), (8, 124, 128, 0), (1, 112, 112, 1), (2, 128, 128, 1), (3, 33, 47, 0), (2, 40, 260, 0)]),
    ((17, 50, 3, 3), [(3, 30, 33, 1), (3, 30, 32, 1), (1, 12, 12, 0), (40, 12, 13, 0)]),
    ((48, 16, 19, 2), [(20, 40, 12, 0), (20, 41, 13, 0), (1, 24, 21, 1)]),                   # 38 pairs of tap and channel block
    ((5, 33, 4, 3), [(2, 20, 24, 0), (2, 21, 25, 0), (2, 20, 24, 1)]),
    ((64, 96, 3, 3), [(2, 20, 24, 0), (2, 21, 25, 1), (1, 90, 130, 1)]),                   # wholly stacked
    ((130, 40, 3, 3), [(2, 20, 24, 0), (2, 21, 25, 1), (1, 90, 130, 1)]),
]


def _values(shape, seed):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return torch.empty(shape, device="cuda").normal_(generator=gen)


def _call(x, w, pad, ws, flags, stride=1):
    import torch
    import paper_1705_10591_b200 as lib
    (N, C, H, W), (K, _, R, S) = x.shape, w.shape
    y = torch.full((N, K, (H + 2 * pad - R) // stride + 1, (W + 2 * pad - S) // stride + 1), float("nan"), device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    if stride > 1:
        lib.conv2d_fwd_general_strided(x.data_ptr(), w.data_ptr(), y.data_ptr(), N, C, H, W, K, R, S, pad, pad, stride, lib.ALGO_TF32,
                                       ws.data_ptr(), ws.numel(), flags, stream)
    elif pad:
        lib.conv2d_fwd_general_padded(x.data_ptr(), w.data_ptr(), y.data_ptr(), N, C, H, W, K, R, S, pad, pad, lib.ALGO_TF32,
                                      ws.data_ptr(), ws.numel(), flags, stream)
    else:
        lib.conv2d_fwd_general(x.data_ptr(), w.data_ptr(), y.data_ptr(), N, C, H, W, K, R, S, lib.ALGO_TF32,
                               ws.data_ptr(), ws.numel(), flags, stream)
    lib.conv2d_get_status(ws.data_ptr(), stream)
    return y.cpu()


@pytest.mark.gpu
@pytest.mark.parametrize("layer,images", LAYERS)
def test_packed_filters_serve_other_images(layer, images):
    import torch
    import paper_1705_10591_b200 as lib
    K, C, R, S = layer
    w = _values((K, C, R, S), 1)
    size = max(lib.conv2d_fwd_padded_workspace_size(N, C, H, W, K, R, S, p, p, lib.ALGO_TF32) for N, H, W, p in images)
    xs = [_values((N, C, H, W), 2 + i) for i, (N, H, W, p) in enumerate(images)]
    expect = [_call(x, w, im[3], torch.zeros(size, dtype=torch.uint8, device="cuda"), 0) for x, im in zip(xs, images)]
    for i, packer in enumerate(images):
        ws = torch.zeros(size, dtype=torch.uint8, device="cuda")
        _call(xs[i], w, packer[3], ws, 0)
        for x, im, y in zip(xs, images, expect):
            # (a contraction split between blocks that add into y: two sums in any order give the same bits)
            assert torch.equal(_call(x, w, im[3], ws, lib.FLAG_WEIGHTS_PACKED), y), (packer, im)


# K, C, R, S, stride, padding; then N, H, W: rows of whole quads and others
STRIDED = [
    ((70, 33, 3, 3, 2, 1), [(2, 20, 24), (2, 21, 25), (3, 18, 27), (1, 40, 132)]), ((64, 48, 5, 5, 2, 1), [(2, 20, 24), (2, 21, 26)]),
    ((40, 20, 4, 4, 2, 1), [(2, 20, 24), (2, 21, 25)]), ((40, 20, 2, 3, 2, 0), [(2, 20, 24), (2, 21, 25)]),
    ((64, 3, 7, 7, 2, 3), [(2, 32, 32), (2, 33, 33), (1, 50, 46)]), ((33, 3, 4, 4, 2, 1), [(2, 32, 32), (2, 33, 33)]),
    ((20, 4, 3, 2, 2, 1), [(2, 20, 24), (2, 21, 25)]), ((20, 17, 5, 4, 3, 1), [(2, 20, 24), (2, 21, 25)]),
]


@pytest.mark.gpu
@pytest.mark.parametrize("layer,images", STRIDED)
def test_packed_filters_of_strided_layers_serve_other_images(layer, images):
    import torch
    import paper_1705_10591_b200 as lib
    K, C, R, S, stride, pad = layer
    w = _values((K, C, R, S), 11)
    size = max(lib.conv2d_fwd_strided_workspace_size(N, C, H, W, K, R, S, pad, pad, stride, lib.ALGO_TF32) for N, H, W in images)
    xs = [_values((N, C, H, W), 12 + i) for i, (N, H, W) in enumerate(images)]
    expect = [_call(x, w, pad, torch.zeros(size, dtype=torch.uint8, device="cuda"), 0, stride) for x in xs]
    for i, packer in enumerate(images):
        ws = torch.zeros(size, dtype=torch.uint8, device="cuda")
        _call(xs[i], w, pad, ws, 0, stride)
        for x, im, y in zip(xs, images, expect):
            assert torch.equal(_call(x, w, pad, ws, lib.FLAG_WEIGHTS_PACKED, stride), y), (packer, im)


@pytest.mark.parametrize("algo", [2, 3])
def test_layout_of_packed_filters_follows_from_the_layer(algo):
    import paper_1705_10591_b200 as lib
    rng = np.random.default_rng(5)
    compact = 0
    for _ in range(400):
        R, S = (int(v) for v in rng.choice([(3, 3), (3, 3), (5, 5), (2, 2), (7, 7), (4, 3), (2, 9), (6, 6), (19, 2), (1, 5), (3, 5)]))
        C, K = int(rng.choice([4, 15, 16, 33, 48, 50, 64, 96, 130, 300])), int(rng.integers(1, 200) if rng.random() < 0.3 else rng.integers(1, 65))
        layouts = set()
        for _ in range(8):
            N, H, W = int(rng.integers(1, 100)), int(rng.integers(R, 200)), int(rng.integers(S, 200))
            plan = lib.conv2d_fwd_plan_describe(N, C, H, W, K, R, S, algo)
            if plan["tensor_core"]:
                layouts.add((plan["bank"], plan["fold"]))
                compact += plan["stacked_compact"]
        assert len(layouts) <= 1, (K, C, R, S, layouts)
    assert compact > 0 or algo == 3                       # (the rule that depends on the image was met)
