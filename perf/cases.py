"""Workloads of the convolution library, as a program that uses it calls them.

``listed()`` names one workload per way of using the library, ``draw(rng)`` gives another of the same ranges,
``prepare`` makes a workload's inputs and buffers, ``run`` is one call through the public binding and returns the
whole output tensor.  ``work`` counts what the operation cannot do without; ``tolerance`` is what another correct
implementation at the same precision would differ by; ``exact`` is the result in 64 bits.

A case is a dict of
  entry   "single" | "general" | "16bit" | "padded" | "strided" | "noalloc" | "host"
  N C H W K R S, pad (both directions), stride
  algo    "auto" | "fp32" (the exact fp32 algorithm); operand "fp32" | "bf16" | "fp16"
  packed  the filters of a layer do not change between calls: re-ordered once, as an inference program keeps them
  data    "uniform_pm1" | "uniform_01" | "relu" (activations after a ReLU, about half zeros)
"""
import math

import torch

import paper_1705_10591_b200 as lib

_DEFAULTS = dict(entry="general", N=1, C=1, H=64, W=64, K=8, R=3, S=3, pad=0, stride=1,
                 algo="auto", operand="fp32", packed=False, data="relu")


def _case(name=None, **kw):
    c = dict(_DEFAULTS, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # one grey-scale tile through a small filter bank: a call in a loop over tiles, all launch latency
        _case("one_channel_tile", entry="single", H=64, W=64, K=8, R=3, S=3, data="uniform_pm1"),
        # a large single-channel frame through a bank of 5 x 5 filters: the repository's headline workload
        _case("one_channel_large", entry="single", H=4096, W=4096, K=32, R=5, S=5, data="uniform_pm1"),
        # frames as cameras deliver them: a few at a time, extents that no tile divides
        _case("one_channel_ragged", entry="single", N=3, H=1083, W=1917, K=16, R=3, S=3, data="uniform_01"),
        # early layer of an image network, output as large as the input, filters fixed between calls
        _case("early_layer_same", entry="padded", N=32, C=64, H=56, W=56, K=64, R=3, S=3, pad=1, packed=True),
        # deep layer on small maps, complete call (filters handed over each time, as after a weight update)
        _case("deep_layer", entry="general", N=32, C=256, H=14, W=14, K=256, R=3, S=3),
        # large filters on many channels: the most arithmetic of one call
        _case("large_filters", entry="general", N=64, C=128, H=32, W=32, K=128, R=7, S=7, data="uniform_01"),
        # channel mixing between spatial layers
        _case("pointwise", entry="general", N=64, C=128, H=32, W=32, K=128, R=1, S=1, data="uniform_01"),
        # 16-bit inference, filters fixed
        _case("bf16_layer", entry="16bit", N=64, C=128, H=32, W=32, K=128, R=3, S=3, operand="bf16", packed=True,
              data="uniform_01"),
        # results to fp32 rounding, for callers who check or calibrate against exact arithmetic; ragged extents
        _case("fp32_exact", entry="general", N=32, C=96, H=27, W=35, K=112, R=3, S=3, algo="fp32"),
        # first layer of an image network: three channels, large window, down-sampling by two
        _case("strided_first_layer", entry="strided", N=32, C=3, H=224, W=224, K=64, R=7, S=7, pad=3, stride=2,
              data="uniform_01"),
        # down-sampling layer between stages, filters fixed
        _case("strided_layer", entry="strided", N=32, C=128, H=56, W=56, K=128, R=3, S=3, pad=1, stride=2, packed=True),
        # a program whose tensors live in host memory
        _case("host_buffers", entry="host", N=32, C=64, H=56, W=56, K=64, R=3, S=3),
    ]


def _out_hw(c):
    return ((c["H"] + 2 * c["pad"] - c["R"]) // c["stride"] + 1, (c["W"] + 2 * c["pad"] - c["S"]) // c["stride"] + 1)


def work(case):
    c = case
    P, Q = _out_hw(c)
    flops = 2 * c["N"] * c["K"] * c["C"] * c["R"] * c["S"] * P * Q
    # a filter smaller than the stride leaves input rows and columns untouched
    rows = c["H"] if c["R"] >= c["stride"] else min(c["H"], P * c["R"])
    cols = c["W"] if c["S"] >= c["stride"] else min(c["W"], Q * c["S"])
    size = 4 if c["operand"] == "fp32" else 2
    nbytes = size * (c["N"] * c["C"] * rows * cols + c["K"] * c["C"] * c["R"] * c["S"]) + 4 * c["N"] * c["K"] * P * Q
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # four times the largest error measured against the same convolution in float64, over the listed cases and forty
    # drawn ones (2-norm / largest): one channel 1.0e-7 / 8.6e-7; fp32 and exact 16-bit products with fp32 sums over
    # up to 9408 terms 1.8e-6 / 7.9e-6; operands rounded to TF32 3.1e-4 / 1.9e-3; 1 x 1 filters, whose operands are
    # truncated to TF32, 7.6e-4 / 2.8e-3
    if case["entry"] == "single":
        return {"rel": 4e-7, "max": 4e-6}
    if case["operand"] != "fp32" or case["algo"] == "fp32":
        return {"rel": 7e-6, "max": 3.2e-5}
    if case["R"] == 1 and case["S"] == 1:
        return {"rel": 3e-3, "max": 1.1e-2}
    return {"rel": 1.2e-3, "max": 8e-3}


# ---- drawn cases ------------------------------------------------------------------------------------------------

def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _channels(rng, lo, hi):
    """Channel and filter counts: mostly multiples of 16, sometimes anything."""
    v = _log(rng, lo, hi)
    return max(lo, (v + 8) // 16 * 16) if lo >= 16 and rng.random() < 0.7 else v


def _fits(c, flops, nbytes):
    P, Q = _out_hw(c)
    w = work(c)
    return P >= 1 and Q >= 1 and flops[0] <= w["flops"] <= flops[1] and w["bytes"] <= nbytes


def _draw_single(rng):
    r = rng.choice((1, 3, 3, 5, 5, 7))
    s = r if rng.random() < 0.85 else rng.choice((2, 3, 4, 5))
    c = _case(entry="single", N=_log(rng, 1, 16), H=_log(rng, 48, 4096), W=_log(rng, 48, 4096), K=_log(rng, 1, 64),
              R=r, S=s, data=rng.choice(("uniform_pm1", "uniform_01")))
    return c, (0, 2.7e10), 2.2e9


def _draw_layer(rng, entry):
    r = rng.choice((3, 3, 3, 5, 7) if entry == "padded" else (1, 3, 3, 3, 5, 7))
    few = entry == "strided" and rng.random() < 0.4
    size = _log(rng, 32, 256) if few else _log(rng, 8, 128)
    square = rng.random() < 0.6
    c = _case(entry=entry, N=_log(rng, 1, 64), C=rng.choice((1, 3, 3, 4)) if few else _channels(rng, 16, 512),
              H=size, W=size if square else _log(rng, max(8, size // 2), min(256, size * 2)), K=_channels(rng, 16, 512),
              R=r, S=r, data=rng.choice(("relu", "relu", "uniform_01")))
    if entry == "padded":
        c["pad"] = r // 2
    if entry == "strided":
        c["stride"] = rng.choice((2, 2, 2, 3, 4))
        c["pad"] = r // 2
    if entry in ("general", "16bit", "padded", "strided"):
        c["packed"] = rng.random() < 0.5
    if entry == "16bit":
        c["operand"] = rng.choice(("bf16", "bf16", "fp16"))
    return c


def draw(rng):
    kind = rng.choice(("single", "single", "single", "general", "general", "padded", "16bit", "exact", "strided", "strided",
                       "noalloc", "host"))
    while True:
        if kind == "single":
            c, flops, nbytes = _draw_single(rng)
        elif kind == "exact":
            c = _draw_layer(rng, rng.choice(("general", "general", "padded")))
            c["algo"], c["packed"] = "fp32", False
            flops, nbytes = (1e7, 1.2e10), 2e8
        elif kind == "host":
            c = _draw_layer(rng, "host")
            flops, nbytes = (1e7, 2e10), 5e7
        else:
            c = _draw_layer(rng, kind)
            flops, nbytes = (1e8, 7e10), 3e8
        if kind == "noalloc" and 8 * (c["C"] + 32) * (c["K"] + 128) * c["R"] * c["S"] > 8 << 20:
            continue                                        # its filters have to fit the library's own array
        if kind == "strided" and c["N"] * c["C"] > 65535 or not _fits(c, flops, nbytes):
            continue
        return c


# ---- one workload -----------------------------------------------------------------------------------------------

def _values(shape, kind, gen):
    x = torch.empty(shape, device="cuda")
    if kind == "relu":
        return x.normal_(generator=gen).clamp_(min=0)
    return x.uniform_(-1.0 if kind == "uniform_pm1" else 0.0, 1.0, generator=gen)


def _algo(c):
    return {"auto": lib.ALGO_AUTO, "fp32": lib.ALGO_FFMA}[c["algo"]]


def _inputs(c, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    N, C, H, W, K, R, S = (c[k] for k in "NCHWKRS")
    x = _values((N, C, H, W), c["data"], gen)
    w = torch.empty((K, C, R, S), device="cuda").normal_(0.0, (2.0 / (C * R * S)) ** 0.5, generator=gen)
    if c["entry"] == "16bit":
        kind = torch.bfloat16 if c["operand"] == "bf16" else torch.float16
        x, w = x.to(kind), w.to(kind)
    return x, w


def prepare(case, seed):
    c = case
    N, C, H, W, K, R, S = (c[k] for k in "NCHWKRS")
    P, Q = _out_hw(c)
    x, w = _inputs(c, seed)
    st = {"case": c, "y": torch.empty((N, K, P, Q), device="cuda"), "workspace": None, "bytes": 0}
    if c["entry"] == "16bit":
        st["bytes"] = lib.conv2d_fwd_workspace_size(N, C, H, W, K, R, S, lib.ALGO_16BIT)
    elif c["entry"] in ("general", "host"):
        st["bytes"] = lib.conv2d_fwd_workspace_size(N, C, H, W, K, R, S, _algo(c))
    elif c["entry"] == "padded":
        st["bytes"] = lib.conv2d_fwd_padded_workspace_size(N, C, H, W, K, R, S, c["pad"], c["pad"], _algo(c))
    elif c["entry"] == "strided":
        st["bytes"] = lib.conv2d_fwd_strided_workspace_size(N, C, H, W, K, R, S, c["pad"], c["pad"], c["stride"], _algo(c))
    if st["bytes"]:
        st["workspace"] = torch.empty(st["bytes"], dtype=torch.uint8, device="cuda")
    st["x"], st["w"] = x, w
    if c["entry"] == "host":
        for name in ("x", "w", "y"):
            st[name + "_host"] = torch.empty(st[name].shape, pin_memory=True)
        st["x_host"].copy_(x)
        st["w_host"].copy_(w)
    st["flags"] = 0
    if c["packed"]:
        run(st)                                             # the first call leaves the re-ordered filters in the workspace
        st["flags"] = lib.FLAG_WEIGHTS_PACKED
    return st


def exact(case, seed):
    """The same convolution in float64, an image or a few at a time: one tap's plane of products after the other."""
    c = case
    x, w = _inputs(c, seed)
    P, Q = _out_hw(c)
    pad, st, C, R, S = (c[k] for k in ("pad", "stride", "C", "R", "S"))
    wd = w.double()
    out = torch.empty((c["N"], c["K"], P, Q), dtype=torch.float64, device="cuda")
    for n in range(c["N"]):
        xd = torch.nn.functional.pad(x[n].double(), (pad, pad, pad, pad))
        y = torch.zeros((c["K"], P * Q), dtype=torch.float64, device="cuda")
        for r in range(R):
            for s in range(S):
                taps = xd[:, r:r + st * (P - 1) + 1:st, s:s + st * (Q - 1) + 1:st].reshape(C, P * Q)
                y += wd[:, :, r, s] @ taps
        out[n] = y.view(c["K"], P, Q)
    return out


def run(state):
    st, c = state, state["case"]
    N, C, H, W, K, R, S, pad = (c[k] for k in ("N", "C", "H", "W", "K", "R", "S", "pad"))
    x, w, y = st["x"].data_ptr(), st["w"].data_ptr(), st["y"].data_ptr()
    ws = st["workspace"].data_ptr() if st["workspace"] is not None else 0
    size, flags, entry = st["bytes"], st["flags"], c["entry"]
    stream = torch.cuda.current_stream().cuda_stream
    if entry == "single":
        lib.conv2d_fwd_single_channel(x, w, y, N, H, W, K, R, S, stream=stream)
    elif entry == "general":
        lib.conv2d_fwd_general(x, w, y, N, C, H, W, K, R, S, _algo(c), ws, size, flags, stream)
    elif entry == "16bit":
        operand = lib.OPERAND_BF16 if c["operand"] == "bf16" else lib.OPERAND_FP16
        lib.conv2d_fwd_general_16bit(x, w, y, N, C, H, W, K, R, S, operand, ws, size, flags, stream)
    elif entry == "padded":
        lib.conv2d_fwd_general_padded(x, w, y, N, C, H, W, K, R, S, pad, pad, _algo(c), ws, size, flags, stream)
    elif entry == "strided":
        lib.conv2d_fwd_general_strided(x, w, y, N, C, H, W, K, R, S, pad, pad, c["stride"], _algo(c), ws, size, flags, stream)
    elif entry == "noalloc":
        lib.conv2d_fwd_general_noalloc(x, w, y, N, C, H, W, K, R, S, 0, stream)
    else:
        lib.conv2d_fwd_host(st["x_host"].data_ptr(), st["w_host"].data_ptr(), st["y_host"].data_ptr(), x, w, y,
                            N, C, H, W, K, R, S, _algo(c), ws, size, stream)
        return st["y_host"]
    return st["y"]
