"""The multiplies, convolutions and recurrent passes that a user of this library runs, for timing them.

Every case goes through the calls of ``paper_2108_11033_b200.binding``: a weight matrix pruned to block-wise kept rows
and columns is packed once (``prepare``) and then used again and again (``run``).  Nothing is tuned per size: the
library's own choice of kernel and tile is what runs.  Weights are N(0, std) at every position (the mask decides what
stays), activations N(0, 1), convolution inputs ReLU(N(0, 1)), all made on the GPU from the seed.
"""
from __future__ import annotations

import math

import torch

from paper_2108_11033_b200 import binding as B

VGG16_CHANNELS = (64, 64, 128, 128, 256, 256, 256, 512, 512, 512, 512, 512, 512)
VGG16_POOL_AFTER = (1, 3, 6, 9, 12)  # zero-based convolutions that a 2x2 max-pool follows
BLOCKS = ((4, 16), (8, 32), (16, 64))
RATES = (4, 8, 16)


def _spmm(name, m, k, n, rate, bh, bw, dtype, dist="uniform", reorder=True):
    c = dict(op="spmm", m=m, k=k, n=n, rate=rate, bh=bh, bw=bw, dtype=dtype, dist=dist, reorder=reorder)
    return dict(c, name=name) if name else c


def _conv(name, batch, cin, cout, h, w, ksize, stride, pad, rate, bh, bw, dtype):
    c = dict(op="conv", batch=batch, cin=cin, cout=cout, h=h, w=w, ksize=ksize, stride=stride, pad=pad, rate=rate, bh=bh, bw=bw,
             dtype=dtype, dist="uniform", reorder=True)
    return dict(c, name=name) if name else c


def _vgg(name, batch, image, rate, bh, bw, dtype):
    c = dict(op="vgg", batch=batch, image=image, rate=rate, bh=bh, bw=bw, dtype=dtype, dist="uniform", reorder=True)
    return dict(c, name=name) if name else c


def _gru(name, op, steps, batch, features, hidden, layers, rate, bh, bw):
    c = dict(op=op, steps=steps, batch=batch, features=features, hidden=hidden, layers=layers, rate=rate, bh=bh, bw=bw, dtype="f32",
             dist="uniform", reorder=True)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small product, as of a small layer on a few dozen samples: the call itself is what it costs
        _spmm("spmm_256_n64_f32", 256, 256, 64, 4, 16, 16, "f32"),
        # one large layer on one sample (a recurrent or fully connected layer at batch 1): bound by reading the weights
        _spmm("gemv_8192_c4_f32", 8192, 8192, 1, 4, 8, 32, "f32"),
        # a handful of samples on a layer of odd sizes, small blocks, heavy-tailed kept-row counts
        _spmm("skinny_3001x5003_n7_f32", 3001, 5003, 7, 8, 4, 16, "f32", "zipf"),
        # a decoding batch of sixteen in bf16
        _spmm("batch16_4096_bf16", 4096, 4096, 16, 8, 8, 32, "bf16"),
        # an ordinary batch, nothing a multiple of anything
        _spmm("ragged_1533x2050_n131_f32", 1533, 2050, 131, 16, 16, 64, "f32", "uniform", False),
        # the largest product of the benchmark's sweep, both data types
        _spmm("spmm_8192_n1024_f32", 8192, 8192, 1024, 8, 8, 32, "f32"),
        _spmm("spmm_8192_n1024_bf16", 8192, 8192, 1024, 8, 8, 32, "bf16"),
        # a deep convolution layer: one image in fp32 (latency), a batch in bf16 (throughput)
        _conv("conv_512_28_b1_f32", 1, 512, 512, 28, 28, 3, 1, 1, 8, 16, 64, "f32"),
        _conv("conv_512_28_b32_bf16", 32, 512, 512, 28, 28, 3, 1, 1, 8, 16, 64, "bf16"),
        # the whole convolutional part of VGG-16 with its max-pools on a batch of images
        _vgg("vgg16_b16_bf16", 16, 224, 8, 8, 32, "bf16"),
        # speech-sized recurrent network: a whole utterance of one speaker, and one step of 32 speakers
        _gru("gru_2x1024_t200_f32", "gru", 200, 1, 153, 1024, 2, 10, 8, 32),
        _gru("gru_step_2x1024_b32_f32", "gru_step", 1, 32, 153, 1024, 2, 10, 8, 32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """A size, log-uniform; half of them multiples of 64 where that is not below the range, half as they fall."""
    v = _log(rng, lo, hi)
    return v if rng.random() < 0.5 else min(hi, max(lo, (v + 32) // 64 * 64))


def draw(rng):
    kind = rng.random()
    bh, bw = rng.choice(BLOCKS)
    rate = rng.choice(RATES)
    dtype = rng.choice(("f32", "bf16"))
    if kind < 0.5:
        m, k = _size(rng, 256, 8192), _size(rng, 256, 8192)
        if rng.random() < 0.4:
            k = m
        n = rng.choice((1, _log(rng, 2, 16), _size(rng, 17, 1024), _log(rng, 17, 1024)))
        n = max(1, min(n, (8192 * 8192 // 8 * 1024) // (m * k // rate)))
        if bh == 4:
            n = min(n, 512)
        return _spmm(None, m, k, n, rate, bh, bw, dtype, rng.choice(("uniform", "zipf")), rng.random() < 0.7)
    if kind < 0.75:
        ksize, stride, pad = rng.choice(((3, 1, 1), (3, 1, 1), (3, 1, 1), (1, 1, 0), (3, 2, 1), (5, 1, 2)))
        cin, cout = _size(rng, 16, 512), _size(rng, 32, 512)
        h = rng.choice((7, 14, 28, 56, 112, _log(rng, 7, 112)))
        w = h if rng.random() < 0.7 else _log(rng, 7, 112)
        most = 512 * 4608 * 784 * (32 if dtype == "bf16" and stride == 1 else 8)
        batch = max(1, min(_log(rng, 1, 32), most // (cin * cout * ksize * ksize * max(1, h * w // stride ** 2))))
        return _conv(None, batch, cin, cout, h, w, ksize, stride, pad, rate, bh, bw, dtype)
    if kind < 0.82:
        dtype = "bf16" if rng.random() < 0.8 else "f32"
        return _vgg(None, _log(rng, 1, 16 if dtype == "bf16" else 2), rng.choice((96, 128, 160, 192, 224)), rng.choice((8, 16)), bh, bw, dtype)
    hidden = rng.choice((256, 512, 768, 1024, 16 * _log(rng, 16, 64)))
    layers = rng.choice((1, 2, 2, 3))
    features = _size(rng, 16, 512)
    rate = rng.choice((8, 10, 16))
    if kind < 0.92:
        return _gru(None, "gru", max(1, min(_log(rng, 2, 400), 400 // layers)), 1, features, hidden, layers, rate, bh, bw)
    return _gru(None, "gru_step", 1, _log(rng, 1, 64), features, hidden, layers, rate, bh, bw)


def _mask(m, k, bh, bw, rate, dist, g):
    """Keep-mask: per block a random number of kept rows (uniform on 1 .. bh, or P(r) ~ r^-1.2), as many kept columns as give
    the pruning rate on average, and random rows and columns of those counts."""
    dev = g.device
    nbr, nbc = -(-m // bh), -(-k // bw)
    hb = torch.clamp(m - bh * torch.arange(nbr, device=dev), max=bh)[:, None].expand(nbr, nbc)
    wb = torch.clamp(k - bw * torch.arange(nbc, device=dev), max=bw)[None, :].expand(nbr, nbc)
    p = torch.arange(1, bh + 1, device=dev, dtype=torch.float64) ** (-1.2 if dist == "zipf" else 0.0)
    have = torch.arange(1, bh + 1, device=dev)[None, :] <= torch.arange(1, bh + 1, device=dev)[:, None]
    p = p * have  # row e - 1: blocks that have e rows
    p = p / p.sum(1, keepdim=True)
    mean = (p * torch.arange(1, bh + 1, device=dev)).sum(1)[hb - 1]
    u = torch.rand(nbr, nbc, device=dev, generator=g)
    kr = torch.minimum(1 + (u[:, :, None] >= p.cumsum(1).float()[hb - 1]).sum(2), hb)
    t = torch.minimum(torch.clamp(hb * wb / (rate * mean), min=1.0), wb.double())
    kc = torch.floor(t + torch.rand(nbr, nbc, device=dev, generator=g)).long()
    kc = torch.minimum(torch.clamp(kc, min=1), wb)

    def subset(count, extent, width):
        keys = torch.rand(nbr, nbc, width, device=dev, generator=g)
        keys.masked_fill_(torch.arange(width, device=dev) >= extent[:, :, None], 2.0)
        return torch.argsort(torch.argsort(keys, dim=2), dim=2) < count[:, :, None]

    rows, cols = subset(kr, hb, bh), subset(kc, wb, bw)
    full = (rows[:, :, :, None] & cols[:, :, None, :]).permute(0, 2, 1, 3).reshape(nbr * bh, nbc * bw)
    return full[:m, :k].to(torch.uint8).cpu().numpy()


def _pack(m, k, c, std, g):
    """A packed matrix of the case's block shape, rate and data type."""
    w = (torch.randn(m, k, device=g.device, generator=g) * std).cpu().numpy()
    return B.grim_bcr_pack(w, _mask(m, k, c["bh"], c["bw"], c["rate"], c["dist"], g), c["bh"], c["bw"],
                           B.GRIM_BF16 if c["dtype"] == "bf16" else B.GRIM_F32, B.GRIM_PACK_REORDER if c["reorder"] else 0)


def _reserve(h, ncols, c):
    """The workspace that the library asks users of bf16 handles to set up once (it takes at most 1 GiB of it)."""
    if c["dtype"] == "bf16" and B.grim_bcr_info(h).M * ncols * 4 <= 1 << 30:
        B.grim_bcr_reserve(h, ncols)


class _State:
    """What a user's program keeps: the handles and its own tensors."""

    def __init__(self, case):
        self.case, self.handles, self.gru = case, [], None

    def __del__(self):
        if self.gru is not None:
            B.grim_gru_destroy(self.gru)
        for h in self.handles:
            B.grim_bcr_destroy(h)


def _conv_out(c):
    return (c["h"] + 2 * c["pad"] - c["ksize"]) // c["stride"] + 1, (c["w"] + 2 * c["pad"] - c["ksize"]) // c["stride"] + 1


def prepare(case, seed):
    c = case
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    s = _State(c)

    def normal(*shape):
        return torch.randn(*shape, device=dev, generator=g)

    if c["op"] == "spmm":
        s.handles.append(_pack(c["m"], c["k"], c, 0.05, g))
        _reserve(s.handles[0], c["n"], c)
        s.x = normal(c["k"], c["n"]).to(dt)
        s.y = torch.empty(c["m"], c["n"], device=dev, dtype=dt)
    elif c["op"] == "conv":
        s.handles.append(_pack(c["cout"], c["cin"] * c["ksize"] ** 2, c, 0.05, g))
        oh, ow = _conv_out(c)
        _reserve(s.handles[0], c["batch"] * oh * ow, c)
        s.bias = normal(c["cout"]) * 0.05
        s.x = torch.relu(normal(c["batch"], c["cin"], c["h"], c["w"])).to(dt)
        s.y = torch.empty(c["batch"], c["cout"], oh, ow, device=dev, dtype=dt)
    elif c["op"] == "vgg":
        n, hw, cin, s.bias, s.act, s.pooled = c["batch"], c["image"], 3, [], [], []
        s.x = normal(n, 3, hw, hw).to(dt)
        for i, cout in enumerate(VGG16_CHANNELS):
            # a spread that keeps the size of the activations from layer to layer, as trained weights do
            s.handles.append(_pack(cout, cin * 9, c, math.sqrt(2.0 * c["rate"] / (cin * 9)), g))
            _reserve(s.handles[-1], n * hw * hw, c)
            s.bias.append(normal(cout) * 0.05)
            s.act.append(torch.empty(n, cout, hw, hw, device=dev, dtype=dt))
            cin = cout
            hw = hw // 2 if i in VGG16_POOL_AFTER else hw
            s.pooled.append(torch.empty(n, cout, hw, hw, device=dev, dtype=dt) if i in VGG16_POOL_AFTER else None)
    else:
        hid, ih, hh, b_ih, b_hh = c["hidden"], [], [], [], []
        for l in range(c["layers"]):
            ih.append(_pack(3 * hid, c["features"] if l == 0 else hid, c, 0.05, g))
            hh.append(_pack(3 * hid, hid, c, 0.05, g))
            b_ih.append((normal(3 * hid) * 0.05).cpu().numpy())
            b_hh.append((normal(3 * hid) * 0.05).cpu().numpy())
        s.handles = ih + hh
        s.gru = B.grim_gru_create(ih, hh, b_ih, b_hh, max(c["steps"], 2 * c["batch"]))
        if c["op"] == "gru":
            s.x = normal(c["steps"], c["features"])
            s.h0 = torch.tanh(normal(c["layers"], hid))
            s.y = torch.empty(c["steps"], hid, device=dev)
            s.h = torch.empty(c["layers"], hid, device=dev)
        else:
            s.x = normal(c["batch"], c["features"])
            s.h = torch.tanh(normal(c["layers"], c["batch"], hid))  # carried from step to step
            s.y = torch.empty(c["batch"], hid, device=dev)
    return s


def run(s):
    c = s.case
    if c["op"] == "spmm":
        B.grim_bcr_spmm(s.handles[0], s.x, s.y)
        return s.y
    if c["op"] == "conv":
        B.grim_bcr_conv2d(s.handles[0], s.x, s.y, c["ksize"], c["stride"], c["pad"], s.bias, True)
        return s.y
    if c["op"] == "vgg":
        x = s.x
        for h, bias, act, pooled in zip(s.handles, s.bias, s.act, s.pooled):
            B.grim_bcr_conv2d(h, x, act, 3, 1, 1, bias, True)
            x = act
            if pooled is not None:
                B.grim_maxpool2x2(act, pooled)
                x = pooled
        return x
    if c["op"] == "gru":
        B.grim_gru_seq(s.gru, s.x, s.y, s.h0, s.h)
    else:
        B.grim_gru_step(s.gru, s.x, s.h, s.y)
    return [s.y, s.h]


def _weights(m, k, c):
    """Kept values, and one keep bit per row and column of every block."""
    return m * k / c["rate"] * (2 if c["dtype"] == "bf16" else 4) + -(-m // c["bh"]) * -(-k // c["bw"]) * (c["bh"] + c["bw"]) / 8


def work(case):
    c = case
    e = 2 if c["dtype"] == "bf16" else 4
    if c["op"] == "spmm":
        return {"bytes": _weights(c["m"], c["k"], c) + (c["k"] + c["m"]) * c["n"] * e, "flops": 2 * c["m"] * c["k"] / c["rate"] * c["n"]}
    if c["op"] == "conv":
        (oh, ow), k = _conv_out(c), c["cin"] * c["ksize"] ** 2
        return {"bytes": _weights(c["cout"], k, c) + 4 * c["cout"] + c["batch"] * (c["cin"] * c["h"] * c["w"] + c["cout"] * oh * ow) * e,
                "flops": 2 * c["cout"] * k / c["rate"] * c["batch"] * oh * ow}
    if c["op"] == "vgg":
        nbytes, flops, cin, hw = 0.0, 0.0, 3, c["image"]
        for i, cout in enumerate(VGG16_CHANNELS):  # every call's input and output: the calls are separate
            nbytes += _weights(cout, cin * 9, c) + 4 * cout + c["batch"] * (cin + cout) * hw * hw * e
            flops += 2 * cout * cin * 9 / c["rate"] * c["batch"] * hw * hw
            cin = cout
            if i in VGG16_POOL_AFTER:
                nbytes += c["batch"] * cout * hw * hw * 1.25 * e
                hw //= 2
        return {"bytes": nbytes, "flops": flops}
    hid, nbytes, weights = c["hidden"], 0.0, 0.0
    for l in range(c["layers"]):
        kin = c["features"] if l == 0 else hid
        nbytes += _weights(3 * hid, kin, c) + _weights(3 * hid, hid, c) + 6 * hid * 4
        weights += 3 * hid * (kin + hid) / c["rate"]
    rows = c["steps"] * c["batch"]
    return {"bytes": nbytes + 4 * (rows * (c["features"] + hid) + 2 * c["layers"] * c["batch"] * hid), "flops": 2 * weights * rows}


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}
    # one rounding to bf16 per output; the stack rounds the outputs of thirteen layers in turn
    return {"rel": 1e-2, "max": 1e-1 if case["op"] == "vgg" else 2e-2}
