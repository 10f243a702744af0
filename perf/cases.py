"""Workloads of the layer library: what a training program has one convolutional layer do.

A case is one layer (batch, channels, image or volume, kernel, storage type, number r of probing vectors) and the
calls the program makes on it:

  train      forward (Y and the sketch S), weight-gradient estimate, exact input gradient: a layer in the middle of a
             network, one training step
  first      forward and weight-gradient estimate: the first layer of a network, whose input needs no gradient
  estimator  sketch and weight-gradient estimate: the part of the step that the method adds to the convolutions
  backward   weight-gradient estimate and exact input gradient from a sketch kept since the forward pass
  seeded     sketch and estimate with the probing vectors redrawn from a seed in both passes, so that between the
             passes a layer keeps S and eight bytes (the paper's Algorithm 1)

Tensors are channels-last on the GPU, as the library takes them, with the distributions of the library's own
workloads: X rectified normal (an activation), W normal with the fan-in variance, dY normal with standard
deviation 0.1, Z Rademacher or standard normal.
"""
from __future__ import annotations

import math

import torch

from paper_2106_06998_b200 import binding as xb

_DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
# An FP32 multiply-add takes about this many times the time of a 16-bit one on the tensor cores; it keeps drawn layers
# of both kinds within the time of the largest listed one.
_F32_COST = 24


def _case(name, op, dtype, B, Cin, Cout, H, W, r, K=3, D=1, z="rademacher"):
    return dict(name=name, op=op, dtype=dtype, B=B, Cin=Cin, Cout=Cout, D=D, H=H, W=W, K=K, r=r, z=z)


def listed():
    return [
        # A small layer of a small network, float storage, a handful of probes: the latency of the calls.
        _case("small_f32", "train", "f32", 8, 16, 16, 32, 32, 8),
        # A residual block's convolution on small images, float storage.
        _case("resnet_f32", "train", "f32", 128, 64, 64, 32, 32, 64, z="gaussian"),
        # An ImageNet network's middle stage with few probes, mixed precision.
        _case("stage_bf16", "train", "bf16", 64, 128, 128, 56, 56, 32),
        # The outermost level of a U-Net: large images, few channels, small batch, more probes than samples.
        _case("unet_bf16", "train", "bf16", 16, 32, 32, 256, 256, 64, z="gaussian"),
        # A wide layer on a large batch, the whole step: the largest case.
        _case("wide_bf16", "train", "bf16", 512, 256, 256, 28, 28, 64),
        # The same layer, only what the method adds to the convolutions.
        _case("wide_estimator_bf16", "estimator", "bf16", 512, 256, 256, 28, 28, 64),
        # 5 x 5 kernels of the CIFAR-10 network in half precision.
        _case("cifar_5x5_f16", "train", "f16", 128, 16, 32, 32, 32, 32, K=5),
        # Many probes on large images: too many to store, so both passes redraw them from the seed.
        _case("unet_seeded_bf16", "seeded", "bf16", 16, 32, 32, 256, 256, 256),
        # A 3 x 3 x 3 layer of a segmentation network on volumes, few probes.
        _case("volume_bf16", "train", "bf16", 4, 32, 32, 48, 48, 8, D=48),
        # The last, short batch of an epoch on images of odd size; channel counts between the powers of two.
        _case("ragged_bf16", "train", "bf16", 50, 96, 160, 35, 27, 50),
        # The first layer of an image network, three input channels, half precision.
        _case("first_f16", "first", "f16", 32, 3, 64, 112, 112, 64),
        # A pointwise convolution of a bottleneck block, backward pass, more probes than samples.
        _case("pointwise_bf16", "backward", "bf16", 64, 256, 64, 56, 56, 128, K=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    w = work(c)
    return w["flops"] * (_F32_COST if c["dtype"] == "f32" else 1), w["bytes"]


def draw(rng):
    """One more layer of the same ranges: channel counts as networks have them (multiples of 8, or one or three image
    channels), any image size, batches and probe counts half the time powers of two and half the time anything."""
    flops_max, bytes_max = _cost(next(c for c in listed() if c["name"] == "wide_bf16"))
    while True:
        op = rng.choice(["train"] * 8 + ["first"] * 2 + ["estimator"] * 4 + ["backward"] * 3 + ["seeded"] * 3)
        dtype = rng.choice(["f32"] * 3 + ["bf16"] * 4 + ["f16"] * 3)
        K = rng.choice([3] * 7 + [1] * 2 + [5])
        volume = K == 3 and rng.random() < 0.2
        channels = [16, 24, 32, 48, 64, 96, 128] + ([] if K == 5 or volume else [160, 192, 256])
        Cin = rng.choice([1, 3]) if op == "first" else rng.choice(channels)
        Cout = rng.choice([n for n in channels if op == "first" or Cin / 8 <= n <= Cin * 8])
        D = _log_int(rng, 4, 64) if volume else 1
        H = _log_int(rng, 7, 96 if volume else 256)
        W = H if rng.random() < 0.6 else max(7, min(256, int(round(H * rng.uniform(0.5, 2.0)))))
        B = 2 ** rng.randint(2, 9) if rng.random() < 0.5 else _log_int(rng, 4, 512)
        if volume:
            B = max(1, B // 16)
        r = 2 ** rng.randint(3, 9) if rng.random() < 0.5 else _log_int(rng, 8, 512)
        c = dict(op=op, dtype=dtype, B=B, Cin=Cin, Cout=Cout, D=D, H=H, W=W, K=K, r=r,
                 z="rademacher" if op == "seeded" else rng.choice(["rademacher", "gaussian"]))
        if dtype == "f16" and r > B and D * H * W * Cin * r > 2.4e8:
            continue        # the activation rebuilt from its sketch would leave half precision's range (6 sigma = 65504)
        flops, nbytes = _cost(c)
        if 1e6 <= nbytes <= bytes_max and flops <= flops_max:
            return c


def _geometry(c):
    """Image extents, kernel extents and memory format of a planar layer or a volume."""
    if c["D"] > 1:
        return (c["D"], c["H"], c["W"]), (c["K"],) * 3, torch.channels_last_3d
    return (c["H"], c["W"]), (c["K"],) * 2, torch.channels_last


def _inputs(c, seed):
    geo, kgeo, fmt = _geometry(c)
    dtype = _DTYPES[c["dtype"]]
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(shape, scale=1.0, relu=False):
        t = torch.empty(shape, dtype=torch.float32, device="cuda", memory_format=fmt).normal_(generator=gen)
        t = t.relu_() if relu else t.mul_(scale)
        return t.to(dtype)

    s = dict(op=c["op"], K=c["K"], KD=kgeo[0] if c["D"] > 1 else 1, Cin=c["Cin"], r=c["r"])
    if c["op"] == "seeded":
        s["seed"] = 0x9E3779B97F4A7C15 * (seed + 1) & (2 ** 64 - 1)
    elif c["z"] == "gaussian":
        s["Z"] = normal((c["r"], c["Cin"]) + geo)
    else:
        signs = torch.empty((c["r"], c["Cin"]) + geo, dtype=torch.int8, device="cuda", memory_format=fmt)
        s["Z"] = signs.random_(0, 2, generator=gen).mul_(2).sub_(1).to(dtype)
    s["X"] = normal((c["B"], c["Cin"]) + geo, relu=True)
    s["dY"] = normal((c["B"], c["Cout"]) + geo, scale=0.1)
    if c["op"] in ("train", "first", "backward"):
        s["W"] = normal((c["Cout"], c["Cin"]) + kgeo, scale=(2.0 / (c["Cin"] * math.prod(kgeo))) ** 0.5)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    if case["op"] == "backward":
        s["S"] = xb.xconv_sketch(s.pop("X"), s["Z"])       # kept since the forward pass, in the place of X
    return s


def run(state):
    s = state
    op, K, KD = s["op"], s["K"], s["KD"]
    if op == "seeded":
        S = xb.xconv_sketch_seeded(s["X"], s["seed"], s["r"])
        return {"S": S, "dW": xb.xconv_wgrad_seeded(S, s["dY"], s["seed"], s["Cin"], kernel_size=K, kernel_depth=KD)}
    out = {}
    if op == "estimator":
        S = out["S"] = xb.xconv_sketch(s["X"], s["Z"])
    elif op == "backward":
        S = s["S"]
    else:
        out["Y"], S = xb.xconv_forward(s["X"], s["W"], s["Z"])
        out["S"] = S
    out["dW"] = xb.xconv_wgrad(S, s["dY"], s["Z"], kernel_size=K, kernel_depth=KD)
    if op in ("train", "backward"):
        out["dX"] = xb.xconv_dgrad(s["dY"], s["W"])
    return out


def _signs(seed, count, device="cuda"):
    """The first `count` entries (a multiple of 128) of the Rademacher stream that include/xconv.h defines: entry e is
    bit e mod 128 of Philox-4x32-10 block e div 128."""
    blk = torch.arange(count // 128, dtype=torch.int64, device=device)
    m32 = 0xFFFFFFFF
    c0, c1, c2, c3 = blk & m32, blk >> 32, torch.zeros_like(blk), torch.zeros_like(blk)
    k0, k1 = seed & m32, seed >> 32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57           # 64-bit products; the shift below masks off the sign
        c0, c1, c2, c3 = ((p1 >> 32) & m32) ^ c1 ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ c3 ^ k1, p0 & m32
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    bit = torch.arange(32, dtype=torch.int64, device=device)
    words = torch.stack((c0, c1, c2, c3), dim=1).reshape(-1, 1)
    return (1 - 2 * ((words >> bit) & 1).to(torch.int8)).reshape(-1)


def _shifted(t, off):
    """t[:, z + dz, y + dy, x + dx, :] with zeros outside (t: [n, D, H, W, C])."""
    out = torch.zeros_like(t)
    src, dst = [slice(None)], [slice(None)]
    for d, n in zip(off, t.shape[1:4]):
        dst.append(slice(max(0, -d), max(0, min(n, n - d))))
        src.append(slice(max(0, d), max(0, min(n, n + d))))
    out[dst] = t[src]
    return out


def exact(case, seed):
    """What run returns, in 64 bits: the definitions in include/xconv.h, one kernel offset at a time."""
    c = case
    geo, kgeo, fmt = _geometry(c)
    s = _inputs(c, seed)
    shape = (c["D"], c["H"], c["W"])
    offsets = [(z, y, x) for z in range(kgeo[0] if c["D"] > 1 else 1) for y in range(c["K"]) for x in range(c["K"])]
    pads = ((kgeo[0] - 1) // 2 if c["D"] > 1 else 0, (c["K"] - 1) // 2, (c["K"] - 1) // 2)
    offsets = [tuple(k - p for k, p in zip(o, pads)) for o in offsets]

    def rows(t):                                             # [n, D, H, W, C] in 64 bits
        return t.movedim(1, -1).reshape(t.shape[0], *shape, t.shape[1]).double()

    def back(t):                                             # ... and back to (n, C, [D,] H, W)
        return t.reshape(t.shape[0], *geo, t.shape[-1]).movedim(-1, 1)

    X, dY = rows(s["X"]), rows(s["dY"])
    if c["op"] == "seeded":
        n = X[0].numel() * c["r"]
        Z = _signs(s["seed"], (n + 127) // 128 * 128)[:n].double().reshape(c["r"], *X.shape[1:])
    else:
        Z = rows(s["Z"])
    S = Z.flatten(1) @ X.flatten(1).T
    out = {} if c["op"] == "backward" else {"S": S}
    if c["op"] in ("train", "first"):
        Wt = s["W"].double().flatten(2)                      # [Cout, Cin, offset]
        out["Y"] = back(sum(_shifted(X, o) @ Wt[:, :, t].T for t, o in enumerate(offsets)))
    if c["r"] > c["B"]:
        P, Q = dY, (S.T @ Z.flatten(1)).reshape(c["B"], *Z.shape[1:])
    else:
        P, Q = (S @ dY.flatten(1)).reshape(c["r"], *dY.shape[1:]), Z
    P = P.flatten(0, 3).T / c["r"]
    dW = torch.stack([P @ _shifted(Q, o).flatten(0, 3) for o in offsets], dim=-1)
    out["dW"] = dW.reshape(c["Cout"], c["Cin"], *kgeo)
    del P, Q, Z, X
    if c["op"] in ("train", "backward"):
        Wt = s["W"].double().flatten(2)
        out["dX"] = back(sum(_shifted(dY, tuple(-d for d in o)) @ Wt[:, :, t] for t, o in enumerate(offsets)))
    return out


def work(case):
    """Every input read once and every output written once; the estimate counted in the cheaper of its two orders of
    summation (over the batch first, or over the probes first)."""
    c = case
    N = c["D"] * c["H"] * c["W"]
    T = c["K"] ** (3 if c["D"] > 1 else 2)
    B, Ci, Co, r, op = c["B"], c["Cin"], c["Cout"], c["r"], c["op"]
    es = 4 if c["dtype"] == "f32" else 2
    x, dy, z, w = es * B * N * Ci, es * B * N * Co, es * r * N * Ci, es * Co * T * Ci
    conv = 2 * B * N * T * Ci * Co
    nbytes = dy + 4 * Co * T * Ci + 4 * r * B                                    # dY in, dW out, S in or out
    flops = min(2 * r * Co * N * (B + T * Ci), 2 * B * Ci * N * (r + T * Co))
    if op != "seeded":
        nbytes += z
    if op != "backward":
        nbytes += x
        flops += 2 * r * B * Ci * N
    if op in ("train", "first"):
        nbytes += w + dy                                                         # W in, Y out
        flops += conv
    if op in ("train", "backward"):
        nbytes += x + (w if op == "backward" else 0)                             # dX out
        flops += conv
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Relative errors against 64 bits on these layers: float storage up to 1.3e-6 (sums of up to a few
    million products), bfloat16 1.7e-3 and float16 2.1e-4 (each two independent roundings to the storage type)."""
    return {"rel": {"f32": 5e-6, "bf16": 7e-3, "f16": 9e-4}[case["dtype"]]}
