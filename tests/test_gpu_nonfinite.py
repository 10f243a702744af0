"""Infinities and NaN through the 16-bit kernels: a value that is not finite shows in every result it enters, as an infinity of
the right sign where the definition gives one, and nowhere else (in the contraction: in no other channel -- products with
positions outside the image are multiplications by zero there)."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from paper_2106_06998_b200 import binding as xb
from paper_2106_06998_b200 import inputs
from tests._util import host

pytestmark = pytest.mark.gpu
INF, NAN = float("inf"), float("nan")


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


def _rand(shape, seed, dtype, scale=1.0):
    return inputs.draw("normal", shape, seed, dtype, scale)


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("r,B,C,H,W", [
    (20, 21, 24, 11, 13),            # the float S as two 16-bit values: 32 rows,
    (50, 130, 40, 9, 11),            # 64 rows,
    (9, 19, 24, 11, 13),             # 16 rows
    (9, 64, 8, 24, 24),              # S rounded once
    (12, 72, 64, 13, 11),
    (72, 16, 64, 8, 8),              # the tcgen05 kernel
])
def test_backprobe(dtype, r, B, C, H, W):
    dY = _rand((B, C, H, W), r + B, dtype, 0.1)
    S = _rand((r, B), r * B, "f32")
    S[2, 3] = S[5, 3] = 1.0                                   # exactly a 16-bit value: its second value is zero
    S[7, 3] = -1.0 - 2.0 ** -12
    S[r - 1, 3] = 2.0 ** -141 if dtype == "bf16" else 2.0 ** -60      # rounds to zero in 16 bits
    dY[3, 1, 2, 3], dY[3, 4, 5, 6], dY[4, 2, 0, 0] = INF, -INF, NAN
    plain = dY.copy()
    plain[~np.isfinite(plain)] = 0.0
    Sd = torch.from_numpy(S).cuda()
    L = host(xb.xconv_backprobe(Sd, xb.to_device(dY, dtype)))
    Lp = host(xb.xconv_backprobe(Sd, xb.to_device(plain, dtype)))
    hit = np.zeros(dY.shape[1:], bool)
    hit[1, 2, 3] = hit[4, 5, 6] = hit[2, 0, 0] = True
    assert np.array_equal(L[:, ~hit], Lp[:, ~hit]) and np.isfinite(Lp).all()
    rows = np.arange(r)
    if B % 8 == 0 and (C * H * W) % 64 == 0:                  # there S itself is rounded to 16 bits first
        rows = rows[:-1]
    assert np.array_equal(L[rows, 1, 2, 3], np.sign(S[rows, 3]) * INF)
    assert np.array_equal(L[rows, 4, 5, 6], -np.sign(S[rows, 3]) * INF)
    assert np.isnan(L[:, 2, 0, 0]).all()


@pytest.mark.parametrize("dtype,r,Cin,Cout,D,H,W,K,KD", [
    ("bf16", 5, 32, 32, 1, 33, 30, 3, 1),      # L moved by rows
    ("f16", 2, 48, 24, 1, 9, 30, 5, 1),        # one dy per unit
    ("bf16", 3, 3, 5, 1, 9, 17, 3, 1),         # padded copies
    ("bf16", 2, 32, 16, 5, 6, 20, 3, 3),       # a volume
])
def test_contraction(dtype, r, Cin, Cout, D, H, W, K, KD):
    geo = (D, H, W) if D > 1 else (H, W)
    L, Z = _rand((r, Cout) + geo, 1, dtype), _rand((r, Cin) + geo, 2, dtype)
    call = lambda l, z: host(xb.xconv_contract(xb.to_device(l, dtype), xb.to_device(z, dtype), kernel_size=K, kernel_depth=KD))
    want = call(L, Z)
    corner, inner = (0,) * len(geo), tuple(n // 2 for n in geo)
    for at in (corner, inner):
        for bad in (INF, NAN):
            Z2, L2 = Z.copy(), L.copy()
            Z2[(1, 2) + at] = bad
            L2[(0, Cout - 1) + at] = bad
            dW = call(L, Z2)
            others = np.arange(Cin) != 2
            assert np.array_equal(dW[:, others], want[:, others])
            # the terms of the offset 0 hold the value itself
            centre = tuple(n // 2 for n in dW.shape[2:])
            assert not np.isfinite(dW[(slice(None), 2) + centre]).any()
            if bad == INF:
                assert np.array_equal(dW[(slice(None), 2) + centre], np.sign(L[(1, slice(None)) + at]) * INF)
            dW = call(L2, Z)
            assert np.array_equal(dW[:-1], want[:-1]) and not np.isfinite(dW[(-1, slice(None)) + centre]).any()


@pytest.mark.parametrize("dtype,B,Cin,Cout,H,W,K", [
    ("bf16", 2, 16, 16, 7, 7, 3), ("f16", 2, 48, 24, 35, 27, 5), ("bf16", 3, 3, 16, 13, 20, 3), ("bf16", 7, 136, 72, 13, 17, 1),
    ("bf16", 5, 96, 160, 11, 29, 3), ("f32", 16, 16, 24, 30, 41, 3),
])
def test_convolution_and_input_gradient(dtype, B, Cin, Cout, H, W, K):
    X, dY = _rand((B, Cin, H, W), 3, dtype), _rand((B, Cout, H, W), 4, dtype)
    Wt = _rand((Cout, Cin, K, K), 5, dtype, 0.05)
    Z = np.ones((1, Cin, H, W), np.float32)
    Wd, Zd = xb.to_device(Wt, dtype), xb.to_device(Z, dtype)
    fwd = lambda x: host(xb.xconv_forward(xb.to_device(x, dtype), Wd, Zd)[0])
    bwd = lambda y: host(xb.xconv_dgrad(xb.to_device(y, dtype), Wd))
    p = (K - 1) // 2
    for y, x in ((0, 0), (H // 2, W - 1), (H - 1, W // 2)):
        hit = np.zeros((H, W), bool)
        hit[max(0, y - p):y + p + 1, max(0, x - p):x + p + 1] = True
        for f, t, c in ((fwd, X, 2), (bwd, dY, Cout - 1)):
            bad = t.copy()
            bad[1, c, y, x] = INF
            got, want = f(bad), f(t)
            keep = np.ones((B, H, W), bool)
            keep[1] = ~hit
            keep = np.broadcast_to(keep[:, None], got.shape)
            assert np.array_equal(got[keep], want[keep]) and not np.isfinite(got[~keep]).any()


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
def test_streaming_sketch(dtype):
    r, B, C, H, W = 8, 4, 8, 17, 31
    X, Z = _rand((B, C, H, W), 6, dtype), _rand((r, C, H, W), 7, dtype)
    S = host(xb.xconv_sketch(xb.to_device(X, dtype), xb.to_device(Z, dtype)))
    X[2, 3, 16, 30] = -INF
    got = host(xb.xconv_sketch(xb.to_device(X, dtype), xb.to_device(Z, dtype)))
    others = [0, 1, 3]
    assert np.array_equal(got[:, others], S[:, others]) and np.array_equal(got[:, 2], -np.sign(Z[:, 3, 16, 30]) * INF)
    seeded = host(xb.xconv_sketch_seeded(xb.to_device(X, dtype), 5, r))
    Zs = host(xb.xconv_probes_from_seed(5, r, C, H, W, torch.bfloat16 if dtype == "bf16" else torch.float16))
    assert np.array_equal(seeded[:, 2], -Zs[:, 3, 16, 30] * INF) and np.isfinite(seeded[:, others]).all()
