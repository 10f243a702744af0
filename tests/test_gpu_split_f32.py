"""The float kernels on the tensor cores (three bfloat16 parts a float): edges of their tiles, channel counts that are no multiple of
four, every form of the contraction's rows, calls whose scratch is too small for them, and values that cannot be split.

Bounds against 64 bits.  A product's parts leave out 2^-25 of it, an accumulator loses at most 2^-23 of its value an MMA (rounded
towards zero) over chains of at most ten, and chains are added in float, one rounding of 2^-24 each: with random signs below 6e-7 of the
result's norm for the sums taken here (a few million products)."""
import ctypes

import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from oracle import xconv_oracle as O
from paper_2106_06998_b200 import binding as xb
from paper_2106_06998_b200 import inputs
from tests._util import check, host

pytestmark = pytest.mark.gpu
TOL = 1e-6


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


def _n(shape, seed, scale=1.0):
    return inputs.draw("normal", shape, seed, "f32", scale)


@pytest.mark.parametrize("B,Cin,Cout,D,H,W,K,KD", [
    (70, 3, 68, 1, 29, 31, 3, 1),        # padded copy of the input, two column tiles, the second of four channels
    (9, 40, 20, 1, 37, 26, 5, 1),        # a last block of 8 channels; 25 offsets
    (33, 132, 36, 1, 28, 28, 1, 1),      # pointwise: chains over several blocks
    (3, 20, 100, 7, 19, 23, 3, 3),       # planes outside the volume
    (5, 16, 64, 6, 33, 20, 3, 1),        # a planar kernel on the planes of a volume; blocks of 16 channels
    (2, 48, 48, 1, 5, 300, 3, 1),        # rows wider than a patch
])
def test_convolution(B, Cin, Cout, D, H, W, K, KD):
    geo, kgeo = ((D, H, W), (KD, K, K)) if D > 1 else ((H, W), (K, K))
    X, dY = _n((B, Cin) + geo, 1), _n((B, Cout) + geo, 2)
    Wt = _n((Cout, Cin) + kgeo, 3, (2.0 / (K * K * KD * Cin)) ** 0.5)
    desc = xb.make_desc(B, Cin, Cout, H, W, 1, torch.float32, K, D=D, KD=KD)
    assert xb.engine_for(desc, xb.OP_FORWARD) == "tcgen05_f32"
    d = {k: xb.to_device(v, "f32") for k, v in dict(X=X, dY=dY, W=Wt, Z=np.ones((1, Cin) + geo, np.float32)).items()}
    Y, _ = xb.xconv_forward(d["X"], d["W"], d["Z"])
    dX = xb.xconv_dgrad(d["dY"], d["W"])
    Yo, dXo = (O.conv_forward3d(X, Wt), O.dx_exact3d(dY, Wt)) if D > 1 else (O.conv_forward(X, Wt), O.dx_exact(dY, Wt))
    check("Y", host(Y), Yo, TOL)
    check("dX", host(dX), dXo, TOL)
    # scratch for the header only: the multiply-adds take the call
    small, dX2 = torch.empty(256, dtype=torch.uint8, device="cuda"), torch.empty_like(dX)
    xb.dgrad_into(desc, d["dY"], d["W"], dX2, small)
    check("dX without scratch", host(dX2), dXo, 1e-5)


@pytest.mark.parametrize("r,Cin,Cout,D,H,W,K,KD", [
    (40, 64, 64, 1, 31, 33, 3, 1),       # L moved by rows
    (50, 33, 130, 1, 14, 30, 3, 1),      # one dy per unit, padded copies, channels behind whole tiles
    (300, 3, 64, 1, 7, 7, 3, 1),         # images narrower than a k-step
    (20, 24, 48, 1, 40, 29, 5, 1),       # pixel shifts in two units, two row tiles
    (120, 72, 40, 1, 40, 40, 1, 1),      # pointwise, two blocks of columns
    (120, 40, 200, 1, 40, 41, 1, 1),     # ... and two row tiles
    (6, 20, 36, 9, 12, 17, 3, 3),
])
def test_contraction(r, Cin, Cout, D, H, W, K, KD):
    geo = (D, H, W) if D > 1 else (H, W)
    L, Z = _n((r, Cout) + geo, 4), _n((r, Cin) + geo, 5)
    desc = xb.make_desc(1, Cin, Cout, H, W, r, torch.float32, K, D=D, KD=KD)
    assert xb.engine_for(desc, xb.OP_CONTRACT) == "tcgen05_f32"
    scale = torch.rand(Cin, device="cuda") + 0.5
    dW = xb.xconv_contract(xb.to_device(L, "f32"), xb.to_device(Z, "f32"), kernel_size=K, kernel_depth=KD, chan_scale=scale)
    want = O.wgrad_contract3d(L, Z, (KD, K, K)) if D > 1 else O.wgrad_contract(L, Z, K, K)
    want = want * r * host(scale).reshape((1, -1) + (1,) * (want.ndim - 2))
    check("dW", host(dW), want, TOL)
