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
