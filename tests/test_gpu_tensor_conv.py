"""The tensor-core convolution and input gradient at the edges of their tiles: patches that overhang the image, channel
counts that are not whole blocks, one and several column tiles, weights kept and weights streamed, volumes.  Bars as in
test_gpu_parity.py: one rounding to the storage type."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from oracle import xconv_oracle as O
from paper_2106_06998_b200 import binding as xb
from paper_2106_06998_b200 import inputs
from tests._util import TOL, check, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("dtype,B,Cin,Cout,D,H,W,K,KD", [
    ("bf16", 1, 8, 8, 1, 1, 1, 3, 1),          # one pixel, half a k-step of channels
    ("bf16", 2, 16, 16, 1, 7, 7, 3, 1),        # one patch per image, 32-byte tile rows
    ("f16", 3, 24, 40, 1, 9, 130, 3, 1),       # rows longer than a tile; channels beyond the last block
    ("f16", 2, 48, 24, 1, 35, 27, 5, 1),       # 25 offsets, three k-steps per block
    ("bf16", 5, 96, 160, 1, 11, 29, 3, 1),     # a last channel block of 32, weights streamed, an odd number of patches
    ("f16", 3, 320, 272, 1, 6, 10, 3, 1),      # two column tiles, the second nearly empty; five channel blocks
    ("bf16", 40, 128, 128, 1, 28, 28, 3, 1),   # two patches per weight tile on every CTA
    ("bf16", 7, 136, 72, 1, 13, 17, 1, 1),     # pointwise: all pixels of the batch one row, a ragged last patch
    ("f16", 2, 32, 16, 5, 6, 20, 3, 3),        # 27 offsets, planes outside the volume
    ("bf16", 1, 128, 64, 3, 10, 12, 3, 3),     # the same with streamed weights
    ("bf16", 3, 16, 32, 4, 9, 9, 5, 1),        # planar kernel on the planes of a volume
])
def test_convolution_and_input_gradient(dtype, B, Cin, Cout, D, H, W, K, KD):
    g = np.random.Generator(np.random.PCG64([B, Cin, Cout, H, W, K]))
    geo, kgeo = ((D, H, W), (KD, K, K)) if D > 1 else ((H, W), (K, K))
    X, dY = (inputs.round_to_storage(g.standard_normal((B, c) + geo).astype(np.float32), dtype) for c in (Cin, Cout))
    Wt = inputs.round_to_storage((g.standard_normal((Cout, Cin) + kgeo) * (2.0 / (K * K * KD * Cin)) ** 0.5).astype(np.float32), dtype)
    Z = inputs.round_to_storage(g.standard_normal((4, Cin) + geo).astype(np.float32), dtype)
    dev = {k: xb.to_device(v, dtype) for k, v in dict(X=X, dY=dY, W=Wt, Z=Z).items()}
    desc = xb.make_desc(B, Cin, Cout, H, W, 4, dev["X"].dtype, K, D=D, KD=KD)
    for op in (xb.OP_FORWARD, xb.OP_DGRAD):
        assert xb.engine_for(desc, op) == "tcgen05_" + dtype
    Y, _ = xb.xconv_forward(dev["X"], dev["W"], dev["Z"])
    dX = xb.xconv_dgrad(dev["dY"], dev["W"])
    torch.cuda.synchronize()
    conv, dx = (O.conv_forward3d, O.dx_exact3d) if D > 1 else (O.conv_forward, O.dx_exact)
    check("Y", host(Y), conv(X, Wt), TOL[dtype])
    check("dX", host(dX), dx(dY, Wt), TOL[dtype])
