"""The float convolution and input gradient at the edges of their tiles: strips and patches that overhang the image, several
small images per patch, channel counts that are not multiples of 4 or of a tile, the three channel-tile widths, volumes and
circular shifts.  Sums of up to a few thousand float products: the float bar of test_gpu_parity.py."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from oracle import xconv_oracle as O
from paper_2106_06998_b200 import binding as xb
from tests._util import TOL, check, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("B,Cin,Cout,D,H,W,K,KD,circular", [
    (64, 3, 64, 1, 33, 35, 3, 1, False),       # three channels in; 8 x 8 channel tile
    (96, 16, 18, 1, 30, 41, 3, 1, False),      # channels out beyond whole float4s
    (200, 64, 16, 1, 7, 7, 3, 1, False),       # several images per patch, the narrow channel tile
    (120, 20, 36, 1, 14, 9, 5, 1, False),      # 25 offsets, the middle channel tile
    (40, 33, 64, 1, 28, 28, 1, 1, False),      # pointwise, an input channel over a whole chunk
    (6, 16, 24, 9, 13, 11, 3, 3, False),       # 27 offsets, planes outside the volume
    (6, 8, 32, 5, 20, 20, 3, 1, False),        # planar kernel on the planes of a volume
    (64, 12, 40, 1, 17, 31, 3, 1, True),       # circular shifts
    (2, 5, 7, 1, 9, 11, 3, 1, False),          # a layer too small for the tiles
])
def test_convolution_and_input_gradient(B, Cin, Cout, D, H, W, K, KD, circular):
    g = np.random.Generator(np.random.PCG64([B, Cin, Cout, H, W, K]))
    geo, kgeo = ((D, H, W), (KD, K, K)) if D > 1 else ((H, W), (K, K))
    X, dY = (g.standard_normal((B, c) + geo).astype(np.float32) for c in (Cin, Cout))
    Wt = (g.standard_normal((Cout, Cin) + kgeo) * (2.0 / (K * K * KD * Cin)) ** 0.5).astype(np.float32)
    Z = np.ones((1, Cin) + geo, np.float32)
    d = {k: xb.to_device(v, "f32") for k, v in dict(X=X, dY=dY, W=Wt, Z=Z).items()}
    Y, _ = xb.xconv_forward(d["X"], d["W"], d["Z"], circular=circular)
    dX = xb.xconv_dgrad(d["dY"], d["W"], circular=circular)
    torch.cuda.synchronize()
    if D > 1:
        Yo, dXo = O.conv_forward3d(X, Wt), O.dx_exact3d(dY, Wt)
    else:
        Yo, dXo = O.conv_forward(X, Wt, circular=circular), O.dx_exact(dY, Wt, circular=circular)
    check("Y", host(Y), Yo, TOL["f32"])
    check("dX", host(dX), dXo, TOL["f32"])
