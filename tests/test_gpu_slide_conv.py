"""The convolutions that walk along an axis (conv_slide.cuh), at the edges of their walk: runs of outputs that start and end inside a column, columns shorter
than the kernel, rows of several images in a tile with a last group that is not full, several blocks of channels, accumulators whose ring ends
inside an MMA, rows longer than a tile, volumes; and the ones done in patches with more than four input boxes in flight.  Bars as in test_gpu_parity.py: one rounding to the storage type."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from paper_2106_06998_b200 import binding as xb
from paper_2106_06998_b200 import inputs
from tests._util import TOL, check, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("dtype,B,Cin,Cout,D,H,W,K", [
    ("bf16", 3, 32, 32, 1, 131, 128, 3),      # one tile a row, runs that end inside an image
    ("f16", 2, 32, 24, 1, 101, 257, 3),       # rows of three tiles, the last nearly empty; channels out off the block
    ("bf16", 160, 16, 16, 1, 33, 30, 3),      # four images a tile
    ("f16", 149, 24, 16, 1, 40, 30, 3),       # ... and a last group of one
    ("bf16", 5, 8, 8, 1, 90, 120, 3),         # half a k-step of channels, the smallest number of channels out
    ("f16", 20, 16, 16, 1, 67, 70, 5),        # 25 offsets
    ("bf16", 7, 64, 48, 1, 50, 100, 5),       # ... four k-steps; 240 columns an MMA, a ring of ten
    ("bf16", 4, 136, 32, 1, 60, 110, 3),      # three blocks of channels
    ("f16", 7, 64, 64, 1, 64, 120, 3),        # 192 columns, a ring of eight
    ("bf16", 3, 32, 32, 33, 20, 24, 3),       # volumes
    ("f16", 30, 48, 16, 2, 40, 50, 3),        # ... of fewer planes than the kernel has
    ("bf16", 2, 64, 24, 27, 33, 40, 3),       # ... whose weights were streamed
])
def test_walked_convolution_and_input_gradient(dtype, B, Cin, Cout, D, H, W, K):
    convolutions_against_64_bits(dtype, B, Cin, Cout, D, H, W, K)


@pytest.mark.parametrize("dtype,B,Cin,Cout,H,W,K", [
    ("f16", 19, 72, 8, 131, 128, 1),          # pointwise: sixteen patches a CTA and some CTAs with fewer, two blocks of channels
    ("bf16", 46, 192, 24, 129, 129, 1),       # ... forty, three blocks, a last patch of few pixels
    ("f16", 37, 24, 64, 83, 83, 3),           # patches, whose input gradient walks
    ("bf16", 9, 96, 16, 133, 131, 3),         # ... whose input gradient is done in patches
])
def test_long_runs_of_patches(dtype, B, Cin, Cout, H, W, K):
    convolutions_against_64_bits(dtype, B, Cin, Cout, 1, H, W, K)


def convolutions_against_64_bits(dtype, B, Cin, Cout, D, H, W, K):
    g = np.random.Generator(np.random.PCG64([B, Cin, Cout, H, W, K]))
    geo, kgeo, KD = ((D, H, W), (K, K, K), K) if D > 1 else ((H, W), (K, K), 1)
    X, dY = (inputs.round_to_storage(g.standard_normal((B, c) + geo, dtype=np.float32), dtype) for c in (Cin, Cout))
    Wt = inputs.round_to_storage((g.standard_normal((Cout, Cin) + kgeo) * (2.0 / (K * K * KD * Cin)) ** 0.5).astype(np.float32), dtype)
    Xd, dYd, Wd = (xb.to_device(v, dtype) for v in (X, dY, Wt))
    Zd = xb.to_device(np.ones((1, Cin) + geo, np.float32), dtype)
    Y, _ = xb.xconv_forward(Xd, Wd, Zd)
    dX = xb.xconv_dgrad(dYd, Wd)
    # the same convolutions in 64 bits
    t = lambda v: torch.from_numpy(v).double().cuda()
    conv = torch.nn.functional.conv3d if D > 1 else torch.nn.functional.conv2d
    back = torch.nn.functional.conv_transpose3d if D > 1 else torch.nn.functional.conv_transpose2d
    check("Y", host(Y), host(conv(t(X), t(Wt), padding=(K - 1) // 2)), TOL[dtype])
    check("dX", host(dX), host(back(t(dY), t(Wt), padding=(K - 1) // 2)), TOL[dtype])
