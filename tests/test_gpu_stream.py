"""The kernels that stream one large operand through registers (few samples or few probes) at the edges of their tiles: rows
and terms that are not whole tiles, columns and terms whose last 16-byte piece stands alone, both roles of probes and
samples, signs redrawn from rows that start in the middle of a Philox block.  Bars as in test_gpu_parity.py."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from oracle import xconv_oracle as O
from paper_2106_06998_b200 import binding as xb
from paper_2106_06998_b200 import inputs
from tests._util import TOL, check, host, sketch_tol

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("dtype,r,B,C,H,W", [
    ("bf16", 1, 1, 8, 16, 16),       # one row on both sides, the fewest terms
    ("f16", 8, 4, 8, 17, 31),        # half an MMA row tile, half a column tile
    ("bf16", 16, 16, 24, 13, 29),    # whole tiles, terms that end inside a k-step
    ("bf16", 17, 16, 8, 40, 41),     # a second row tile of one row
    ("f16", 100, 9, 8, 24, 24),      # two blocks of rows
    ("bf16", 3, 75, 16, 19, 8),      # samples on the rows
    ("f16", 16, 33, 64, 30, 30),
])
def test_sketch(dtype, r, B, C, H, W):
    lay = inputs.make_custom(B, C, 8, H, W, r, dtype=dtype, seed=r + B + C + H, z="gaussian", x="normal")
    X, Z = xb.to_device(lay["X"], dtype), xb.to_device(lay["Z"], dtype)
    S, S2 = xb.xconv_sketch(X, Z), xb.xconv_sketch(X, Z)
    torch.cuda.synchronize()
    check("sketch", host(S), O.sketch(lay["X"], lay["Z"]), sketch_tol(C * H * W))
    assert torch.equal(S, S2)


@pytest.mark.parametrize("dtype,r,B,C,H,W", [
    ("bf16", 1, 1, 64, 8, 8),        # one probe, one sample
    ("f16", 65, 9, 64, 5, 13),       # rows of an odd number of half Philox blocks; a second block of one probe
    ("bf16", 130, 16, 32, 20, 20),   # whole Philox blocks, 3 blocks of rows, the last nearly empty
    ("bf16", 40, 3, 16, 36, 41),     # rows that start in the middle of a Philox block
])
def test_seeded_sketch_and_estimate(dtype, r, B, C, H, W):
    seed = 0x1234567890ABCDEF ^ (r * B * C)
    lay = inputs.make_custom(B, C, 8, H, W, r, dtype=dtype, seed=r + B + C + H, z="rademacher", x="normal")
    X, dY = xb.to_device(lay["X"], dtype), xb.to_device(lay["dY"], dtype)
    Z = xb.xconv_probes_from_seed(seed, r, C, H, W, X.dtype)
    S = xb.xconv_sketch_seeded(X, seed, r)
    dW, dW2 = xb.xconv_wgrad_seeded(S, dY, seed, C), xb.xconv_wgrad(S, dY, Z)
    torch.cuda.synchronize()
    Zo = O.rademacher_probes(seed, r, C, H, W)
    So = O.sketch(lay["X"], Zo)
    check("seeded sketch", host(S), So, sketch_tol(C * H * W))
    assert torch.equal(dW, dW2)
    check("dW", host(dW), O.wgrad_estimate(So, lay["dY"], Zo), TOL[dtype])


@pytest.mark.parametrize("dtype,r,B,C,H,W", [
    ("bf16", 1, 1, 8, 16, 16),       # one row, one term
    ("f16", 4, 8, 8, 17, 19),        # one k-step, columns that end inside a group
    ("bf16", 16, 31, 64, 9, 9),      # two k-steps in one go
    ("f16", 9, 64, 8, 24, 24),       # four
    ("bf16", 12, 70, 128, 50, 50),   # a loop over the terms, the second round mostly padding; two groups per warp
    ("bf16", 20, 21, 24, 11, 13),    # rows and terms the tcgen05 kernel does not take
    ("f16", 50, 130, 40, 9, 11),
    ("bf16", 64, 3, 8, 31, 33),
])
def test_backprobe(dtype, r, B, C, H, W):
    g = np.random.Generator(np.random.PCG64([r, B, C, H, W]))
    dY = inputs.round_to_storage((0.1 * g.standard_normal((B, C, H, W))).astype(np.float32), dtype)
    S = g.standard_normal((r, B)).astype(np.float32)
    desc = xb.make_desc(B, 8, C, H, W, r, {"bf16": torch.bfloat16, "f16": torch.float16}[dtype])
    assert xb.engine_for(desc, xb.OP_BACKPROBE) == "tcgen05_" + dtype
    Yd, Sd = xb.to_device(dY, dtype), torch.from_numpy(S).cuda()
    L, L2 = xb.xconv_backprobe(Sd, Yd), xb.xconv_backprobe(Sd, Yd)
    torch.cuda.synchronize()
    check("L", host(L), O.backprobe(S, dY), TOL[dtype])
    assert torch.equal(L, L2)


@pytest.mark.parametrize("dtype,bar", [("bf16", 2.0 ** -9), ("f16", 2.0 ** -12)])
def test_backprobe_keeps_the_float_sketch_where_the_tcgen05_kernel_does_not_go(dtype, bar):
    """Odd batches used the float S all along.  The result is then off by its own rounding alone (relative 2-norm at most
    half a unit in the last place: 2^-9 in bfloat16, 2^-12 in float16); a rounded S would add as much again."""
    g = np.random.Generator(np.random.PCG64(7))
    r, B, C, H, W = 20, 21, 24, 21, 13
    dY = inputs.round_to_storage((0.1 * g.standard_normal((B, C, H, W))).astype(np.float32), dtype)
    scale = 2.0 ** np.arange(-12, 20, 1.6)[:r, None]                # rows of very different size
    S = (scale * (1.0 + g.random((r, B)))).astype(np.float32)
    if dtype == "f16":
        S[-1] *= np.float32(2.0 ** -3)                              # entries beyond 65504, sums within
    L = host(xb.xconv_backprobe(torch.from_numpy(S).cuda(), xb.to_device(dY, dtype)))
    want = O.backprobe(S, dY)
    for j in range(2 if dtype == "f16" else 0, r):                  # (the smallest float16 rows are subnormal)
        if np.abs(want[j]).max() < 6e4 or dtype == "bf16":
            assert O.rel_fro(L[j], want[j]) < bar, j
