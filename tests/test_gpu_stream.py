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
    ("f16", 4, 8, 8, 17, 19),        # columns that end inside a group
    ("bf16", 16, 31, 64, 9, 9),      # 16 rows
    ("f16", 9, 64, 8, 24, 24),       # (a multiple of 8 terms, of 64 columns: S rounded once)
    ("bf16", 12, 70, 128, 50, 50),   # the second round of terms mostly padding; two groups per warp
    ("bf16", 20, 21, 24, 11, 13),    # 32 rows
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


# Half a unit in the last place of the storage type: what the rounding of the result alone leaves, as a relative 2-norm.
ROUNDING = {"bf16": 2.0 ** -9, "f16": 2.0 ** -12}


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("r,B,C,H,W,rounded", [
    (4, 8, 16, 17, 20, True),        # one k-step in one go, half of it padding
    (16, 16, 64, 5, 7, True),        # one whole k-step
    (9, 24, 64, 9, 9, True),         # two, the second half padding
    (16, 32, 8, 24, 24, True),       # two whole ones
    (3, 40, 64, 9, 9, True),         # four, the last one padding
    (16, 64, 8, 24, 24, True),
    (12, 72, 128, 50, 52, True),     # a loop over the terms, two groups per warp
    (16, 200, 64, 72, 72, True),
    (16, 9, 64, 5, 7, False),        # 16 rows, S as two values
    (12, 70, 128, 50, 52, False),
    (17, 33, 24, 11, 13, False),     # 32 rows
    (64, 65, 8, 17, 16, False),      # 64 rows
])
def test_backprobe_by_the_rounding_of_the_sketch(dtype, r, B, C, H, W, rounded):
    """Which kernel a layer reaches shows in what is multiplied: S rounded to storage where the tcgen05 back-probe serves the
    layer too (terms a multiple of 8, columns of 64), the float S elsewhere.  The entries of S lie a quarter of a unit off a
    16-bit value, in one direction: against the wrong one of the two L is off by that (2^-9, 2^-12) and its rounding."""
    assert rounded == (B % 8 == 0 and (C * H * W) % 64 == 0)
    g = np.random.Generator(np.random.PCG64([r, B, C, H, W, 1]))
    dY = inputs.round_to_storage((0.1 * g.standard_normal((B, C, H, W))).astype(np.float32), dtype)
    unit = 2.0 ** -7 if dtype == "bf16" else 2.0 ** -10
    S16 = inputs.round_to_storage((g.choice([-1.0, 1.0], (r, B)) * g.uniform(1.0, 1.99, (r, B))).astype(np.float32), dtype)
    S = (S16 * (1.0 + 0.25 * unit)).astype(np.float32)
    assert np.array_equal(inputs.round_to_storage(S, dtype), S16)
    want, other = (O.backprobe(S16 if q else S, dY) for q in (rounded, not rounded))
    L = host(xb.xconv_backprobe(torch.from_numpy(S).cuda(), xb.to_device(dY, dtype)))
    assert O.rel_fro(L, want) < ROUNDING[dtype] < O.rel_fro(L, other)


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


def test_a_call_of_streaming_kernels_alone_reports_its_own_outcome():
    """On scratch memory whose header a timed-out call has written, through every streaming kernel by itself."""
    lay = inputs.make_custom(4, 64, 64, 9, 9, 8, dtype="bf16", seed=3, z="gaussian", x="normal")
    X, Z, dY = (xb.to_device(lay[k], "bf16") for k in ("X", "Z", "dY"))
    desc = xb.make_desc(4, 64, 64, 9, 9, 8, torch.bfloat16)
    ws = torch.zeros(max(xb.workspace_bytes(desc, o) for o in (xb.OP_SKETCH, xb.OP_SKETCH_SEEDED, xb.OP_WGRAD)), dtype=torch.uint8, device="cuda")
    S, L = torch.empty((8, 4), device="cuda"), torch.empty((8, 64, 9, 9), dtype=torch.bfloat16, device="cuda", memory_format=torch.channels_last)
    for call in (lambda: xb.sketch_into(desc, X, Z, S, ws), lambda: xb.sketch_seeded_into(desc, X, 7, S, ws),
                 lambda: xb.backprobe_into(desc, S, dY, L, ws)):
        assert xb.lib().xconv_selftest_wait_limit(ws.data_ptr(), ws.numel(), 5, torch.cuda.current_stream().cuda_stream) == 0
        assert xb.workspace_status(ws) == 6                      # XCONV_ERR_TIMEOUT
        call()
        assert xb.workspace_status(ws) == 0
