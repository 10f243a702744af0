"""Sketches and back-probes of long rows (tc_kernels.cu: operands copied in boxes of eight rows), on whole numbers: signs times samples of
-3 .. 3 sum to less than 2^24, so the sketch is exact in any order of summation; a back-probe of whole numbers is its exact sum rounded once."""
import pytest
import torch

import __graft_entry__ as entry
from paper_2106_06998_b200 import binding as xb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("dtype,r,B,C,H,W", [
    ("bf16", 72, 16, 64, 96, 128),        # the shortest row served; the last box of eight rows is the ninth
    ("f16", 71, 3, 64, 97, 128),          # rows that are no whole box, on either side; k-blocks that are no whole stage
    ("bf16", 9, 70, 64, 95, 128),         # one k-block less than the line: one box of all rows
    ("bf16", 70, 33, 8, 1001, 104),       # k-blocks: no multiple of four
    ("f16", 130, 65, 64, 100, 131),       # two tiles of probes, the second of two; stages of two k-blocks
    ("bf16", 140, 67, 64, 101, 127),      # ... 80 columns
    ("bf16", 66, 258, 64, 96, 129),       # samples on the MMA rows, three tiles
    ("f16", 66, 1, 64, 129, 96),          # a single sample
])
def test_sketch_of_long_rows_is_exact(dtype, r, B, C, H, W):
    g = torch.Generator(device="cuda").manual_seed(r * 1000 + B)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float16
    X = torch.randint(-3, 4, (B, H, W, C), generator=g, device="cuda", dtype=torch.int8).to(dt)
    Z = (torch.randint(0, 2, (r, H, W, C), generator=g, device="cuda", dtype=torch.int8) * 2 - 1).to(dt)
    S = xb.xconv_sketch(X.permute(0, 3, 1, 2), Z.permute(0, 3, 1, 2))      # (channels last, as the data lies)
    want = torch.zeros(r, B, dtype=torch.float64, device="cuda")
    for j in range(0, r, 16):
        want[j:j + 16] = Z[j:j + 16].reshape(-1, H * W * C).double() @ X.reshape(B, -1).double().T
    assert torch.equal(S.double().reshape(r, B), want)


@pytest.mark.parametrize("dtype,r,B,C,H,W", [
    ("bf16", 72, 66, 64, 128, 128),       # the shortest row served; two stages of samples, the second of two rows
    ("f16", 131, 128, 64, 127, 131),      # blocks that are no multiple of four; three rows in the second tile of probes
    ("bf16", 300, 21, 32, 257, 130),      # one stage of two k-steps, its last box of eight rows past the samples
    ("bf16", 65, 130, 64, 128, 127),      # below the line: boxes of all rows
])
def test_backprobe_of_long_rows_is_rounded_once(dtype, r, B, C, H, W):
    g = torch.Generator(device="cuda").manual_seed(r * 1000 + B)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float16
    S = torch.randint(-8, 9, (r, B), generator=g, device="cuda").float()
    dY = torch.randint(-3, 4, (B, H, W, C), generator=g, device="cuda", dtype=torch.int8).to(dt)
    L = xb.xconv_backprobe(S, dY.permute(0, 3, 1, 2))
    want = (S.double() @ dY.reshape(B, -1).double()).to(dt)
    assert torch.equal(L.permute(0, 2, 3, 1).reshape(r, -1), want)
