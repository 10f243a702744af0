"""Float sketches and back-probes whose stages are converted by teams of warps in turn (gemm_split.cu), with as many k-blocks a CTA as make the
teams' last turns differ; and sums of many splits with 32 threads to an output, of each kernel that leaves such.  Whole numbers: every product and partial sum is exact, so the results are too."""
import pytest
import torch

import __graft_entry__ as entry
from paper_2106_06998_b200 import binding as xb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("r,B,C,H,W", [
    (64, 64, 32, 12, 12),       # one k-block a CTA at most
    (64, 64, 32, 16, 16),       # two for some
    (70, 33, 32, 20, 22),       # three
    (128, 64, 32, 37, 17),      # four and five, the largest boxes
    (16, 130, 36, 41, 23),      # a last k-block of 12 terms; two row tiles, seven and eight blocks
    (300, 100, 8, 61, 60),      # three row tiles, two column tiles
    (64, 16, 32, 128, 128),     # a hundred
])
def test_float_sketch_of_whole_numbers_is_exact(r, B, C, H, W):
    g = torch.Generator(device="cuda").manual_seed(r * 1000 + B)
    X = torch.randint(-9, 10, (B, H, W, C), generator=g, device="cuda").float()
    Z = (torch.randint(0, 2, (r, H, W, C), generator=g, device="cuda") * 2 - 1).float()
    S = xb.xconv_sketch(X.permute(0, 3, 1, 2), Z.permute(0, 3, 1, 2))
    assert torch.equal(S.double(), Z.reshape(r, -1).double() @ X.reshape(B, -1).double().T)


@pytest.mark.parametrize("r,B,C,H,W", [
    (64, 16, 32, 40, 40),       # one k-block a tile
    (33, 130, 32, 64, 64),      # five, the last of two terms; rows of S off the column group
    (64, 200, 16, 100, 100),    # seven
    (130, 70, 32, 50, 50),      # three column tiles
])
def test_float_backprobe_of_whole_numbers_is_exact(r, B, C, H, W):
    g = torch.Generator(device="cuda").manual_seed(r * 1000 + B)
    S = torch.randint(-8, 9, (r, B), generator=g, device="cuda").float()
    dY = torch.randint(-9, 10, (B, H, W, C), generator=g, device="cuda").float()
    L = xb.xconv_backprobe(S, dY.permute(0, 3, 1, 2))
    assert torch.equal(L.permute(0, 2, 3, 1).reshape(r, -1).double(), S.double() @ dY.reshape(B, -1).double())


@pytest.mark.parametrize("dtype,r,B,C,H,W,wide", [
    ("f32", 7, 3, 16, 32, 32, True),          # multiply-adds; a last block of five outputs
    ("f32", 96, 98, 32, 64, 64, True),        # split operands, nearly the most outputs that 32 threads share
    ("f32", 97, 98, 32, 64, 64, False),       # ... and some of the first that eight share; a last block of two
    ("f32", 70, 33, 32, 128, 128, True),
    ("f32", 128, 128, 32, 64, 64, False),     # ... the most that are added in pairs
    ("f32", 129, 128, 32, 64, 64, False),     # ... and the first that are not
    ("bf16", 101, 5, 16, 64, 64, True),       # in a stream
    ("bf16", 2001, 5, 16, 64, 64, False),
])
def test_sums_of_many_splits_are_exact(dtype, r, B, C, H, W, wide):
    storage = torch.float32 if dtype == "f32" else torch.bfloat16
    assert ("wide_sums" in xb.variants_for(xb.make_desc(B, C, 1, H, W, r, storage), xb.OP_SKETCH)) == wide
    g = torch.Generator(device="cuda").manual_seed(r * 1000 + B)
    X = torch.randint(-9, 10, (B, H, W, C), generator=g, device="cuda").to(storage)
    Z = (torch.randint(0, 2, (r, H, W, C), generator=g, device="cuda") * 2 - 1).to(storage)
    S = xb.xconv_sketch(X.permute(0, 3, 1, 2), Z.permute(0, 3, 1, 2))
    assert torch.equal(S.double(), Z.reshape(r, -1).double() @ X.reshape(B, -1).double().T)
