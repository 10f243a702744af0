"""Sketches and back-probes of long rows (tc_kernels.cu: operands copied in boxes of eight rows), on whole numbers: signs times samples of
-3 .. 3 sum to less than 2^24, so the sketch is exact in any order of summation; a back-probe of whole numbers is its exact sum rounded once.
Each case says whether it takes the boxes, and the library is asked."""
import pytest
import torch

import __graft_entry__ as entry
from paper_2106_06998_b200 import binding as xb

pytestmark = pytest.mark.gpu
TYPES = {"bf16": torch.bfloat16, "f16": torch.float16}
INF = float("inf")


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


def _boxes(op, *layer):
    return "row_boxes" in xb.variants_for(xb.make_desc(*layer), op)


def _samples(dtype, r, B, C, H, W):
    g = torch.Generator(device="cuda").manual_seed(r * 1000 + B)
    X = torch.randint(-3, 4, (B, H, W, C), generator=g, device="cuda", dtype=torch.int8).to(TYPES[dtype])
    Z = (torch.randint(0, 2, (r, H, W, C), generator=g, device="cuda", dtype=torch.int8) * 2 - 1).to(TYPES[dtype])
    return X.permute(0, 3, 1, 2), Z.permute(0, 3, 1, 2)                   # (channels last, as the data lies)


@pytest.mark.parametrize("dtype,r,B,C,H,W,boxes", [
    ("bf16", 72, 16, 64, 96, 128, True),       # the shortest row served; the last box of eight rows is the ninth
    ("f16", 71, 3, 64, 97, 128, True),         # rows that are no whole box, on either side; k-blocks that are no whole stage
    ("bf16", 9, 70, 64, 95, 128, False),       # one k-block less than the line: one box of all rows
    ("bf16", 70, 33, 8, 1001, 104, True),      # k-blocks: no multiple of four
    ("f16", 130, 65, 64, 100, 131, True),      # two tiles of probes, the second of two; stages of two k-blocks
    ("bf16", 140, 67, 64, 101, 127, True),     # ... 80 columns
    ("bf16", 66, 258, 64, 96, 129, True),      # samples on the MMA rows, three tiles
    ("f16", 66, 1, 64, 129, 96, True),         # a single sample
])
def test_sketch_of_long_rows_is_exact(dtype, r, B, C, H, W, boxes):
    assert _boxes(xb.OP_SKETCH, B, C, 1, H, W, r, TYPES[dtype]) == boxes
    X, Z = _samples(dtype, r, B, C, H, W)
    S = xb.xconv_sketch(X, Z)
    flat = lambda t: t.permute(0, 2, 3, 1).reshape(len(t), -1).double()
    want = torch.cat([flat(Z[j:j + 16]) @ flat(X).T for j in range(0, r, 16)])
    assert torch.equal(S.double().reshape(r, B), want)


@pytest.mark.parametrize("dtype,r,B,C,H,W,boxes", [
    ("bf16", 72, 72, 64, 128, 128, True),      # the shortest row served; two stages of samples, the second of eight rows
    ("f16", 131, 128, 64, 127, 131, True),     # blocks that are no multiple of four; three rows in the second tile of probes
    ("bf16", 300, 24, 32, 257, 130, True),     # one stage of two k-steps, its last box of eight rows past the samples
    ("f16", 66, 8, 64, 129, 128, True),        # ... of one k-step, half of it past the samples
    ("bf16", 65, 136, 64, 128, 127, False),    # below the line: boxes of all rows
    ("bf16", 72, 66, 64, 128, 128, False),     # samples off the multiples of 8: another kernel
])
def test_backprobe_of_long_rows_is_rounded_once(dtype, r, B, C, H, W, boxes):
    assert _boxes(xb.OP_BACKPROBE, B, 1, C, H, W, r, TYPES[dtype]) == boxes
    g = torch.Generator(device="cuda").manual_seed(r * 1000 + B)
    S = torch.randint(-8, 9, (r, B), generator=g, device="cuda").float()
    dY = torch.randint(-3, 4, (B, H, W, C), generator=g, device="cuda", dtype=torch.int8).to(TYPES[dtype])
    L = xb.xconv_backprobe(S, dY.permute(0, 3, 1, 2))
    want = (S.double() @ dY.reshape(B, -1).double()).to(TYPES[dtype])
    assert torch.equal(L.permute(0, 2, 3, 1).reshape(r, -1), want)


@pytest.mark.parametrize("dtype,B,r", [("bf16", 24, 64), ("f16", 66, 72)])
def test_redrawn_probes_give_the_bits_of_stored_ones_in_boxes(dtype, B, r):
    """Summed over the probes first, the stored ones are copied in boxes of eight rows and the redrawn ones are not."""
    Cin, Cout, H, W = 64, 8, 128, 129
    layer = (B, Cin, Cout, H, W, r, TYPES[dtype])
    assert _boxes(xb.OP_WGRAD, *layer) and not _boxes(xb.OP_WGRAD_SEEDED, *layer)
    g = torch.Generator(device="cuda").manual_seed(B)
    dY = (torch.randn(B, H, W, Cout, generator=g, device="cuda") * 0.1).to(TYPES[dtype]).permute(0, 3, 1, 2)
    S = torch.randn(r, B, generator=g, device="cuda")
    Z = xb.xconv_probes_from_seed(77, r, Cin, H, W, TYPES[dtype])
    assert torch.equal(xb.xconv_wgrad_seeded(S, dY, 77, Cin), xb.xconv_wgrad(S, dY, Z))


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("bad", [INF, -INF, float("nan")])
def test_values_that_are_not_finite_stay_where_they_belong(dtype, bad):
    r, B, C, H, W = 71, 9, 64, 97, 128
    X, Z = _samples(dtype, r, B, C, H, W)
    want = xb.xconv_sketch(X, Z)
    X[0, 0, 0, 0] = X[B - 1, C - 1, H - 1, W - 1] = X[4, 3, 50, 60] = bad
    S = xb.xconv_sketch(X, Z)
    hit = [0, 4, B - 1]
    others = [b for b in range(B) if b not in hit]
    assert torch.equal(S[:, others], want[:, others])
    signs = torch.stack([Z[:, 0, 0, 0], Z[:, 3, 50, 60], Z[:, C - 1, H - 1, W - 1]], dim=1).float()
    assert torch.isnan(S[:, hit]).all() if bad != bad else torch.equal(S[:, hit], signs * bad)
    r, B, C, H, W = 72, 72, 64, 128, 128
    S = torch.ones(r, B, device="cuda")
    S[1] = -1.0
    dY = torch.ones(B, H, W, C, device="cuda", dtype=TYPES[dtype])
    dY[B - 1, H - 1, W - 1, C - 1] = dY[3, 0, 0, 0] = bad
    L = xb.xconv_backprobe(S, dY.permute(0, 3, 1, 2)).permute(0, 2, 3, 1).reshape(r, -1).float()
    sign = torch.sign(S[:, :1])
    assert torch.equal(L[:, 1:-1], (sign * B).expand(r, L.shape[1] - 2))
    assert torch.isnan(L[:, [0, -1]]).all() if bad != bad else torch.equal(L[:, [0, -1]], (sign * bad).expand(r, 2))
