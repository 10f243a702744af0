"""The convolutions that walk along an axis (conv_slide.cuh), at the edges of their walk: runs of outputs that start and end inside a column, columns shorter
than the kernel, rows of several images in a tile with a last group that is not full, several blocks of channels, accumulators whose ring ends
inside an MMA, rows longer than a tile, volumes; infinities and NaN at the ends of runs; and the layers done in patches beside them, some with more than four
input boxes in flight.  Each case says which of its two convolutions walks, and the library is asked.  Bars as in test_gpu_parity.py: one rounding to
the storage type."""
import pytest
import torch

import __graft_entry__ as entry
from paper_2106_06998_b200 import binding as xb
from tests._util import MAX_C, TOL

gpu = pytest.mark.gpu
TYPES = {"bf16": torch.bfloat16, "f16": torch.float16}


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    if torch.cuda.is_available():
        torch.cuda.set_device(0)


# (storage, B, Cin, Cout, D, H, W, K, what walks: F the convolution, D the input gradient)
WALKED = [
    ("bf16", 13, 32, 32, 1, 131, 128, 3, "FD"),      # one tile a row, runs that end inside an image
    ("f16", 17, 32, 24, 1, 101, 257, 3, "FD"),       # rows of three tiles, the last nearly empty; channels out off the block
    ("bf16", 481, 16, 16, 1, 33, 30, 3, "FD"),       # four images a tile, and a last group of one
    ("f16", 451, 24, 16, 1, 40, 30, 3, "FD"),        # ... of three
    ("bf16", 7, 8, 8, 1, 90, 120, 3, "FD"),          # half a k-step of channels, the smallest number of channels out
    ("f16", 81, 16, 16, 1, 67, 70, 5, "FD"),         # 25 offsets, a ring of 32 or 16
    ("bf16", 28, 16, 16, 1, 40, 259, 5, "FD"),       # ... rows of three tiles
    ("bf16", 7, 64, 48, 1, 50, 100, 5, "F"),         # ... four k-steps; 240 columns an MMA, a ring of ten
    ("f16", 61, 64, 64, 1, 64, 120, 3, "FD"),        # 192 columns, a ring of eight
    ("f16", 27, 16, 80, 1, 61, 120, 3, "F"),         # 240 columns, a ring of six
    ("bf16", 1936, 32, 32, 1, 2, 64, 3, "FD"),       # images of fewer rows than the kernel has
    ("f16", 701, 32, 32, 1, 4, 64, 5, "FD"),         # ...
    ("bf16", 13, 32, 32, 33, 20, 24, 3, "FD"),       # volumes
    ("f16", 13, 32, 80, 5, 30, 40, 3, "FD"),         # ... a ring of six
    ("f16", 121, 48, 16, 2, 40, 50, 3, "F"),         # ... of fewer planes than the kernel has
    ("bf16", 12, 24, 48, 2, 40, 50, 3, "D"),         # ...
    ("bf16", 9, 64, 24, 27, 33, 40, 3, "FD"),        # ... whose weights were streamed
    ("bf16", 5, 96, 24, 22, 34, 34, 3, "F"),         # ... two blocks of channels,
    ("f16", 5, 24, 96, 9, 22, 34, 3, "D"),           # ... of the input gradient,
    ("f16", 5, 160, 16, 9, 22, 34, 3, "F"),          # ... three, narrow ones
]
PATCHES = [
    ("bf16", 3, 32, 32, 1, 131, 128, 3, ""), ("f16", 2, 32, 24, 1, 101, 257, 3, ""), ("bf16", 160, 16, 16, 1, 33, 30, 3, ""), ("f16", 149, 24, 16, 1, 40, 30, 3, ""),
    ("bf16", 5, 8, 8, 1, 90, 120, 3, ""), ("f16", 20, 16, 16, 1, 67, 70, 5, ""), ("bf16", 4, 136, 32, 1, 60, 110, 3, ""), ("f16", 7, 64, 64, 1, 64, 120, 3, ""),
    ("bf16", 3, 32, 32, 33, 20, 24, 3, ""), ("f16", 30, 48, 16, 2, 40, 50, 3, ""), ("bf16", 2, 64, 24, 27, 33, 40, 3, ""),
    ("f16", 19, 72, 8, 1, 131, 128, 1, ""),          # pointwise: sixteen patches a CTA and some CTAs with fewer, two blocks of channels
    ("bf16", 46, 192, 24, 1, 129, 129, 1, ""),       # ... forty, three blocks, a last patch of few pixels
    ("f16", 37, 24, 64, 1, 83, 83, 3, "D"),          # patches, whose input gradient walks
    ("bf16", 9, 96, 16, 1, 133, 131, 3, ""),         # more than four boxes in flight
]


def _walks(dtype, B, Cin, Cout, D, H, W, K):
    desc = xb.make_desc(B, Cin, Cout, H, W, 1, TYPES[dtype], K, D=D, KD=K if D > 1 else 1)
    return "".join(n for n, op in (("F", xb.OP_FORWARD), ("D", xb.OP_DGRAD)) if "walk" in xb.variants_for(desc, op))


@pytest.mark.parametrize("case", WALKED + PATCHES)
def test_what_walks(case):
    assert _walks(*case[:-1]) == case[-1]


def _draw(dtype, B, Cin, Cout, D, H, W, K, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    geo, fmt = ((D, H, W), torch.channels_last_3d) if D > 1 else ((H, W), torch.channels_last)
    rnd = lambda scale, *s: (torch.randn(s, generator=g, device="cuda") * scale).to(TYPES[dtype]).contiguous(memory_format=fmt)
    kgeo = (K,) * len(geo)
    return rnd(1.0, B, Cin, *geo), rnd(1.0, B, Cout, *geo), rnd((2.0 / (Cin * K ** len(geo))) ** 0.5, Cout, Cin, *kgeo), torch.ones_like(rnd(1.0, 1, Cin, *geo))


def _close(name, got, want, tol):
    """As tests._util.check, on the device."""
    diff = got.double() - want
    rms = want.pow(2).mean().sqrt()
    assert diff.norm() <= tol * want.norm(), name
    assert diff.abs().max() <= MAX_C * tol * rms, name


@gpu
@pytest.mark.parametrize("case", WALKED + PATCHES)
def test_convolution_and_input_gradient_against_64_bits(case):
    dtype, B, Cin, Cout, D, H, W, K, _ = case
    X, dY, Wt, Z = _draw(dtype, B, Cin, Cout, D, H, W, K, 11)
    Y, _ = xb.xconv_forward(X, Wt, Z)
    dX = xb.xconv_dgrad(dY, Wt)
    conv, back = (torch.nn.functional.conv3d, torch.nn.functional.conv_transpose3d) if D > 1 else (torch.nn.functional.conv2d, torch.nn.functional.conv_transpose2d)
    for name, got, f, t in (("Y", Y, conv, X), ("dX", dX, back, dY)):
        want = torch.cat([f(t[i:i + 64].double().contiguous(), Wt.double().contiguous(), padding=(K - 1) // 2) for i in range(0, B, 64)])
        _close(name, got, want, TOL[dtype])


@gpu
@pytest.mark.parametrize("case", [WALKED[i] for i in (0, 2, 5, 8, 10, 12, 14, 17)])
@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
def test_values_that_are_not_finite_stay_where_they_belong(case, bad):
    """An entry that is not finite makes what it enters not finite, and every other result keeps its bits: at the corners, in the middle, at the first and last
    position along the axis that the runs are cut from, and at an arbitrary place in the last image."""
    dtype, B, Cin, Cout, D, H, W, K, _ = case
    X, dY, Wt, Z = _draw(dtype, B, Cin, Cout, D, H, W, K, 12)
    geo = (D, H, W) if D > 1 else (H, W)
    places = [(0,) * len(geo), tuple(n - 1 for n in geo), tuple(n // 2 for n in geo), (0,) + tuple(n // 2 for n in geo[1:]), (geo[0] - 1,) + tuple(n // 3 for n in geo[1:])]
    for f, t in ((lambda x: xb.xconv_forward(x, Wt, Z)[0], X), (lambda y: xb.xconv_dgrad(y, Wt), dY)):
        want = f(t)
        assert torch.isfinite(want).all()
        worse, hit = t.clone(), torch.zeros((B,) + geo, dtype=torch.bool, device="cuda")
        for i, place in enumerate(places):
            b = (B - 1) * i // (len(places) - 1)
            worse[(b, i % t.shape[1]) + place] = bad
            hit[(b,) + tuple(slice(max(0, q - K // 2), q + K // 2 + 1) for q in place)] = True
        got = f(worse).movedim(1, -1)
        assert torch.equal(got[~hit], want.movedim(1, -1)[~hit]) and not torch.isfinite(got[hit]).any()
