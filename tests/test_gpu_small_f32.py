"""The kernels of small float layers (small_f32.cu) at the edges of their tiles: strips of four pixels that overhang the row, a last block of strips that is not full,
channel counts off the tiles of 16 and 32 and off the 8 or 16 that go through shared memory together, blocks that split the channels in and blocks that do not,
volumes, one work item and several per block of the contraction, circular shifts there, infinities and NaN; the library is asked whether these kernels serve a layer.
Bars as in test_gpu_parity.py for float storage."""
import itertools

import pytest
import torch

import __graft_entry__ as entry
from paper_2106_06998_b200 import binding as xb
from tests._util import TOL, check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


def _tensors(B, Cin, Cout, geo, r, K, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    fmt = torch.channels_last if len(geo) == 2 else torch.channels_last_3d
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").contiguous(memory_format=fmt)
    return rnd(B, Cin, *geo), rnd(B, Cout, *geo), rnd(Cout, Cin, *([K] * len(geo))), rnd(r, Cin, *geo), rnd(r, Cout, *geo)


LAYERS = [
    (1, 4, 4, (1, 1), 1, 3), (8, 16, 16, (32, 32), 8, 3), (3, 20, 36, (9, 13), 5, 3), (2, 128, 16, (9, 7), 3, 3), (30, 16, 12, (24, 23), 4, 3),
    (6, 12, 40, (11, 10), 4, 5), (30, 8, 16, (19, 18), 3, 5), (7, 64, 48, (7, 9), 6, 1), (128, 16, 20, (15, 14), 3, 1), (1, 256, 8, (5, 3), 2, 1),
    (2, 24, 16, (8, 9, 11), 4, 3), (3, 4, 20, (2, 5, 6), 3, 3), (12, 8, 8, (5, 12, 10), 2, 3),
]


def _small(op, B, Cin, Cout, geo, r, K, circular=False):
    D = geo[0] if len(geo) == 3 else 1
    return "small_tiles" in xb.variants_for(xb.make_desc(B, Cin, Cout, geo[-2], geo[-1], r, torch.float32, K, D=D, KD=K if D > 1 else 1, circular=circular), op)


@pytest.mark.parametrize("B,Cin,Cout,geo,r,K", LAYERS)
def test_small_convolution_and_input_gradient(B, Cin, Cout, geo, r, K):
    X, dY, W, Z, _ = _tensors(B, Cin, Cout, geo, r, K, 3)
    assert _small(xb.OP_FORWARD, B, Cin, Cout, geo, r, K) and _small(xb.OP_DGRAD, B, Cin, Cout, geo, r, K)
    Y, _ = xb.xconv_forward(X, W, Z)
    dX = xb.xconv_dgrad(dY, W)
    f = torch.nn.functional
    conv, back = (f.conv3d, f.conv_transpose3d) if len(geo) == 3 else (f.conv2d, f.conv_transpose2d)
    wide = lambda t: t.double().cpu().numpy()
    check("Y", wide(Y), wide(conv(X.double(), W.double(), padding=(K - 1) // 2)), TOL["f32"])
    check("dX", wide(dX), wide(back(dY.double(), W.double(), padding=(K - 1) // 2)), TOL["f32"])


# (Cin, Cout, image, probes, kernel)
CONTRACTIONS = [
    (4, 4, (1, 1), 1, 3), (16, 16, (32, 32), 8, 3), (20, 36, (9, 13), 5, 3), (128, 16, (9, 7), 3, 3), (12, 40, (11, 10), 4, 5), (8, 16, (19, 18), 3, 5), (16, 20, (15, 14), 3, 1),
    (256, 8, (5, 3), 2, 1), (16, 16, (40, 65), 2, 3), (4, 20, (33, 40), 1, 5), (24, 16, (8, 9, 11), 1, 3), (4, 20, (2, 5, 6), 3, 3), (8, 8, (5, 12, 10), 1, 3),
]


@pytest.mark.parametrize("Cin,Cout,geo,r,K,circular", [c + (False,) for c in CONTRACTIONS] + [c + (True,) for c in CONTRACTIONS if len(c[2]) == 2])
def test_small_contraction(Cin, Cout, geo, r, K, circular):
    _, _, _, Z, L = _tensors(1, Cin, Cout, geo, r, K, 4)
    assert _small(xb.OP_CONTRACT, 1, Cin, Cout, geo, r, K, circular)
    got = xb.xconv_contract(L, Z, K, kernel_depth=K if len(geo) == 3 else 1, circular=circular)
    p = (K - 1) // 2
    Zd, Ld, dims = Z.double(), L.double(), tuple(range(2, 2 + len(geo)))
    Zp = torch.nn.functional.pad(Zd, (p,) * (2 * len(geo)))
    want = torch.zeros(got.shape, dtype=torch.float64, device="cuda")
    for k in itertools.product(range(K), repeat=len(geo)):
        moved = (torch.roll(Zd, tuple(p - o for o in k), dims) if circular
                 else Zp[(slice(None), slice(None)) + tuple(slice(o, o + n) for o, n in zip(k, geo))])
        want[(slice(None), slice(None)) + k] = torch.einsum("jmq,jnq->mn", Ld.flatten(2), moved.flatten(2)) / r
    check("dW", got.double().cpu().numpy(), want.cpu().numpy(), TOL["f32"])


@pytest.mark.parametrize("B,Cin,Cout,geo,r,K", [LAYERS[i] for i in (1, 2, 3, 5, 7, 10)])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_values_that_are_not_finite_stay_where_they_belong(B, Cin, Cout, geo, r, K, bad):
    """In the convolutions every other result keeps its bits; in the contraction those of other channels do (see include/xconv.h)."""
    X, dY, W, Z, _ = _tensors(B, Cin, Cout, geo, r, K, 5)
    for at in ((0,) * len(geo), tuple(n - 1 for n in geo), tuple(n // 2 for n in geo)):
        hit = torch.zeros((B,) + geo, dtype=torch.bool, device="cuda")
        hit[(B - 1,) + tuple(slice(max(0, q - K // 2), q + K // 2 + 1) for q in at)] = True
        for f, t in ((lambda x: xb.xconv_forward(x, W, Z)[0], X), (lambda y: xb.xconv_dgrad(y, W), dY)):
            worse = t.clone()
            worse[(B - 1, t.shape[1] - 1) + at] = bad
            got, want = f(worse).movedim(1, -1), f(t).movedim(1, -1)
            assert torch.equal(got[~hit], want[~hit]) and not torch.isfinite(got[hit]).any()


@pytest.mark.parametrize("Cin,Cout,geo,r,K", [CONTRACTIONS[i] for i in (1, 2, 4, 6, 11)])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_small_contraction_of_values_that_are_not_finite(Cin, Cout, geo, r, K, bad):
    _, _, _, Z, L = _tensors(1, Cin, Cout, geo, r, K, 6)
    assert _small(xb.OP_CONTRACT, 1, Cin, Cout, geo, r, K)
    call = lambda l, z: xb.xconv_contract(l, z, K, kernel_depth=K if len(geo) == 3 else 1)
    want, centre = call(L, Z), (K // 2,) * len(geo)
    for at in ((0,) * len(geo), tuple(n - 1 for n in geo), tuple(n // 2 for n in geo)):
        Z2, L2 = Z.clone(), L.clone()
        Z2[(r - 1, 2) + at] = bad
        L2[(0, Cout - 1) + at] = bad
        dW, others = call(L, Z2), [n for n in range(Cin) if n != 2]
        assert torch.equal(dW[:, others], want[:, others]) and not torch.isfinite(dW[(slice(None), 2) + centre]).any()
        dW = call(L2, Z)
        assert torch.equal(dW[:-1], want[:-1]) and not torch.isfinite(dW[(-1, slice(None)) + centre]).any()
