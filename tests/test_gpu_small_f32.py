"""The kernels of small float layers (small_f32.cu) at the edges of their tiles: strips of four pixels that overhang the row, a last block of strips that is not full,
channel counts off the tiles of 16 and 32 and off the 8 or 16 that go through shared memory together, blocks that split the channels in and blocks that do not,
volumes, one work item and several per block of the contraction, and circular shifts there.  Bars as in test_gpu_parity.py for float storage."""
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


@pytest.mark.parametrize("B,Cin,Cout,geo,r,K", LAYERS)
def test_small_convolution_and_input_gradient(B, Cin, Cout, geo, r, K):
    X, dY, W, Z, _ = _tensors(B, Cin, Cout, geo, r, K, 3)
    D = geo[0] if len(geo) == 3 else 1
    desc = xb.make_desc(B, Cin, Cout, geo[-2], geo[-1], r, torch.float32, K, D=D, KD=K if D > 1 else 1)
    assert xb.engine_for(desc, xb.OP_FORWARD) == "simt_f32" and xb.engine_for(desc, xb.OP_DGRAD) == "simt_f32"
    Y, _ = xb.xconv_forward(X, W, Z)
    dX = xb.xconv_dgrad(dY, W)
    f = torch.nn.functional
    conv, back = (f.conv3d, f.conv_transpose3d) if D > 1 else (f.conv2d, f.conv_transpose2d)
    wide = lambda t: t.double().cpu().numpy()
    check("Y", wide(Y), wide(conv(X.double(), W.double(), padding=(K - 1) // 2)), TOL["f32"])
    check("dX", wide(dX), wide(back(dY.double(), W.double(), padding=(K - 1) // 2)), TOL["f32"])


@pytest.mark.parametrize("circular", [False, True])
@pytest.mark.parametrize("B,Cin,Cout,geo,r,K", [l for l in LAYERS if l[3] != (24, 23)] + [(1, 16, 16, (40, 65), 3, 3), (1, 4, 20, (33, 40), 2, 5)])
def test_small_contraction(B, Cin, Cout, geo, r, K, circular):
    D = geo[0] if len(geo) == 3 else 1
    if circular and D > 1:
        pytest.skip("circular shifts are planar")
    _, _, _, Z, L = _tensors(B, Cin, Cout, geo, r, K, 4)
    KD = K if D > 1 else 1
    if xb.engine_for(xb.make_desc(1, Cin, Cout, geo[-2], geo[-1], r, torch.float32, K, D=D, KD=KD, circular=circular), xb.OP_CONTRACT) != "simt_f32":
        pytest.skip("not small")
    got = xb.xconv_contract(L, Z, K, kernel_depth=KD, circular=circular)
    p = (K - 1) // 2
    Zd, Ld = Z.double(), L.double()
    if circular:
        Zp = torch.nn.functional.pad(Zd, (p,) * 4, mode="circular") if min(geo) >= p else None
        if Zp is None:
            pytest.skip("shift beyond the image")
    else:
        Zp = torch.nn.functional.pad(Zd, (p,) * (2 * len(geo)))
    want = torch.zeros(got.shape, dtype=torch.float64, device="cuda")
    for k in itertools.product(range(K), repeat=len(geo)):
        moved = Zp[(slice(None), slice(None)) + tuple(slice(o, o + n) for o, n in zip(k, geo))]
        want[(slice(None), slice(None)) + k] = torch.einsum("jmq,jnq->mn", Ld.flatten(2), moved.flatten(2)) / r
    check("dW", got.double().cpu().numpy(), want.cpu().numpy(), TOL["f32"])
