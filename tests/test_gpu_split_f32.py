"""The float kernels on the tensor cores (three bfloat16 parts a float): edges of their tiles, channel counts that are no multiple of
four, every form of the contraction's rows, calls whose scratch is too small for them, and values that cannot be split.

Bounds against 64 bits.  A product's parts leave out 2^-24 of it, an accumulator loses at most 2^-23 of its value an MMA (rounded
towards zero) over chains of at most ten (in the contraction thirty, of which the last five are at full size: the products of the small
parts come first), and chains are added in float, one rounding of 2^-24 each: with random signs below 6e-7 of the result's norm for the
sums taken here (a few million products)."""
import ctypes

import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from oracle import xconv_oracle as O
from paper_2106_06998_b200 import binding as xb
from paper_2106_06998_b200 import inputs
from tests._util import check, host

pytestmark = pytest.mark.gpu
TOL = 1e-6


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


def _n(shape, seed, scale=1.0):
    return inputs.draw("normal", shape, seed, "f32", scale)


@pytest.mark.parametrize("B,Cin,Cout,D,H,W,K,KD", [
    (70, 3, 68, 1, 29, 31, 3, 1),        # padded copy of the input, two column tiles, the second of four channels (input gradient: multiply-adds)
    (70, 68, 13, 1, 29, 31, 3, 1),       # ... of the input gradient (forward: multiply-adds, 13 channels out)
    (9, 40, 20, 1, 37, 26, 5, 1),        # a last block of 8 channels; 25 offsets
    (33, 132, 36, 1, 28, 28, 1, 1),      # pointwise: chains over several blocks
    (3, 20, 100, 7, 19, 23, 3, 3),       # planes outside the volume
    (5, 16, 64, 6, 33, 20, 3, 1),        # a planar kernel on the planes of a volume; blocks of 16 channels
    (2, 48, 48, 1, 5, 300, 3, 1),        # rows wider than a patch
])
def test_convolution(B, Cin, Cout, D, H, W, K, KD):
    geo, kgeo = ((D, H, W), (KD, K, K)) if D > 1 else ((H, W), (K, K))
    X, dY = _n((B, Cin) + geo, 1), _n((B, Cout) + geo, 2)
    Wt = _n((Cout, Cin) + kgeo, 3, (2.0 / (K * K * KD * Cin)) ** 0.5)
    desc = xb.make_desc(B, Cin, Cout, H, W, 1, torch.float32, K, D=D, KD=KD)
    split = {op: xb.engine_for(desc, op) == "tcgen05_f32" for op in (xb.OP_FORWARD, xb.OP_DGRAD)}
    assert split == {xb.OP_FORWARD: Cout % 4 == 0, xb.OP_DGRAD: Cin % 4 == 0}
    d = {k: xb.to_device(v, "f32") for k, v in dict(X=X, dY=dY, W=Wt, Z=np.ones((1, Cin) + geo, np.float32)).items()}
    Y, _ = xb.xconv_forward(d["X"], d["W"], d["Z"])
    dX = xb.xconv_dgrad(d["dY"], d["W"])
    Yo, dXo = (O.conv_forward3d(X, Wt), O.dx_exact3d(dY, Wt)) if D > 1 else (O.conv_forward(X, Wt), O.dx_exact(dY, Wt))
    check("Y", host(Y), Yo, TOL if split[xb.OP_FORWARD] else 1e-5)
    check("dX", host(dX), dXo, TOL if split[xb.OP_DGRAD] else 1e-5)
    # scratch for the header only: the multiply-adds take the call
    small, dX2 = torch.empty(256, dtype=torch.uint8, device="cuda"), torch.empty_like(dX)
    xb.dgrad_into(desc, d["dY"], d["W"], dX2, small)
    check("dX without scratch", host(dX2), dXo, 1e-5)


@pytest.mark.parametrize("r,Cin,Cout,D,H,W,K,KD", [
    (40, 64, 64, 1, 31, 33, 3, 1),       # L moved by rows
    (50, 33, 130, 1, 14, 30, 3, 1),      # one dy per unit, padded copies, channels behind whole tiles
    (300, 3, 64, 1, 7, 7, 3, 1),         # images narrower than a k-step
    (20, 24, 48, 1, 40, 29, 5, 1),       # pixel shifts in two units, two row tiles
    (120, 72, 40, 1, 40, 40, 1, 1),      # pointwise, two blocks of columns
    (120, 40, 200, 1, 40, 41, 1, 1),     # ... and two row tiles
    (6, 20, 36, 9, 12, 17, 3, 3),
])
def test_contraction(r, Cin, Cout, D, H, W, K, KD):
    geo = (D, H, W) if D > 1 else (H, W)
    L, Z = _n((r, Cout) + geo, 4), _n((r, Cin) + geo, 5)
    desc = xb.make_desc(1, Cin, Cout, H, W, r, torch.float32, K, D=D, KD=KD)
    assert xb.engine_for(desc, xb.OP_CONTRACT) == "tcgen05_f32"
    scale = torch.rand(Cin, device="cuda") + 0.5
    dW = xb.xconv_contract(xb.to_device(L, "f32"), xb.to_device(Z, "f32"), kernel_size=K, kernel_depth=KD, chan_scale=scale)
    want = O.wgrad_contract3d(L, Z, (KD, K, K)) if D > 1 else O.wgrad_contract(L, Z, K, K)
    want = want * r * host(scale).reshape((1, -1) + (1,) * (want.ndim - 2))
    check("dW", host(dW), want, TOL)


@pytest.mark.parametrize("r,B,C,H,W", [
    (64, 128, 64, 32, 32), (130, 200, 24, 31, 28), (300, 7, 48, 40, 37), (5, 140, 36, 45, 33), (72, 65, 20, 33, 31), (300, 70, 40, 33, 17),
])
def test_sketch_and_backprobe(r, B, C, H, W):
    X, Z, S = _n((B, C, H, W), 6), _n((r, C, H, W), 7), _n((r, B), 8)
    desc = xb.make_desc(B, C, C, H, W, r, torch.float32)
    assert xb.engine_for(desc, xb.OP_SKETCH) == "tcgen05_f32"
    assert xb.engine_for(desc, xb.OP_BACKPROBE) == ("simt_f32" if B == 7 else "tcgen05_f32")      # (7 terms: multiply-adds)
    check("S", host(xb.xconv_sketch(xb.to_device(X, "f32"), xb.to_device(Z, "f32"))), O.sketch(X, Z), TOL)
    L = host(xb.xconv_backprobe(torch.from_numpy(S).cuda(), xb.to_device(X, "f32")))
    check("L", L, np.tensordot(S.astype(np.float64), X.astype(np.float64), 1), TOL)


@pytest.mark.parametrize("dt,u", [("bf16", 2.0 ** -8), ("f16", 2.0 ** -11)])
@pytest.mark.parametrize("r,B,C,H,W", [
    (70, 131, 24, 31, 28),       # two column tiles of 48, a last block of 3 terms, 96 positions in the last tile
    (300, 45, 40, 33, 17),       # 8 positions in the last tile, 60 columns in the last column tile
    (129, 97, 64, 8, 8),         # one term in the last block, fewer tiles than SMs
])
def test_backprobe_of_16_bit_rows(dt, u, r, B, C, H, W):
    """S in three parts, the rows whole.  Bound: the rounding of the result, u of it, and TOL of its norm for the sums; float16 rows of S
    scaled by 2^-30 and 2^20 keep their precision, and values that are not finite reach what the definition says, and nothing else."""
    t = xb.to_device(inputs.draw("normal", (B, C, H, W), 21, dt, 1.0), dt)
    if dt == "f16":
        t = t * 2.0 ** -10
    Y, S = host(t), _n((r, B), 22)
    S[3] *= 2.0 ** -30
    S[5] *= 2.0 ** 20
    desc = xb.make_desc(B, C, C, H, W, r, t.dtype)
    assert xb.engine_for(desc, xb.OP_BACKPROBE) == "tcgen05_" + dt
    want = np.tensordot(S.astype(np.float64), Y, 1)
    L = host(xb.xconv_backprobe(torch.from_numpy(S).cuda(), t)).astype(np.float64)
    tiny = 2.0 ** -25 if dt == "f16" else 0.0                 # half the spacing of float16's subnormal numbers
    norm = np.sqrt(np.square(want).mean(axis=(1, 2, 3), keepdims=True))
    assert (np.abs(L - want) <= u * np.abs(want) * (1 + TOL) + 4 * TOL * norm + tiny).all()
    S[r - 1, B - 1] = np.inf
    t[2, 5, 1, 2] = float("nan")
    L2 = host(xb.xconv_backprobe(torch.from_numpy(S).cuda(), t)).astype(np.float64)
    assert np.isnan(L2[:, 5, 1, 2]).all()
    got, exact = L2[r - 1], np.where(Y[B - 1] > 0, np.inf, np.where(Y[B - 1] < 0, -np.inf, np.nan))
    got[5, 1, 2] = exact[5, 1, 2] = 0.0
    assert np.array_equal(got, exact, equal_nan=True)
    L[:, 5, 1, 2] = L2[:, 5, 1, 2] = 0.0
    assert np.array_equal(L2[:r - 1], L[:r - 1])


@pytest.mark.parametrize("dt,tol", [("f32", TOL), ("bf16", 1e-2), ("f16", 2e-3)])
@pytest.mark.parametrize("r,B,Cin,Cout,H,W", [(131, 70, 24, 16, 31, 28), (97, 75, 40, 24, 33, 17)])
def test_estimate_summed_over_the_probes_first(dt, tol, r, B, Cin, Cout, H, W):
    """More probes than samples: the rebuilt activation is the back-probe kernel's, S read by its columns."""
    X, Z, dY = (inputs.draw("normal", s, 30 + i, dt, 1.0 if i else 0.05) for i, s in enumerate(((B, Cin, H, W), (r, Cin, H, W), (B, Cout, H, W))))
    d = {k: xb.to_device(v, dt) for k, v in dict(X=X, Z=Z, dY=dY).items()}
    swapped = xb.make_desc(r, Cin, Cin, H, W, B, d["X"].dtype)                # what the first step is, as a layer
    assert xb.engine_for(swapped, xb.OP_BACKPROBE) == "tcgen05_" + dt
    S = xb.xconv_sketch(d["X"], d["Z"])
    dW = host(xb.xconv_wgrad(S, d["dY"], d["Z"]))
    check("dW", dW, O.wgrad_estimate(host(S), host(d["dY"]), host(d["Z"])), 4 * tol if dt == "f32" else tol)


def test_values_that_cannot_be_split():
    """Infinities, NaN and the largest floats: every result they enter is what the definition gives, the others keep their bits."""
    r, B, Cin, Cout, H, W = 70, 64, 20, 36, 24, 30
    X, Z, Wt = _n((B, Cin, H, W), 9), _n((r, Cin, H, W), 10), _n((Cout, Cin, 3, 3), 11, 0.1)
    desc = xb.make_desc(B, Cin, Cout, H, W, r, torch.float32)
    assert all(xb.engine_for(desc, op) == "tcgen05_f32" for op in (xb.OP_FORWARD, xb.OP_SKETCH, xb.OP_CONTRACT))
    dev = lambda a: xb.to_device(a, "f32")
    Y, S = map(host, xb.xconv_forward(dev(X), dev(Wt), dev(Z)))
    L, dW = _n((r, Cout, H, W), 12), None
    dW = host(xb.xconv_contract(dev(L), dev(Z)))
    for bad in (np.inf, -np.inf, np.nan, np.float32(3.4e38)):
        X2 = X.copy()
        X2[3, 5, 10, 29] = bad
        Y2, S2 = map(host, xb.xconv_forward(dev(X2), dev(Wt), dev(Z)))
        hit = np.zeros((B, H, W), bool)
        hit[3, 9:12, 28:] = True
        hit = np.broadcast_to(hit[:, None], Y.shape)
        assert np.array_equal(Y2[~hit], Y[~hit])
        with np.errstate(all="ignore"):
            want = O.conv_forward(X2[3:4], Wt)[0] if np.isfinite(bad) else float(bad) * np.ones_like(Y[3])
        got = Y2[3][:, 9:12, 28:]
        if np.isfinite(bad):
            check("Y at the value", got, want[:, 9:12, 28:], 1e-5)
        elif np.isnan(bad):
            assert np.isnan(got).all()
        else:
            for dy in range(3):
                for dx in range(2):
                    sign = np.sign(Wt[:, 5, 2 - dy, (29 - (28 + dx)) + 1])
                    assert np.array_equal(got[:, dy, dx], sign * bad)
        others = np.arange(B) != 3
        assert np.array_equal(S2[:, others], S[:, others])
        if np.isinf(bad):
            assert np.array_equal(S2[:, 3], np.sign(Z[:, 5, 10, 29]) * bad)
        else:
            assert np.isnan(bad) == np.isnan(S2[:, 3]).all()
        Z2 = Z.copy()
        Z2[7, 4, 0, 0] = bad
        dW2 = host(xb.xconv_contract(dev(L), dev(Z2)))
        others = np.arange(Cin) != 4
        assert np.array_equal(dW2[:, others], dW[:, others])
        if np.isinf(bad):
            assert np.array_equal(dW2[:, 4, 1, 1], np.sign(L[7, :, 0, 0]) * bad)
            assert np.isfinite(dW2[:, 4, 2, 2]).all()          # that offset pairs the corner with a position outside
