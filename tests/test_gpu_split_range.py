"""The ends of the range that the kernels on split operands keep: small floats, and rows of S with small and large entries."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from oracle import xconv_oracle as O
from paper_2106_06998_b200 import binding as xb
from paper_2106_06998_b200 import inputs
from tests._util import check, host

pytestmark = pytest.mark.gpu
# Parts of floats are exact down to the smallest normal number; the sums as in the tests of ordinary values.
TOL = 1e-6
SMALL = 2.0 ** -120                     # 6 bits above the smallest normal number; a bfloat16 part of an unscaled remainder ends at 2^-133


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


def _n(shape, seed, scale=1.0):
    return inputs.draw("normal", shape, seed, "f32", 1.0) * np.float32(scale)


@pytest.mark.parametrize("which", [0, 1])
def test_small_floats(which):
    """One operand of every sum of the size of SMALL: the results have the precision that they have of operands of the size of 1."""
    a, b = (SMALL, 1.0) if which == 0 else (1.0, SMALL)
    B, Cin, Cout, H, W, r = 64, 20, 36, 24, 30, 70
    desc = xb.make_desc(B, Cin, Cout, H, W, r, torch.float32)
    for op in (xb.OP_FORWARD, xb.OP_DGRAD, xb.OP_SKETCH, xb.OP_BACKPROBE, xb.OP_CONTRACT):
        assert xb.engine_for(desc, op) == "tcgen05_f32"
    dev = lambda t: xb.to_device(t, "f32")
    X, dY, Wt, Z = _n((B, Cin, H, W), 1, a), _n((B, Cout, H, W), 2, a), _n((Cout, Cin, 3, 3), 3, b), _n((r, Cin, H, W), 4, b)
    L, S = _n((r, Cout, H, W), 5, a), _n((r, B), 6, b)
    Y, Sk = map(host, xb.xconv_forward(dev(X), dev(Wt), dev(Z)))
    up = 1.0 / SMALL                                          # (the bounds' squares would run under)
    check("Y", Y * up, O.conv_forward(X, Wt) * up, TOL)
    check("S", Sk * up, O.sketch(X, Z) * up, TOL)
    check("dX", host(xb.xconv_dgrad(dev(dY), dev(Wt))) * up, O.dx_exact(dY, Wt) * up, TOL)
    check("L", host(xb.xconv_backprobe(torch.from_numpy(S).cuda(), dev(dY))) * up, np.tensordot(S.astype(np.float64), dY.astype(np.float64), 1) * up, TOL)
    check("dW", host(xb.xconv_contract(dev(L), dev(Z))) * up, O.wgrad_contract(L, Z, 3, 3) * up, TOL)


@pytest.mark.parametrize("dt,u,tiny", [("bf16", 2.0 ** -8, 0.0), ("f16", 2.0 ** -11, 2.0 ** -25)])
@pytest.mark.parametrize("r,B,C,H,W", [(70, 131, 24, 31, 28), (300, 45, 40, 33, 17)])
def test_rows_of_the_sketch_with_a_wide_range(dt, u, tiny, r, B, C, H, W):
    """Large entries of S meet a sample of zeros, so that the small ones decide.  Bound: the rounding of the result (u of it, half the spacing
    of float16's subnormal numbers), and TOL of the sum of the terms' magnitudes."""
    Y, S = inputs.draw("normal", (B, C, H, W), 7, dt, 2.0 ** -6), _n((r, B), 8)
    Y[7] = 0.0
    S[4] *= np.float32(2.0 ** -10); S[4, 7] = 2.0 ** 20                     # 2^30 within the row: parts
    S[6, 7] = 2.0 ** 34
    S[9] *= (2.0 ** -np.linspace(0, 60, B)).astype(np.float32)              # every size down to 2^-60 of the largest: multiply-adds
    S[r - 1, 7] = 2.0 ** 50
    S[33, 7] = -2.0 ** 90
    desc = xb.make_desc(B, C, C, H, W, r, torch.bfloat16 if dt == "bf16" else torch.float16)
    assert xb.engine_for(desc, xb.OP_BACKPROBE) == "tcgen05_" + dt
    Yd = xb.to_device(Y, dt)
    exact = host(Yd)
    L = host(xb.xconv_backprobe(torch.from_numpy(S).cuda(), Yd))
    S64 = S.astype(np.float64)
    want, size = np.tensordot(S64, exact, 1), np.tensordot(np.abs(S64), np.abs(exact), 1)
    over = np.abs(L - want) > u * np.abs(want) * (1 + TOL) + TOL * size + tiny
    assert not over.any(), np.unique(np.argwhere(over)[:, 0])
