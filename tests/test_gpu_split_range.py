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
