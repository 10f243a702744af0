"""Kernels that start under the one before them: where that one holds the SMs or splits them for its own shared memory they would run slower than behind
its end, so a call must not take longer than its parts, each measured alone (device times; the bounds lie between what both forms measured)."""
import pytest
import torch

import __graft_entry__ as entry
from paper_2106_06998_b200 import binding as xb
from tests._util import device_time

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


def _rnd(*s, seed=3):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(s, generator=g, device="cuda").contiguous(memory_format=torch.channels_last if len(s) == 4 else torch.channels_last_3d)


@pytest.mark.parametrize("B,Cin,Cout,geo,r,K", [(78, 16, 96, (4, 34), 6, 3), (45, 4, 100, (14, 140), 10, 3), (102, 16, 32, (4, 8, 4), 1, 3)])
def test_forward_takes_no_longer_than_convolution_and_sketch(B, Cin, Cout, geo, r, K):
    """Small float sketches behind a convolution on the tensor cores: 0.97 of the parts' sum, started under it 1.12 to 1.22."""
    X, Z, W = _rnd(B, Cin, *geo), _rnd(r, Cin, *geo), _rnd(Cout, Cin, *([K] * len(geo)))
    D = geo[0] if len(geo) == 3 else 1
    assert xb.engine_for(xb.make_desc(B, Cin, Cout, geo[-2], geo[-1], r, torch.float32, K, D=D, KD=K if D > 1 else 1), xb.OP_FORWARD) == "tcgen05_f32"
    Wt = W.movedim(0, 1).contiguous(memory_format=torch.channels_last if D == 1 else torch.channels_last_3d)
    whole = device_time(lambda: xb.xconv_forward(X, W, Z), calls=10)
    conv = device_time(lambda: xb.xconv_dgrad(X, Wt), calls=10)          # the same products, as the input gradient of the layer turned around
    sketch = device_time(lambda: xb.xconv_sketch(X, Z), calls=10)
    assert whole < 1.06 * (conv + sketch), (whole, conv, sketch)
