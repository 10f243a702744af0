"""The offset contraction for few channels at the edges of its tiles: patches that overhang the image, channel counts that are
not whole blocks or not multiples of 8 (padded copies), every way the offsets are spread over the two sides of the MMA.
Fed with an L already rounded to storage: the bar is the one of the contraction alone in test_gpu_parity.py (products of
16-bit values are exact in float, the sums are float)."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from oracle import xconv_oracle as O
from paper_2106_06998_b200 import binding as xb
from paper_2106_06998_b200 import inputs
from tests._util import check, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("dtype,r,Cin,Cout,D,H,W,K,KD", [
    ("bf16", 3, 3, 5, 1, 4, 4, 3, 1),          # one patch mostly outside the image; both channel counts padded
    ("f16", 2, 1, 64, 1, 17, 35, 3, 1),        # one input channel; two row tiles, the second half empty
    ("bf16", 5, 32, 32, 1, 33, 130, 3, 1),     # one MMA for nine offsets
    ("f16", 3, 16, 32, 1, 12, 19, 5, 1),       # 25 offsets, the fifth row shift in a row tile of its own
    ("f16", 2, 48, 24, 1, 9, 30, 5, 1),        # 320 columns: two pieces, one dy per unit, the single L block read four times
    ("bf16", 2, 128, 128, 1, 10, 28, 3, 1),    # one dy per unit, two channel blocks on each side
    ("f16", 4, 96, 120, 1, 7, 16, 3, 1),       # last channel blocks partly padding
    ("bf16", 2, 16, 24, 1, 11, 21, 1, 1),      # pointwise with the rows of one shift
    ("bf16", 2, 32, 16, 5, 6, 20, 3, 3),       # 27 offsets in one unit
    ("f16", 2, 64, 64, 3, 8, 18, 3, 3),        # one dz per unit
    ("bf16", 3, 24, 48, 4, 9, 9, 3, 1),        # planar kernel on the planes of a volume
])
def test_contraction(dtype, r, Cin, Cout, D, H, W, K, KD):
    g = np.random.Generator(np.random.PCG64([r, Cin, Cout, H, W, K]))
    geo = (D, H, W) if D > 1 else (H, W)
    L, Z = (inputs.round_to_storage(g.standard_normal((r, c) + geo).astype(np.float32), dtype) for c in (Cout, Cin))
    Ld, Zd = xb.to_device(L, dtype), xb.to_device(Z, dtype)
    desc = xb.make_desc(8, Cin, Cout, H, W, r, Zd.dtype, K, D=D, KD=KD)
    assert xb.engine_for(desc, xb.OP_CONTRACT) == "tcgen05_" + dtype
    want = (O.wgrad_contract3d(L, Z, (KD, K, K)) if D > 1 else O.wgrad_contract(L, Z, K, K))
    dW = xb.xconv_contract(Ld, Zd, kernel_size=K, kernel_depth=KD)
    again = xb.xconv_contract(Ld, Zd, kernel_size=K, kernel_depth=KD)
    torch.cuda.synchronize()
    check("dW", host(dW), want, 1e-4)
    assert torch.equal(dW, again)
    # nothing is written behind dW, and the scale per input channel is applied to the channels it belongs to
    scale = torch.from_numpy(g.uniform(0.5, 2.0, Cin).astype(np.float32)).cuda()
    buf = torch.full((dW.numel() + 64,), 7.0, device="cuda")
    ws = xb.workspace(xb.workspace_bytes(desc, xb.OP_CONTRACT), "cuda")
    desc.chan_scale = scale.data_ptr()
    status = xb.lib().xconv_contract(xb.ctypes.byref(desc), Ld.data_ptr(), Zd.data_ptr(), buf.data_ptr(), ws.data_ptr(), ws.numel(),
                                     torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert status == 0 and bool((buf[dW.numel():] == 7.0).all())
    taps = KD * K * K
    got = host(buf[:dW.numel()].reshape(Cout, taps, Cin))
    flat = want.reshape(Cout, Cin, taps).transpose(0, 2, 1) * r
    check("dW with chan_scale", got, flat * host(scale), 1e-4)


@pytest.mark.parametrize("dtype,r,Cin,Cout,D,H,W,K,KD", [
    ("bf16", 24, 16, 24, 1, 200, 210, 3, 1),   # long sums, one row tile; some rows of a patch per accumulator set
    ("f16", 8, 3, 48, 1, 190, 200, 3, 1),      # two row tiles in one unit; padded input channels
    ("bf16", 16, 48, 48, 1, 100, 100, 3, 1),   # the two row tiles as units
    ("f16", 5, 16, 48, 1, 30, 45, 5, 1),       # three row tiles as units
    ("bf16", 6, 48, 24, 1, 60, 77, 5, 1),      # pixel shifts in two units, the second with fewer
    ("f16", 3, 24, 24, 12, 40, 44, 3, 3),      # one dz per unit
    ("bf16", 60, 8, 16, 1, 5, 4, 3, 1),        # several patches per accumulator set, the last set with fewer
    ("f16", 7, 200, 104, 1, 33, 40, 1, 1),     # pointwise, four channel blocks of columns
    ("bf16", 2, 24, 104, 1, 33, 40, 1, 1),     # one 32-column chunk for two warps a quadrant
])
def test_drained_contraction_adds_up_like_float(dtype, r, Cin, Cout, D, H, W, K, KD):
    """Channels off the multiples of 32.  An accumulator of the tensor cores holds 16 k-steps and loses less than a unit in its
    last place, 2^-23, in each; the rest of the sum is float: 16 * 2^-23."""
    g = np.random.Generator(np.random.PCG64([r, Cin, Cout, H, W, K, 3]))
    geo = (D, H, W) if D > 1 else (H, W)
    L, Z = (inputs.round_to_storage(g.standard_normal((r, c) + geo).astype(np.float32), dtype) for c in (Cout, Cin))
    Ld, Zd = xb.to_device(L, dtype), xb.to_device(Z, dtype)
    desc = xb.make_desc(8, Cin, Cout, H, W, r, Zd.dtype, K, D=D, KD=KD)
    assert (Cin % 32 or Cout % 32) and xb.engine_for(desc, xb.OP_CONTRACT) == "tcgen05_" + dtype
    dW, again = (xb.xconv_contract(Ld, Zd, kernel_size=K, kernel_depth=KD) for _ in range(2))
    torch.cuda.synchronize()
    want = O.wgrad_contract3d(L, Z, (KD, K, K)) if D > 1 else O.wgrad_contract(L, Z, K, K)
    assert O.rel_fro(host(dW), want) < 16 * 2.0 ** -23
    assert torch.equal(dW, again)


def test_calls_in_a_row_on_layers_that_fill_tensor_memory():
    """Several CTAs of these layers fit one SM beside each other and each takes all of its tensor memory (25 offsets, 320
    columns), so a call's kernel starts while its columns are still held by the call before it.  The allocations have to be
    served in the order of the stream; a hundred calls on each of two streams, interleaved with convolutions."""
    g = np.random.Generator(np.random.PCG64(11))
    B, C, H, W, r = 40, 32, 4, 16, 40
    L, Z, X = (inputs.round_to_storage(g.standard_normal((n, C, H, W)).astype(np.float32), "bf16") for n in (r, r, B))
    Wt = inputs.round_to_storage((0.05 * g.standard_normal((C, C, 5, 5))).astype(np.float32), "bf16")
    Ld, Zd, Xd, Wd = (xb.to_device(v, "bf16") for v in (L, Z, X, Wt))
    desc = xb.make_desc(B, C, C, H, W, r, Zd.dtype, 5)
    streams = [torch.cuda.Stream() for _ in range(2)]
    like = dict(device="cuda", memory_format=torch.channels_last)
    out = [(torch.empty((C, C, 5, 5), dtype=torch.float32, **like), torch.empty((B, C, H, W), dtype=torch.bfloat16, **like),
            torch.empty(xb.workspace_bytes(desc, xb.OP_CONTRACT), dtype=torch.uint8, device="cuda")) for _ in streams]
    torch.cuda.synchronize()
    for _ in range(100):
        for s, (dW, dX, ws) in zip(streams, out):
            with torch.cuda.stream(s):
                xb.contract_into(desc, Ld, Zd, dW, ws)
                xb.dgrad_into(desc, Xd, Wd, dX, ws)
    torch.cuda.synchronize()
    for dW, dX, ws in out:
        check("dW", host(dW), O.wgrad_contract(L, Z, 5, 5), 1e-4)
        check("dX", host(dX), O.dx_exact(X, Wt), 1e-2)
        assert xb.workspace_status(ws) == 0
