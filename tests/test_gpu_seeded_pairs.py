"""The estimator that redraws its signs in a stream: the bits of the estimator on the stored probing vectors.  Up to 16 rows a warp takes two groups of 64 columns
and a whole Philox block of each row: around the size from which it does (2368 groups), with a last group alone, planes whose blocks start
in the middle of a Philox block, and reductions off the 32 rows that are drawn together.  Above 16 rows there are no pairs: two and four row tiles.  Each case
says which form it takes, and the library is asked."""
import pytest
import torch

import __graft_entry__ as entry
from paper_2106_06998_b200 import binding as xb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("B,r,groups,form", [
    (1, 8, 2368, "alone"), (8, 31, 2369, "pairs"), (16, 33, 2370, "pairs"), (16, 64, 4737, "pairs"), (9, 65, 2371, "pairs"),
    (17, 33, 2370, "alone"), (24, 41, 2369, "alone"), (32, 35, 2371, "alone"),      # 17 to 32 rows: S as two values
    (33, 34, 2370, "alone"), (40, 41, 2369, "alone"),                              # 33 to 64
    (24, 40, 2369, "tiles"),                                                        # reductions of a multiple of 8 above 16 rows: another kernel
])
def test_redrawn_probes_give_the_bits_of_stored_ones(dtype, B, r, groups, form):
    H, W, Cin, Cout = 2, groups, 32, 8
    variants = xb.variants_for(xb.make_desc(B, Cin, Cout, H, W, r, dtype), xb.OP_WGRAD_SEEDED)
    assert ("stream" in variants, "sign_pairs" in variants) == dict(alone=(True, False), pairs=(True, True), tiles=(False, False))[form]
    g = torch.Generator(device="cuda").manual_seed(groups + r)
    dY = torch.randn(B, Cout, H, W, generator=g, device="cuda").to(dtype).contiguous(memory_format=torch.channels_last)
    S = torch.randn(r, B, generator=g, device="cuda")
    Z = xb.xconv_probes_from_seed(77, r, Cin, H, W, dtype)
    assert torch.equal(xb.xconv_wgrad_seeded(S, dY, 77, Cin), xb.xconv_wgrad(S, dY, Z))
