"""The estimator that redraws its signs, where a warp takes two groups of 64 columns and a whole Philox block of each row: the bits of the
estimator on the stored probing vectors, around the size from which it does (2368 groups), with a last group alone, planes whose blocks start
in the middle of a Philox block, and reductions off the 32 rows that are drawn together."""
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
@pytest.mark.parametrize("B,r,groups", [(1, 8, 2368), (8, 31, 2369), (16, 33, 2370), (16, 64, 4737), (9, 65, 2371), (24, 40, 2369), (33, 34, 2370)])
def test_pairs_of_groups_give_the_bits_of_stored_probes(dtype, B, r, groups):
    H, W, Cin, Cout = 2, groups, 32, 8
    g = torch.Generator(device="cuda").manual_seed(groups + r)
    dY = torch.randn(B, Cout, H, W, generator=g, device="cuda").to(dtype).contiguous(memory_format=torch.channels_last)
    S = torch.randn(r, B, generator=g, device="cuda")
    Z = xb.xconv_probes_from_seed(77, r, Cin, H, W, dtype)
    assert torch.equal(xb.xconv_wgrad_seeded(S, dY, 77, Cin), xb.xconv_wgrad(S, dY, Z))
