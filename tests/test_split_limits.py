"""Layers beyond what the float tensor-core kernels count in 32 bits stay on the multiply-adds, which count in 64 (host arithmetic only)."""
import pytest
import torch

from paper_2106_06998_b200 import binding as xb


@pytest.mark.parametrize("K,C", [(1, 131072), (3, 38400), (5, 20000)])
def test_contraction_with_too_many_entries(K, C):
    """2^32 groups of four entries: 16 C^2 / 128 x 64 (K = 1), 3 C^2 (K = 3), 12 C^2 (K = 5)."""
    small = xb.make_desc(1, C // 16, C // 16, 64, 64, 2, torch.float32, K)
    assert xb.engine_for(small, xb.OP_CONTRACT) == "tcgen05_f32"
    assert xb.engine_for(xb.make_desc(1, C, C, 64, 64, 2, torch.float32, K), xb.OP_CONTRACT) == "simt_f32"


@pytest.mark.parametrize("K,C", [(1, 98304), (5, 19200)])
def test_convolution_with_too_many_weights(K, C):
    small = xb.make_desc(1, C // 16, C // 16, 64, 64, 2, torch.float32, K)
    for op in (xb.OP_FORWARD, xb.OP_DGRAD):
        assert xb.engine_for(small, op) == "tcgen05_f32"
        assert xb.engine_for(xb.make_desc(1, C, C, 64, 64, 2, torch.float32, K), op) == "simt_f32"
