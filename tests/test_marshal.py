"""The binding's native calls (csrc/marshal.cpp) leave everything but ordinary CUDA tensors to the Python path, which raises the errors.  (No GPU.)"""
import pytest
import torch

from paper_2106_06998_b200 import binding as xb


@pytest.fixture(scope="module")
def native():
    return xb._load_native()


def test_what_is_not_an_ordinary_cuda_tensor_is_left_to_the_python_path(native):
    x = torch.zeros(2, 8, 4, 4).contiguous(memory_format=torch.channels_last)
    w = torch.zeros(8, 8, 3, 3).contiguous(memory_format=torch.channels_last)
    s = torch.zeros(3, 2)
    for args in ((x, w, x, False), (x.numpy(), w, x, False), (None, None, None, False), (x.to("meta"), w.to("meta"), x.to("meta"), False), (x, w, x), ()):
        assert native.forward(*args) is None
    assert native.sketch(x, x) is None and native.sketch_seeded(x, 1, 4) is None and native.dgrad(x, w, False) is None
    assert native.wgrad(s, x, x, 3, 1, False) is None and native.wgrad_seeded(s, x, 1, 8, 3, 1, False) is None
    assert native.backprobe(s, x) is None and native.contract(x, x, 3, 1, False) is None


def test_the_python_path_raises_as_before(native):
    x = torch.zeros(2, 8, 4, 4).contiguous(memory_format=torch.channels_last)
    w = torch.zeros(8, 8, 3, 3).contiguous(memory_format=torch.channels_last)
    for call in (lambda: xb.xconv_forward(x, w, x), lambda: xb.xconv_sketch(x, x), lambda: xb.xconv_sketch_seeded(x, 1, 4), lambda: xb.xconv_dgrad(x, w),
                 lambda: xb.xconv_wgrad(torch.zeros(2, 2), x, x), lambda: xb.xconv_wgrad_seeded(torch.zeros(2, 2), x, 1, 8),
                 lambda: xb.xconv_backprobe(torch.zeros(2, 2), x), lambda: xb.xconv_contract(x, x)):
        with pytest.raises(ValueError, match="must be a CUDA tensor"):
            call()
    with pytest.raises(TypeError):
        native.use_library(1, 2)
