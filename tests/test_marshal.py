"""The binding's native calls (csrc/marshal.cpp) leave everything but ordinary CUDA tensors to the Python path, which raises the errors.  (No GPU.)"""
import sys
import warnings

import pytest
import torch

import paper_2106_06998_b200 as package
from paper_2106_06998_b200 import binding as xb
from paper_2106_06998_b200 import build


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


class _OnDevice(torch.Tensor):
    """A host tensor that passes for one in device memory."""
    is_cuda = True


@pytest.fixture
def python_path(monkeypatch):
    """The Python path on host tensors, up to where it would call the library."""
    class Reached(Exception):
        pass

    def reached():
        raise Reached
    monkeypatch.setattr(xb, "_native", type("Declines", (), {"__getattr__": lambda self, name: lambda *a: None})())
    monkeypatch.setattr(xb, "_cl", lambda t, name: t)
    monkeypatch.setattr(xb, "lib", reached)
    return Reached


def test_a_kernel_that_the_descriptor_cannot_state_is_refused(python_path):
    """The descriptor has one kernel extent, and a planar layer's weights have no planes: with anything else the kernels would read or write past a tensor."""
    x, s = torch.zeros(2, 8, 6, 6), torch.zeros(3, 2).as_subclass(_OnDevice)
    z, l = torch.zeros(3, 8, 6, 6), torch.zeros(3, 8, 6, 6)
    for shape in ((1, 3), (5, 3), (3, 1)):
        w = torch.zeros(8, 8, *shape)
        for call in (lambda: xb.xconv_forward(x, w, z), lambda: xb.xconv_dgrad(x, w)):
            with pytest.raises(ValueError, match="mismatch"):
                call()
    v, vz = torch.zeros(2, 8, 4, 6, 6), torch.zeros(3, 8, 4, 6, 6)
    with pytest.raises(ValueError, match="mismatch"):
        xb.xconv_forward(v, torch.zeros(8, 8, 3, 1, 3), vz)
    for depth in (2, 3):
        for call in (lambda **k: xb.xconv_wgrad(s, x, z, **k), lambda **k: xb.xconv_wgrad_seeded(s, x, 1, 8, **k), lambda **k: xb.xconv_contract(l, z, **k),
                     lambda **k: xb.xconv_wgrad_independent(torch.zeros(3, 8, 2), x, z, **k)):
            with pytest.raises(ValueError, match="kernel_depth"):
                call(kernel_depth=depth)
    for ok in (lambda: xb.xconv_forward(x, torch.zeros(8, 8, 3, 3), z), lambda: xb.xconv_forward(v, torch.zeros(8, 8, 1, 3, 3), vz),
               lambda: xb.xconv_wgrad(s, v, vz, kernel_depth=3), lambda: xb.xconv_wgrad(s, v, vz), lambda: xb.xconv_contract(l, z)):
        with pytest.raises(python_path):
            ok()


def test_what_lies_in_host_memory_is_refused_beside_the_images_too(python_path):
    x, z, s = torch.zeros(2, 8, 6, 6), torch.zeros(3, 8, 6, 6), torch.zeros(3, 2)
    for call in (lambda: xb.xconv_wgrad(s, x, z), lambda: xb.xconv_wgrad_seeded(s, x, 1, 8), lambda: xb.xconv_backprobe(s, x),
                 lambda: xb.xconv_wgrad_independent(torch.zeros(3, 8, 2), x, z)):
        with pytest.raises(ValueError, match="sketch"):
            call()
    device = s.as_subclass(_OnDevice)
    for scale in (torch.ones(8), torch.ones(7).as_subclass(_OnDevice), torch.ones(8, dtype=torch.float16).as_subclass(_OnDevice)):
        for call in (lambda: xb.xconv_wgrad(device, x, z, chan_scale=scale), lambda: xb.xconv_contract(z, z, chan_scale=scale)):
            with pytest.raises(ValueError, match="chan_scale"):
                call()
    with pytest.raises(python_path):
        xb.xconv_wgrad(device, x, z, chan_scale=torch.ones(8).as_subclass(_OnDevice))


def test_without_the_native_module_every_call_takes_the_python_path(monkeypatch):
    """One warning, and the errors of the Python path; a library that is missing is still an error."""
    x = torch.zeros(2, 8, 4, 4).contiguous(memory_format=torch.channels_last)
    monkeypatch.setitem(sys.modules, package.__name__ + "._marshal", None)
    monkeypatch.delattr(package, "_marshal", raising=False)
    monkeypatch.setattr(xb, "_native", None)
    with pytest.warns(RuntimeWarning, match="_marshal.so cannot be loaded"), pytest.raises(ValueError, match="must be a CUDA tensor"):
        xb.xconv_sketch(x, x)
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        for call in (lambda: xb.xconv_forward(x, x, x), lambda: xb.xconv_dgrad(x, x), lambda: xb.xconv_sketch_seeded(x, 1, 4)):
            with pytest.raises(ValueError, match="must be a CUDA tensor"):
                call()
    monkeypatch.setattr(xb, "_native", None)
    monkeypatch.setattr(xb, "_lib", None)
    monkeypatch.setattr(xb, "LIB_PATH", "/nowhere/libxconv.so")
    with pytest.raises(RuntimeError, match="is missing"):
        xb.xconv_sketch(x, x)


def test_a_module_for_another_torch_is_neither_used_nor_kept(monkeypatch):
    build.build()
    x = torch.zeros(2, 8, 4, 4).contiguous(memory_format=torch.channels_last)
    assert build._marshal_current() and xb._load_native().key == build.marshal_key()
    monkeypatch.setattr(xb, "marshal_key", lambda: "another")
    monkeypatch.setattr(xb, "_native", None)
    with pytest.warns(RuntimeWarning, match="not compiled as another"), pytest.raises(ValueError, match="must be a CUDA tensor"):
        xb.xconv_sketch(x, x)
    monkeypatch.setattr(build, "marshal_key", lambda: "another")
    assert not build._marshal_current()


def test_the_library_is_built_where_the_native_module_cannot_be(monkeypatch):
    build.build()
    monkeypatch.setenv("CXX", "/nowhere/g++")
    monkeypatch.setattr(build, "_marshal_current", lambda: False)
    with pytest.warns(RuntimeWarning, match="was not built"):
        assert build.build() == build.LIB
