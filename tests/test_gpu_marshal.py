"""The binding's native calls (csrc/marshal.cpp) against its Python path on the same tensors: the same bits, shapes, strides and types for every form that the
native calls take, the same errors for what is refused; scratch buffers that are bounded, of one thread and stream, and none kept from a capture."""
import threading
import time

import pytest
import torch

import __graft_entry__ as entry
from paper_2106_06998_b200 import binding as xb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


class _PythonPath:
    """Stands in for the native module and declines every call."""
    def __getattr__(self, name):
        return lambda *a: None


class _Counting:
    """The native module, counting the calls that it takes."""
    def __init__(self):
        self.module, self.taken = xb._load_native(), 0

    def __getattr__(self, name):
        def call(*a):
            out = getattr(self.module, name)(*a)
            self.taken += out is not None
            return out
        return call


def _layer(B, Cin, Cout, geo, r, dtype, K=3, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    fmt = torch.channels_last if len(geo) == 2 else torch.channels_last_3d
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(dtype).contiguous(memory_format=fmt)
    return dict(X=rnd(B, Cin, *geo), dY=rnd(B, Cout, *geo), Z=rnd(r, Cin, *geo), W=rnd(Cout, Cin, *([K] * len(geo))), S=torch.randn(r, B, generator=g, device="cuda"),
                L=rnd(r, Cout, *geo), K=K, KD=K if len(geo) == 3 else 1, Cin=Cin, r=r)


def _calls(d, circular=False):
    K, KD = d["K"], d["KD"]
    return [lambda: xb.xconv_forward(d["X"], d["W"], d["Z"], circular), lambda: xb.xconv_sketch(d["X"], d["Z"]), lambda: xb.xconv_sketch_seeded(d["X"], -5, d["r"]),
            lambda: xb.xconv_wgrad(d["S"], d["dY"], d["Z"], K, kernel_depth=KD, circular=circular),
            lambda: xb.xconv_wgrad_seeded(d["S"], d["dY"], 1 << 70, d["Cin"], K, KD, circular), lambda: xb.xconv_dgrad(d["dY"], d["W"], circular),
            lambda: xb.xconv_backprobe(d["S"], d["dY"]), lambda: xb.xconv_contract(d["L"], d["Z"], K, kernel_depth=KD, circular=circular)]


def _compare(calls, monkeypatch, taken):
    native = _Counting()
    monkeypatch.setattr(xb, "_native", native)
    got = [c() for c in calls]
    assert native.taken == taken
    monkeypatch.setattr(xb, "_native", _PythonPath())
    want = [c() for c in calls]
    for a, b in zip(got, want):
        for x, y in zip(a if isinstance(a, tuple) else (a,), b if isinstance(b, tuple) else (b,)):
            assert x.shape == y.shape and x.stride() == y.stride() and x.dtype == y.dtype and x.device == y.device and not x.requires_grad
            assert torch.equal(x, y)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("B,Cin,Cout,geo,r,K,circular", [
    (8, 16, 16, (32, 32), 8, 3, False), (3, 1, 7, (5, 9), 4, 3, True), (1, 1, 1, (1, 1), 1, 1, False), (5, 24, 8, (4, 7, 6), 9, 3, False), (4, 8, 16, (12, 1), 6, 5, False),
])
def test_both_paths_give_the_same(dtype, B, Cin, Cout, geo, r, K, circular, monkeypatch):
    d = _layer(B, Cin, Cout, geo, r, dtype, K)
    _compare(_calls(d, circular), monkeypatch, 8)
    d["W"] = torch.nn.Parameter(d["W"])
    d["X"] = d["X"].detach().requires_grad_()
    _compare(_calls(d, circular), monkeypatch, 8)


def test_forms_of_a_tensor(monkeypatch):
    """Views that are dense in channels-last, one-pixel images whose strides are free, and forms that only the Python path takes."""
    d = _layer(6, 16, 24, (9, 11), 5, torch.bfloat16)
    d["X"], d["Z"] = torch.cat([d["X"], d["X"]])[6:], torch.cat([d["Z"], d["Z"]])[5:]
    _compare(_calls(d), monkeypatch, 8)
    one = _layer(6, 16, 24, (1, 1), 5, torch.float16, K=1)
    one["X"] = one["X"].contiguous()
    _compare(_calls(one), monkeypatch, 8)

    class Sub(torch.Tensor):
        pass
    sub = dict(d, X=d["X"].as_subclass(Sub), dY=d["dY"].as_subclass(Sub), S=d["S"].as_subclass(Sub), L=d["L"].as_subclass(Sub))
    _compare(_calls(sub), monkeypatch, 0)
    odd = [lambda: xb.xconv_wgrad(d["S"], d["dY"], d["Z"], chan_scale=torch.ones(16, device="cuda")), lambda: xb.xconv_forward(d["X"], d["W"], d["Z"], 0),
           lambda: xb.xconv_wgrad(d["S"], d["dY"], d["Z"], circular=1)]
    _compare(odd, monkeypatch, 0)
    with torch.device("cuda"):                     # a mode that sees the Python path's calls
        _compare(_calls(d), monkeypatch, 0)


def test_what_was_refused_is_refused_with_the_same_error(monkeypatch):
    d = _layer(4, 8, 16, (6, 7), 3, torch.bfloat16)
    nchw = dict(d, X=d["X"].contiguous(), dY=d["dY"].contiguous(), L=d["L"].contiguous())
    host = dict(d, X=d["X"].cpu(), dY=d["dY"].cpu(), L=d["L"].cpu())
    double = dict(d, X=d["X"].double(), dY=d["dY"].double(), L=d["L"].double())
    other = dict(d, Z=d["Z"][:, :, :5].contiguous(memory_format=torch.channels_last), S=d["S"].t())
    even = dict(d, W=d["W"][:, :, :2, :2].contiguous(memory_format=torch.channels_last), K=2)
    offset = dict(d, X=torch.empty(d["X"].numel() + 1, dtype=torch.bfloat16, device="cuda")[1:].view(4, 6, 7, 8).permute(0, 3, 1, 2))
    empty = dict(d, X=d["X"][:0], dY=d["dY"][:0], S=d["S"][:, :0].contiguous())
    for case in (nchw, host, double, other, even, offset, empty):
        for i in range(8):
            errors = []
            for native in (xb._load_native(), _PythonPath()):
                monkeypatch.setattr(xb, "_native", native)
                try:
                    _calls(case)[i]()
                    errors.append(None)
                except Exception as e:
                    errors.append((type(e), str(e)))
            assert errors[0] == errors[1]
    torch.cuda.synchronize()


def test_kernels_that_the_descriptor_cannot_state_are_refused_on_both_paths(monkeypatch):
    d = _layer(4, 8, 16, (6, 7), 3, torch.bfloat16)
    flat = [dict(d, W=torch.zeros(16, 8, *k, device="cuda", dtype=torch.bfloat16).contiguous(memory_format=torch.channels_last)) for k in ((1, 3), (5, 3))]
    for native in (xb._load_native(), _PythonPath()):
        monkeypatch.setattr(xb, "_native", native)
        for case, calls in [(c, (0, 5)) for c in flat] + [(dict(d, KD=3), (3, 4, 7))]:
            for i in calls:
                with pytest.raises(ValueError):
                    _calls(case)[i]()
    torch.cuda.synchronize()


def test_a_scale_whose_values_lie_apart():
    d = _layer(4, 8, 16, (6, 7), 3, torch.bfloat16)
    scale = torch.arange(1.0, 17.0, device="cuda")[::2]
    for call in (lambda c: xb.xconv_wgrad(d["S"], d["dY"], d["Z"], chan_scale=c), lambda c: xb.xconv_contract(d["L"], d["Z"], chan_scale=c)):
        assert torch.equal(call(scale), call(scale.contiguous()))
        assert torch.equal(call(torch.ones(1, device="cuda").expand(8)), call(torch.ones(8, device="cuda")))


def test_scratch_buffers_are_bounded_and_given_back():
    d = _layer(16, 32, 64, (40, 40), 32, torch.bfloat16)
    nbytes = xb.workspace_bytes(xb.make_desc(16, 32, 64, 40, 40, 32, torch.bfloat16), xb.OP_WGRAD)
    native = xb._load_native()
    streams = [torch.cuda.Stream() for _ in range(20)]
    seen = []

    def job():
        for s in streams:
            with torch.cuda.stream(s):
                native.wgrad(d["S"], d["dY"], d["Z"], 3, 1, False)
        torch.cuda.synchronize()
        seen.append(torch.cuda.memory_allocated())

    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    t = threading.Thread(target=job)
    t.start()
    t.join()
    assert before + 7 * nbytes < seen[0] < before + 9 * nbytes      # the eight streams used last
    until = time.monotonic() + 10                                   # given back with the thread, whose own end comes a little behind join's
    while torch.cuda.memory_allocated() >= before + nbytes and time.monotonic() < until:
        time.sleep(0.01)
    assert torch.cuda.memory_allocated() < before + nbytes


def test_both_paths_take_one_buffer():
    """A thread that mixes calls of both paths on a stream holds one scratch buffer, the larger one; a smaller call finds it, and it is not held beyond the pool."""
    small, large = _layer(8, 32, 64, (40, 40), 16, torch.bfloat16), _layer(16, 32, 64, (40, 40), 32, torch.bfloat16)
    sizes = [xb.workspace_bytes(xb.make_desc(len(d["X"]), 32, 64, 40, 40, d["r"], torch.bfloat16), xb.OP_WGRAD) for d in (small, large)]
    scale = torch.ones(32, device="cuda")
    held = []

    def job():
        with torch.cuda.stream(torch.cuda.Stream()):
            for d, kw in ((small, {}), (small, dict(chan_scale=scale)), (large, dict(chan_scale=scale)), (large, {}), (small, {})):
                xb.xconv_wgrad(d["S"], d["dY"], d["Z"], **kw)
                held.append(torch.cuda.memory_allocated() - before)
            torch.cuda.current_stream().synchronize()
            del xb._ws_cache.buffers
            held.append(torch.cuda.memory_allocated() - before)
            xb.xconv_wgrad(small["S"], small["dY"], small["Z"])
            torch.cuda.current_stream().synchronize()

    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    t = threading.Thread(target=job)
    t.start()
    t.join()
    slack = 2 << 20                                                 # the allocator hands out whole blocks of 2 MB above 10 MB, and leaves a rest below 1 MB with its block
    assert sizes[0] > 4 * slack and sizes[1] > sizes[0] + slack
    for got, want in zip(held, (sizes[0], sizes[0], sizes[1], sizes[1], sizes[1], 0)):
        assert want <= got <= want + slack


def test_threads_and_streams_share_no_scratch():
    layers = [_layer(16, 3, 32, (40, 44), 32, torch.bfloat16, seed=1), _layer(8, 16, 24, (30, 33), 40, torch.float16, seed=2), _layer(4, 8, 8, (64, 64), 9, torch.float32, seed=3)]
    want = [[t for c in _calls(d) for t in (lambda o: o if isinstance(o, tuple) else (o,))(c())] for d in layers]
    torch.cuda.synchronize()
    wrong = []

    def job(d, expected):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(20):
                got = [t for c in _calls(d) for t in (lambda o: o if isinstance(o, tuple) else (o,))(c())]
                torch.cuda.current_stream().synchronize()
                if not all(torch.equal(a, b) for a, b in zip(got, expected)):
                    wrong.append(d["Cin"])

    threads = [threading.Thread(target=job, args=a) for a in zip(layers, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


def test_a_capture_keeps_its_scratch_to_itself():
    d, other = _layer(8, 3, 48, (20, 24), 4, torch.float16), _layer(32, 5, 64, (56, 56), 48, torch.float16)
    side = torch.cuda.Stream()
    flat = lambda calls: [t for c in calls for t in (lambda o: o if isinstance(o, tuple) else (o,))(c())]
    with torch.cuda.stream(side):
        want = [t.clone() for t in flat(_calls(d))]
        graph = torch.cuda.CUDAGraph()
        side.synchronize()
        with torch.cuda.graph(graph, stream=side):
            out = flat(_calls(d))
        for _ in range(3):
            for t in out:
                t.zero_()
            flat(_calls(other))
            graph.replay()
            flat(_calls(other))
            side.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(want, out))
