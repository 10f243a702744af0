"""Calls from several host threads and on several streams at once: the same bits as one call after the other."""
import threading

import pytest
import torch

import __graft_entry__ as entry
from paper_2106_06998_b200 import binding as xb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


def _layer(seed, B, Cin, Cout, geo, r, dtype, K=3):
    g = torch.Generator(device="cuda").manual_seed(seed)
    fmt = torch.channels_last if len(geo) == 2 else torch.channels_last_3d
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(dtype).contiguous(memory_format=fmt)
    return dict(X=rnd(B, Cin, *geo), dY=rnd(B, Cout, *geo), Z=rnd(r, Cin, *geo), W=rnd(Cout, Cin, *([K] * len(geo))),
                K=K, KD=K if len(geo) == 3 else 1)


def _step(d):
    Y, S = xb.xconv_forward(d["X"], d["W"], d["Z"])
    dW = xb.xconv_wgrad(S, d["dY"], d["Z"], kernel_size=d["K"], kernel_depth=d["KD"])
    return Y, S, dW, xb.xconv_dgrad(d["dY"], d["W"])


def _run_threads(jobs):
    errors = []

    def guarded(job):
        try:
            job()
        except Exception as e:          # an assertion of a thread is the test's
            errors.append(e)

    threads = [threading.Thread(target=guarded, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]


@pytest.mark.parametrize("one,two", [
    # both layers of a pair run the same kernel with another amount of shared memory: 53 and 89 KB, 35 and 60 KB
    ((3, 8, 64, (4, 40, 34), 3), (17, 3, 64, (10, 13, 32), 3)),
    ((22, 3, 64, (29, 40), 5), (39, 16, 64, (29, 29), 5)),
])
def test_float_layers_of_different_geometry_from_two_host_threads(one, two):
    def job(shape, seed):
        B, Cin, Cout, geo, K = shape
        d = _layer(seed, B, Cin, Cout, geo, 1, torch.float32, K)
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            ws = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")
            D = geo[0] if len(geo) == 3 else 1
            desc = xb.make_desc(B, Cin, Cout, geo[-2], geo[-1], 1, torch.float32, K, D=D, KD=d["KD"])
            Y = torch.empty_like(d["dY"])
            S = torch.empty((1, B), device="cuda")
            for i in range(1500):
                xb.forward_into(desc, d["X"], d["W"], d["Z"], Y, S, ws)
                if i % 100 == 0:
                    s.synchronize()
            s.synchronize()

    torch.cuda.synchronize()
    _run_threads([lambda: job(one, 1), lambda: job(two, 2)])


@pytest.mark.parametrize("threads", [False, True])
def test_layers_on_two_streams_at_once(threads):
    """Layers whose channels are padded in the scratch memory, and one that keeps much in it, each on a stream of its own; the
    streams of one thread, and of a thread each."""
    layers = [_layer(1, 64, 3, 64, (56, 56), 32, torch.bfloat16), _layer(2, 64, 5, 32, (60, 52), 80, torch.float16),
              _layer(3, 16, 32, 32, (64, 64), 64, torch.bfloat16)]
    want = []
    for d in layers:
        want.append([t.clone() for t in _step(d)])
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in layers]
    got = [[] for _ in layers]

    def one(i, times):
        with torch.cuda.stream(streams[i]):
            for _ in range(times):
                got[i].append(_step(layers[i]))

    if threads:
        _run_threads([lambda i=i: one(i, 30) for i in range(len(layers))])
    else:
        for _ in range(30):
            for i in range(len(layers)):
                one(i, 1)
    torch.cuda.synchronize()
    for w, g in zip(want, got):
        assert len(g) == 30
        for out in g:
            assert all(torch.equal(a, b) for a, b in zip(w, out))


def test_a_captured_step_has_scratch_memory_of_its_own():
    """The public calls captured on a stream that has run them before: eager calls on that stream between the replays, of a layer
    that needs more scratch, touch nothing that the graph uses."""
    d, other = _layer(4, 8, 3, 48, (20, 24), 4, torch.float16), _layer(5, 32, 5, 64, (56, 56), 48, torch.float16)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        want = [t.clone() for t in _step(d)]
        graph = torch.cuda.CUDAGraph()
        side.synchronize()
        with torch.cuda.graph(graph, stream=side):
            out = _step(d)
        for _ in range(3):
            for t in out:
                t.zero_()
            _step(other)
            graph.replay()
            _step(other)
            side.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(want, out))
