"""Infinities, NaN and the largest numbers through the kernels on split operands: what the definition gives, in the results that the value
enters and in no others, at the speed of finite data."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from paper_2106_06998_b200 import binding as xb
from paper_2106_06998_b200 import inputs
from tests._util import device_time, host

pytestmark = pytest.mark.gpu
INF, NAN, BIG = np.inf, np.nan, float(np.float32(3.4e38))
TOP = float(np.finfo(np.float32).max)


@pytest.fixture(scope="module", autouse=True)
def _built():
    entry.build()
    torch.cuda.set_device(0)


def _n(shape, seed, scale=1.0, dt="f32"):
    return inputs.draw("normal", shape, seed, dt, scale)


def _dev(a, dt="f32"):
    return xb.to_device(a, dt)


def _same(got, want, tol, top=TOP):
    """`want` in 64 bits; its values beyond `top` are infinities (within 2 % of it, where a rounding decides, either)."""
    near = (np.abs(want) > 0.98 * top) & (np.abs(want) < 1.02 * top)
    with np.errstate(all="ignore"):
        want = np.where(np.abs(want) > top, np.sign(want) * INF, want)
    fin = np.isfinite(want)
    assert np.array_equal(got[~fin & ~near], want[~fin & ~near], equal_nan=True)
    if (fin & ~near).any():
        rms = max(float(np.sqrt(np.mean(np.square(want[fin & ~near] / top)))) * top, 1e-300)
        assert (np.abs(got[fin & ~near] - want[fin & ~near]) <= tol * rms).all()


def _sum(a, b):
    """Sum over the last axis of a * b in 64 bits, infinities and NaN as the definition has them."""
    with np.errstate(all="ignore"):
        return (np.asarray(a, np.float64) * np.asarray(b, np.float64)).sum(axis=-1)


SETS = [(INF,), (-INF,), (NAN,), (INF, -INF), (INF, INF), (BIG,), (-BIG, 0.0)]


@pytest.mark.parametrize("values", SETS)
def test_sketch(values):
    r, B, C, H, W = 72, 65, 20, 33, 31
    X, Z = _n((B, C, H, W), 1), _n((r, C, H, W), 2)
    assert xb.engine_for(xb.make_desc(B, C, C, H, W, r, torch.float32), xb.OP_SKETCH) == "tcgen05_f32"
    S = host(xb.xconv_sketch(_dev(X), _dev(Z)))
    for t, other, axis in ((X, Z, 1), (Z, X, 0)):
        bad = t.copy()
        for i, v in enumerate(values):
            bad[3, 5, 10 + i, 29] = v
        got = host(xb.xconv_sketch(_dev(bad), _dev(Z)) if axis else xb.xconv_sketch(_dev(X), _dev(bad)))
        hit = np.zeros_like(S, bool)
        hit[(slice(None), 3) if axis else 3] = True
        assert np.array_equal(got[~hit], S[~hit])
        _same(got[hit], _sum(other.reshape(len(other), -1), bad[3].reshape(-1)), 1e-5)


@pytest.mark.parametrize("values", SETS)
def test_backprobe(values):
    r, B, C, H, W = 64, 72, 20, 33, 31
    Y, S = _n((B, C, H, W), 3), _n((r, B), 4)
    assert xb.engine_for(xb.make_desc(B, C, C, H, W, r, torch.float32), xb.OP_BACKPROBE) == "tcgen05_f32"
    call = lambda s, y: host(xb.xconv_backprobe(torch.from_numpy(np.ascontiguousarray(s)).cuda(), _dev(y)))
    L = call(S, Y)
    Y2 = Y.copy()
    for i, v in enumerate(values):
        Y2[7 + i, 4, 32, 30] = v
    got, hit = call(S, Y2), np.zeros(L.shape, bool)
    hit[:, 4, 32, 30] = True
    assert np.array_equal(got[~hit], L[~hit])
    _same(got[hit], _sum(S, Y2[:, 4, 32, 30]), 1e-5)
    S2 = S.copy()
    S2[9, 11:11 + len(values)] = values
    S2[12, 3] = 2.0 ** -140                                   # (its first part would round to zero)
    Y2 = Y.copy()
    Y2[3, 1, 2, 3] = INF
    got, hit = call(S2, Y2), np.zeros(L.shape, bool)
    hit[9] = hit[12] = hit[:, 1, 2, 3] = True
    assert np.array_equal(got[~hit], L[~hit])
    _same(got[9], _sum(np.moveaxis(Y2, 0, -1), S2[9]), 1e-5)
    assert got[12, 1, 2, 3] == INF


@pytest.mark.parametrize("dt", ["bf16", "f16"])
@pytest.mark.parametrize("r,B,C,H,W", [(70, 131, 24, 31, 28), (300, 45, 40, 33, 17)])
@pytest.mark.parametrize("values", SETS[:5])
def test_backprobe_of_16_bit_rows(dt, r, B, C, H, W, values):
    Y, S = _n((B, C, H, W), 5, 2.0 ** -6, dt), _n((r, B), 6)
    S[2, 9] = S[5, 9] = 1.0                                   # its second and third parts are zero
    S[8, 9] = -2.0 ** -140 if dt == "bf16" else -2.0 ** -60   # (its first part would round to zero)
    assert xb.engine_for(xb.make_desc(B, C, C, H, W, r, torch.bfloat16 if dt == "bf16" else torch.float16), xb.OP_BACKPROBE) == "tcgen05_" + dt
    call = lambda s, y: host(xb.xconv_backprobe(torch.from_numpy(np.ascontiguousarray(s)).cuda(), _dev(y, dt)))
    L, exact = call(S, Y), host(_dev(Y, dt))
    Y2 = exact.copy()
    for i, v in enumerate(values):
        Y2[9 + i, 4, 30, 16] = v
    got, hit = call(S, Y2.astype(np.float32)), np.zeros(L.shape, bool)
    hit[:, 4, 30, 16] = True
    assert np.array_equal(got[~hit], L[~hit])
    assert np.array_equal(got[hit], _sum(S, Y2[:, 4, 30, 16]), equal_nan=True)
    S2 = S.copy()
    S2[9, 11:11 + len(values)] = values
    got, hit = call(S2, Y), np.zeros(L.shape, bool)
    hit[9] = True
    assert np.array_equal(got[~hit], L[~hit])
    assert np.array_equal(got[9], _sum(np.moveaxis(exact, 0, -1), S2[9]), equal_nan=True)


@pytest.mark.parametrize("B,Cin,Cout,D,H,W,K,KD", [(64, 20, 36, 1, 24, 30, 3, 1), (33, 132, 36, 1, 28, 28, 1, 1), (6, 24, 40, 7, 19, 23, 3, 3)])
@pytest.mark.parametrize("values", [(INF,), (-INF,), (NAN,), (INF, -INF), (BIG,)])
def test_convolution(B, Cin, Cout, D, H, W, K, KD, values):
    geo, kgeo = ((D, H, W), (KD, K, K)) if D > 1 else ((H, W), (K, K))
    X, dY, Wt = _n((B, Cin) + geo, 7), _n((B, Cout) + geo, 8), _n((Cout, Cin) + kgeo, 9, 0.1)
    Z = _dev(np.ones((1, Cin) + geo, np.float32))
    desc = xb.make_desc(B, Cin, Cout, H, W, 1, torch.float32, K, D=D, KD=KD)
    assert xb.engine_for(desc, xb.OP_FORWARD) == xb.engine_for(desc, xb.OP_DGRAD) == "tcgen05_f32"
    p = K // 2
    fwd = lambda x, w: host(xb.xconv_forward(_dev(x), _dev(w), Z)[0])
    bwd = lambda y, w: host(xb.xconv_dgrad(_dev(y), _dev(w)))
    for f, t, flip in ((fwd, X, False), (bwd, dY, True)):
        good = f(t, Wt)
        # a value at a corner: results around it see it through the weights of the matching offsets
        bad = t.copy()
        for i, v in enumerate(values):
            bad[(1, 3 + 2 * i) + (0,) * (len(geo) - 1) + (geo[-1] - 1,)] = v
        got = f(bad, Wt)
        hit = np.zeros(good.shape, bool)
        hit[(1, slice(None)) + tuple(slice(0, kg // 2 + 1) for kg in kgeo[:-1]) + (slice(geo[-1] - 1 - p, None),)] = True
        assert np.array_equal(got[~hit], good[~hit])
        # every result there by its definition: channels in summed for the one offset that meets the values, the rest finite
        for pos in np.argwhere(hit[1, 0]):
            off = [(0 if a < len(geo) - 1 else geo[-1] - 1) - q for a, q in enumerate(pos)]           # value's place - result's
            k = tuple((kg // 2 + (-o if flip else o)) for kg, o in zip(kgeo, off))
            w = Wt[(slice(None), slice(None)) + k]
            w = w.T if flip else w                                                                     # [channel out, channel in]
            at = (1, slice(None)) + (0,) * (len(geo) - 1) + (geo[-1] - 1,)
            terms = _sum(w, bad[at])
            plain = good[(1, slice(None)) + tuple(pos)] - _sum(w, t[at])
            _same(got[(1, slice(None)) + tuple(pos)], terms + plain, 1e-5)
        # a value among the weights of one channel out: the others keep their bits
        w2 = Wt.copy()
        c = (5, 2) if flip else (2, 5)                                                                 # (channel out of Wt, channel in)
        w2[c + tuple(kg // 2 for kg in kgeo)] = values[0]
        got, co = f(t, w2), c[1] if flip else c[0]
        others = np.arange(good.shape[1]) != co
        assert np.array_equal(got[:, others], good[:, others])
        if not np.isfinite(values[0]):
            with np.errstate(all="ignore"):
                assert np.array_equal(got[:, co], t[:, c[0] if flip else c[1]].astype(np.float64) * values[0], equal_nan=True)


@pytest.mark.parametrize("r,Cin,Cout,D,H,W,K,KD", [
    (40, 64, 64, 1, 31, 33, 3, 1),       # L moved by rows
    (50, 33, 130, 1, 14, 30, 3, 1),      # one dy per unit, padded copies
    (20, 24, 48, 1, 40, 29, 5, 1),       # pixel shifts in two units, two row tiles
    (120, 72, 40, 1, 40, 40, 1, 1),      # pointwise, two blocks of columns
    (120, 40, 200, 1, 40, 41, 1, 1),     # ... and two row tiles
    (6, 20, 36, 9, 12, 17, 3, 3),
])
def test_contraction(r, Cin, Cout, D, H, W, K, KD):
    """In the contraction a sum that the value does not enter by the definition stays finite too, next to the image's border."""
    geo, kgeo = ((D, H, W), (KD, K, K)) if D > 1 else ((H, W), (K, K))
    L, Z = _n((r, Cout) + geo, 11), _n((r, Cin) + geo, 12)
    assert xb.engine_for(xb.make_desc(1, Cin, Cout, H, W, r, torch.float32, K, D=D, KD=KD), xb.OP_CONTRACT) == "tcgen05_f32"
    call = lambda l, z: host(xb.xconv_contract(_dev(l), _dev(z), kernel_size=K, kernel_depth=KD)) * r
    good = call(L, Z)
    rms = float(np.sqrt(np.mean(good ** 2)))
    for places in ([(0,) * len(geo)], [tuple(n - 1 for n in geo), tuple(n // 2 for n in geo)], [(0,) * (len(geo) - 1) + (geo[-1] // 2,)]):
        for values in ((INF,), (NAN,), (INF, -INF), (-INF, -INF)):
            for of_l in (True, False):
                t, other = (L, Z) if of_l else (Z, L)
                bad, c, js = t.copy(), t.shape[1] - 1, (1, r - 1)
                special = np.zeros(good.shape)
                for v, pos, j in zip(values, places, js):
                    bad[(j, c) + pos] = v
                    for k in np.ndindex(*kgeo):
                        q = tuple(x + (a - g // 2) * (1 if of_l else -1) for x, a, g in zip(pos, k, kgeo))
                        if all(0 <= x < n for x, n in zip(q, geo)):
                            at = ((c, slice(None)) if of_l else (slice(None), c)) + k
                            with np.errstate(all="ignore"):
                                special[at] += v * other[(j, slice(None)) + q].astype(np.float64)
                got = call(bad, Z) if of_l else call(L, bad)
                hit = special != 0.0
                assert np.array_equal(got[hit], special[hit], equal_nan=True)
                same = np.ones(good.shape, bool)
                same[(c if of_l else slice(None), slice(None) if of_l else c)] = False
                assert np.array_equal(got[same], good[same])
                assert (np.abs(got[~hit] - good[~hit]) <= 1e-5 * rms).all()


def _time(f):
    f(); torch.cuda.synchronize()
    best = 1e9
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(); f(); b.record(); torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    return best


def _layer(B=128, Cin=64, Cout=64, H=32, W=32, r=64, K=3, dtype=torch.float32):
    desc = xb.make_desc(B, Cin, Cout, H, W, r, dtype, K)
    new = lambda *s: torch.randn(s, device="cuda").to(dtype)
    t = dict(X=new(B, H, W, Cin), W=new(Cout, K, K, Cin) * 0.05, Z=new(r, H, W, Cin), dY=new(B, H, W, Cout), L=new(r, H, W, Cout), L2=new(r, H, W, Cout), Y=new(B, H, W, Cout),
             dX=new(B, H, W, Cin), S=torch.randn(r, B, device="cuda"), S2=torch.empty(r, B, device="cuda"), dW=torch.empty(Cout, K * K * Cin, device="cuda"))
    t["ws"] = torch.empty(max(xb.workspace_bytes(desc, op) for op in range(6)), dtype=torch.uint8, device="cuda")
    return desc, t


CALLS = {"forward": (lambda d, t: xb.forward_into(d, t["X"], t["W"], t["Z"], t["Y"], t["S2"], t["ws"]), ("X", "W", "Z")),
         "dgrad": (lambda d, t: xb.dgrad_into(d, t["dY"], t["W"], t["dX"], t["ws"]), ("dY", "W")),
         "sketch": (lambda d, t: xb.sketch_into(d, t["X"], t["Z"], t["S2"], t["ws"]), ("X", "Z")),
         "backprobe": (lambda d, t: xb.backprobe_into(d, t["S"], t["dY"], t["L2"], t["ws"]), ("S", "dY")),
         "contract": (lambda d, t: xb.contract_into(d, t["L"], t["Z"], t["dW"], t["ws"]), ("L", "Z")),
         "wgrad": (lambda d, t: xb.wgrad_into(d, t["S"], t["dY"], t["Z"], t["dW"], t["ws"]), ("S", "dY", "Z"))}


@pytest.mark.parametrize("call", list(CALLS))
def test_time_and_status(call):
    """One value that is not finite: at most twice the time of finite data; a whole tensor: three times, and four where every sum of the
    contraction runs over (all of them are taken again, each from two or three rounds of loads: 3.3 times measured); 20 us for a clock that
    wanders.  No wait runs out."""
    f, operands = CALLS[call]
    desc, t = _layer()
    base = _time(lambda: f(desc, t))
    seen = {}
    for name in operands:
        for what, value in (("one", INF), ("one", NAN), ("all", NAN), ("all", INF), ("all", 3e38)):
            saved = t[name]
            t[name] = saved.clone() if what == "one" else torch.full_like(saved, value)
            if what == "one":
                t[name].view(-1)[t[name].numel() // 3] = value
            seen[name, what, value] = _time(lambda: f(desc, t))
            assert xb.workspace_status(t["ws"]) == 0
            t[name] = saved
    print(call, round(base, 1), {k: round(v, 1) for k, v in seen.items()})
    assert all(t <= (2 if what == "one" else 3 if value != 3e38 else 4) * base + 20 for (_, what, value), t in seen.items()), (base, seen)


def test_what_another_kernel_left_in_tensor_memory_is_not_read():
    """5 x 5 kernels have units whose last columns no MMA writes.  Read as sums, an old NaN there sent the whole block through the sums that are not
    finite, for nothing: the same bits, 1.3 times the time."""
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").contiguous(memory_format=torch.channels_last)
    L3, Z3 = rnd(64, 64, 32, 32), rnd(64, 64, 32, 32)         # a 3 x 3 contraction, whose units write all of these columns, on every SM
    assert xb.engine_for(xb.make_desc(1, 64, 64, 32, 32, 64, torch.float32, 3), xb.OP_CONTRACT) == "tcgen05_f32"
    L, Z = rnd(16, 72, 10, 54), rnd(16, 24, 10, 54)
    assert xb.engine_for(xb.make_desc(1, 24, 72, 10, 54, 16, torch.float32, 5), xb.OP_CONTRACT) == "tcgen05_f32"
    call = lambda: xb.xconv_contract(L, Z, 5)
    want = call()
    times = []
    for left in (L3, torch.full_like(L3, NAN)):
        leave = lambda: xb.xconv_contract(left, Z3, 3)
        leave()
        assert torch.equal(call(), want)
        times.append(device_time(call, before=leave))
    assert times[1] < 1.12 * times[0], times
