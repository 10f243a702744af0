"""Source checks of the kernels on split operands that need no GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_06998_b200", "csrc")


def _code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _functions():
    """Name, whether it is a kernel, and body of every device function of the sources."""
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            code = re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", "", _code(name))
            for chunk in code.split("\n}\n"):
                found = re.findall(r"__(device|global)__[^;{}]*?\b(\w+)\s*\([^;]*?\)\s*\{", chunk)
                for kind, function in found:
                    yield function, kind == "global", chunk


def test_every_kernel_that_takes_tensor_memory_does_so_before_it_lets_the_next_one_start():
    """Whatever functions it goes through: a kernel that reaches the allocation does so once, by one warp, and the go-ahead for the next kernel is
    given behind the allocation and nowhere else."""
    functions = list(_functions())
    reach = {f for f, _, body in functions if "tcgen05.alloc." in body}
    assert reach == {"tmem_alloc"}
    calls = lambda body, names: re.findall(r"\b(%s)\(" % "|".join(sorted(names)), body)
    while True:
        more = {f for f, _, body in functions if set(calls(body, reach)) - {f}} | reach
        if more == reach:
            break
        reach = more
    kernels = {f for f, kernel, _ in functions if kernel} & reach
    assert kernels == {"tc_gemm_kernel", "conv_tc_kernel", "contract_halo_kernel", "conv_split_kernel", "contract_split_kernel", "gemm_split_kernel"}
    helpers = reach - kernels
    assert helpers == {"tmem_alloc", "tmem_alloc_then_trigger", "split_begin"}
    bodies = {f: body.split(f + "(", 1)[1] for f, _, body in functions if f in reach}
    order = bodies["tmem_alloc_then_trigger"]
    assert 0 <= order.index("tmem_alloc(") < order.index("pdl_trigger(") and order.count("pdl_trigger(") == 1
    assert "pdl_trigger(" not in bodies["tmem_alloc"]
    for f in kernels | {"split_begin"}:
        taken = calls(bodies[f], helpers - {"tmem_alloc"})
        assert len(taken) == 1 and "tmem_alloc(" not in bodies[f] and "pdl_trigger(" not in bodies[f], f
        if taken == ["tmem_alloc_then_trigger"]:
            assert re.search(r"if \(warp == 1\) \{?\s*tmem_alloc_then_trigger\(", bodies[f]), f


def _body(name, function):
    """The text of a function of one source, from its name to the brace that closes it at the start of a line."""
    return _code(name).split(function + "(", 1)[1].split("\n}\n")[0]


def test_a_wait_by_one_lane_orders_the_reads_of_the_others():
    """One lane asks the barrier for all: the lanes that read behind it need a warp barrier, since a shuffle orders no memory."""
    body = _body("split_f32.cuh", "bool split_wait")
    assert body.index("mbar_wait(") < body.index("__syncwarp()") and body.rindex("__shfl_sync") < body.index("__syncwarp()")


def test_nothing_that_an_earlier_kernel_writes_is_read_as_constant():
    """These kernels may start while the kernel before them still writes what they read: no load through the read-only cache, whose
    lines nothing invalidates within a kernel."""
    for name in ("contract_split.cu", "conv_split.cu", "gemm_split.cu", "split_f32.cuh"):
        assert "__ldg" not in _code(name) and "ld.global.nc" not in _code(name), name
    # (a const pointer that nothing else writes through may be read that way too; chan_scale is the caller's)
    assert re.findall(r"const \w+\* __restrict__ (\w+)", "".join(map(_code, ("contract_split.cu", "conv_split.cu", "gemm_split.cu")))) == ["chan_scale"]
