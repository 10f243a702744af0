"""Source checks of the kernels on split operands that need no GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_06998_b200", "csrc")


def _code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def test_they_take_tensor_memory_before_they_let_the_next_kernel_start():
    """As for the other holders of tensor memory: it is taken through the function that gives the go-ahead behind the allocation (here by
    way of split_take_columns), once, by one warp, and nothing else in those kernels gives it."""
    helper = re.findall(r"void split_take_columns\([^)]*\) \{([^}]*)\}", _code("split_f32.cuh"))
    assert helper == [" tmem_alloc_then_trigger(slot, columns); "]
    holders = []
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        for kernel in _code(name).split("__global__")[1:]:
            body = kernel.split("\n}\n")[0]
            if "split_take_columns" in body:
                holders.append(name)
                assert body.count("if (warp == 1) split_take_columns(") == 1 and body.count("split_take_columns") == 1, name
                assert "tmem_alloc" not in body and "pdl_trigger(" not in body, name
    assert holders == ["contract_split.cu", "conv_split.cu", "gemm_split.cu"]


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
