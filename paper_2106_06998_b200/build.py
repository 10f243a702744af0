"""Builds libxconv.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the binding's native part with the host compiler."""
from __future__ import annotations

import os
import shutil
import subprocess
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libxconv.so")
MARSHAL, MARSHAL_SOURCE = os.path.join(HERE, "_marshal.so"), os.path.join(HERE, "csrc", "marshal.cpp")
SOURCES = ["api.cu", "tc_kernels.cu", "conv_tc.cu", "contract_tc.cu", "stream_tc.cu", "conv_fma.cu", "small_f32.cu", "conv_split.cu", "contract_split.cu", "gemm_split.cu",
           "static_scratch.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--use_fast_math=false", "-Xcompiler", "-fPIC,-O2", "-cudart", "static"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: libxconv cannot be built")


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")] + [os.path.join(HERE, "..", "include", "xconv.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def marshal_key() -> str:
    """What the binding's native part is compiled against, beside its sources: it uses torch's C++ classes and the interpreter's ABI."""
    import sysconfig
    import torch
    return f"xconv marshal for torch {torch.__version__}, {sysconfig.get_config_var('SOABI')}"


def _marshal_current() -> bool:
    if not os.path.exists(MARSHAL):
        return False
    header = os.path.join(HERE, "..", "include", "xconv.h")
    with open(MARSHAL, "rb") as f:
        return os.path.getmtime(MARSHAL) >= max(map(os.path.getmtime, (MARSHAL_SOURCE, header))) and marshal_key().encode() + b"\0" in f.read()


def build_marshal(force: bool = False) -> str:
    """Compiles the binding's calls on ordinary tensors (csrc/marshal.cpp) against the installed torch; returns the module's path."""
    if not force and _marshal_current():
        return MARSHAL
    import sysconfig
    import torch
    top = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    fresh = os.path.join(HERE, "_marshal_fresh.so")
    # (the CUDA runtime that it calls is the one that libc10_cuda brings with it)
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                    f'-DXM_KEY="{marshal_key()}"', "-isystem", os.path.join(top, "include"), "-isystem", os.path.join(top, "include", "torch", "csrc", "api", "include"),
                    "-isystem", sysconfig.get_paths()["include"], "-isystem", os.path.join(cuda, "include"), MARSHAL_SOURCE, "-o", fresh,
                    "-L" + os.path.join(top, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"], check=True)
    os.replace(fresh, MARSHAL)
    return MARSHAL


def _try_build_marshal(force: bool) -> None:
    """The library alone is enough (the binding then calls it through ctypes): a machine without torch's or Python's headers, or without a
    host compiler, gets a warning."""
    try:
        build_marshal(force)
    except (OSError, subprocess.CalledProcessError, ImportError) as e:
        warnings.warn(f"{MARSHAL} was not built ({e}): calls will go through ctypes", RuntimeWarning, stacklevel=3)


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    """Compile every CUDA source into one shared library; returns its path.
    ``extra_flags`` go to nvcc."""
    if not force and not _stale():
        _try_build_marshal(False)
        return LIB
    objs, jobs = [], []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        cmd = [_nvcc(), *[f for f in NVCC_FLAGS if f != "--use_fast_math=false"], *extra_flags, "-c",
               os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        jobs.append((cmd, subprocess.Popen(cmd)))
        objs.append(obj)
    codes = [job.wait() for _, job in jobs]     # the sources compile side by side; none is left running behind an error
    for (cmd, _), code in zip(jobs, codes):
        if code != 0:
            raise subprocess.CalledProcessError(code, cmd)
    subprocess.run([_nvcc(), "-shared", "-cudart", "static", "-o", LIB, *objs, "-ldl"], check=True)
    _try_build_marshal(force)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv, extra_flags=[a for a in sys.argv[1:] if a.startswith("-D")]))
