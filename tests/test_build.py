"""The build with a compiler that fails on one source (a stand-in for nvcc; nothing of the library is compiled)."""
import os
import stat
import subprocess
import time

import pytest

from paper_2106_06998_b200 import build as B


def test_no_compiler_is_left_running_behind_an_error(tmp_path, monkeypatch):
    log = tmp_path / "log"
    nvcc = tmp_path / "nvcc"
    nvcc.write_text(f"#!/bin/sh\ncase \"$*\" in *api.cu*) exit 3;; esac\nsleep 1\necho done >> {log}\n")
    nvcc.chmod(nvcc.stat().st_mode | stat.S_IXUSR)
    monkeypatch.setenv("NVCC", str(nvcc))
    monkeypatch.setattr(B, "CSRC", str(tmp_path))
    monkeypatch.setattr(B, "LIB", str(tmp_path / "lib.so"))
    with pytest.raises(subprocess.CalledProcessError) as e:
        B.build(force=True)
    assert e.value.returncode == 3
    finished = log.read_text().count("done") if os.path.exists(log) else 0
    time.sleep(1.5)
    assert finished == len(B.SOURCES) - 1 == log.read_text().count("done")
