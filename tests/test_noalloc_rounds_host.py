"""The index arithmetic of the allocation-free sweep's staged rounds on the CPU,
up to the last position that an int32 row pointer can name:
tests/cpp/rounds_check.cpp is built with the kernel's own header and run, once
optimised and once under gcc's sanitizers."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT
from test_split_layout_host import SANITIZE, _sanitizers_available


@pytest.mark.parametrize("mode", ["optimised", "sanitized"])
def test_staged_rounds_stay_inside_their_block(tmp_path, mode):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    if mode == "sanitized" and not _sanitizers_available(cxx, str(tmp_path)):
        pytest.skip("the compiler has no AddressSanitizer / UndefinedBehaviorSanitizer runtime")
    exe = os.path.join(str(tmp_path), "rounds_check")
    subprocess.check_call([cxx, "-std=c++17", *(SANITIZE if mode == "sanitized" else ["-O2"]), "-Wall", "-Wextra", "-Werror",
                           "-I", os.path.join(ROOT, "paper_2112_02377_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "cpp", "rounds_check.cpp"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
