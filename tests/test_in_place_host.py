"""Vectors of another GPU, managed and host memory are copied, not dereferenced:
the rule on the CPU (tests/cpp/in_place_check.cpp), and that every vector which a
kernel takes in place is asked about with the owner that the driver names."""
import os
import re
import shutil
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2112_02377_gb300", "csrc")


def test_only_own_device_memory_is_used_in_place(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = os.path.join(str(tmp_path), "in_place_check")
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-Wall", "-Wextra", "-Werror", "-I", CSRC,
                           os.path.join(ROOT, "tests", "cpp", "in_place_check.cpp"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout


def test_the_owner_comes_from_the_driver():
    with open(os.path.join(CSRC, "jac_api.cu")) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    rule = src[src.index("bool in_place("):]
    rule = rule[:rule.index("\n}")]
    assert "cudaPointerGetAttributes(&a, p)" in rule
    assert "usable_in_place(a.type == cudaMemoryTypeDevice, a.device, c->device, (uintptr_t)p)" in rule
