"""sweeps_per_graph is honoured where the matrix is kept in shared memory too: the
rule on the CPU (tests/cpp/resident_step_check.cpp), and on the GPU the same iterates,
counts and histories from launches of any length, down to one sweep."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from conftest import ROOT


def test_the_callers_number_is_used(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = os.path.join(str(tmp_path), "resident_step_check")
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-Wall", "-Wextra", "-Werror", "-I",
                           os.path.join(ROOT, "paper_2112_02377_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "cpp", "resident_step_check.cpp"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("edge,k,resident", [(17, 1, True), (17, 2, True), (17, 3, True), (17, 4, True), (17, 37, True),
                                             (17, 4096, True), (48, 1, False), (48, 2, True), (70, 2, False), (70, 3, True)])
def test_launches_of_any_length(edge, k, resident, local):
    from paper_2112_02377_gb300 import jacobi as J
    from paper_2112_02377_gb300 import workloads as W
    A = W.laplace7(edge)
    b = np.random.default_rng(9).uniform(-1, 1, A.n)
    kw = dict(norm=0, stop=J.JAC_STOP_LOCAL, history=4096) if local else dict(history=4096)
    with J.Solver(A, b, "bandrow", 3, sweeps_per_graph=k, **kw) as a, J.Solver(A, b, "bandrow", 3, **kw) as d:
        assert (a.stats()["ctas_per_sm"] == 1) == resident and d.stats()["ctas_per_sm"] == 1
        tol = 1e-4 if local else 1e-2
        for call in (lambda s: s.sweep(9), lambda s: s.solve(tol, 300), lambda s: s.sweep(2), lambda s: s.solve(0.0, 330)):
            ra, rd = call(a), call(d)
            if resident:
                assert ra == rd and np.array_equal(a.history(), d.history())
            assert np.array_equal(a.x(), d.x()) and a.stats()["k"] == d.stats()["k"]
            assert len(a.history()) == len(d.history())
