"""The waits of the resident kernel.

Its math warps and one spare warp pass two CTA barriers a sweep and leave the
sweep loop on a shared flag; the barriers name their thread count, so a warp that
leaves alone would keep the others waiting without a limit.  The flag is therefore
written by thread 0 alone, between the two barriers (in its grid barrier), and read
after the second: no write can fall between two warps' reads.  The first test checks
that in the source, the second that a missing CTA ends a solve with an error status,
whichever part waits for it.
"""
import os
import re

import numpy as np
import pytest

from conftest import ROOT


def _kernel_source():
    with open(os.path.join(ROOT, "paper_2112_02377_gb300", "csrc", "jac_resident.cu")) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _body(src, opening):
    """The braces' content after the first occurrence of `opening`."""
    at = src.index(opening) + len(opening)
    at = src.index("{", at)
    depth, end = 1, at + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[end], 0)
        end += 1
    return src[at:end]


def test_the_loop_flag_is_written_between_the_barriers_only():
    src = _kernel_source()
    writes = len(re.findall(r"\bs_fail\s*=[^=]", src))
    in_barrier = len(re.findall(r"\bs_fail\s*=[^=]", _body(src, "auto grid_barrier = [&]()")))
    at_start = len(re.findall(r"\bs_fail = 0;", src))
    assert in_barrier >= 1 and at_start == 1 and writes == in_barrier + at_start
    calls = len(re.findall(r"\bgrid_barrier\(\)", src))
    guarded = len(re.findall(r"if \(tid == 0\) grid_barrier\(\);\s*cta_sync<2, SYNC>\(\);", src))
    assert calls == guarded == 2
    # each is behind the first barrier
    for m in re.finditer(r"if \(tid == 0\) grid_barrier\(\);", src):
        before = src[:m.start()]
        assert before.rindex("cta_sync<1, SYNC>") > max(before.rfind("cta_sync<2, SYNC>"), before.rindex("publish_sweep("))


@pytest.mark.gpu
@pytest.mark.parametrize("stop", ["global", "local"])
@pytest.mark.parametrize("cta", [0, 7, 151])                 # CTA 0 takes the decisions
def test_a_missing_cta_ends_the_solve(cta, stop):
    from paper_2112_02377_gb300 import jacobi as J
    from paper_2112_02377_gb300 import workloads as W
    A = W.laplace7((19, 17, 13))
    kw = dict(norm=0, stop=J.JAC_STOP_LOCAL) if stop == "local" else {}
    with J.Solver(A, np.ones(A.n), "bandrow", 3, fault_skip_cta=cta, timeout_cycles=20_000_000, **kw) as s:
        assert s.stats()["ctas_per_sm"] == 1 and s.stats()["stages"] == 0
        with pytest.raises(J.JacobiError) as e:
            s.solve(1e-12, 100000)
        assert e.value.status == J.JAC_ETIMEOUT
    with J.Solver(A, np.ones(A.n), "bandrow", 3, **kw) as s:  # the next context is not affected
        assert s.solve(1e-6, 100000)[2] == J.JAC_OK
