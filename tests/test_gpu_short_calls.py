"""Calls of one or two sweeps on a system that the resident kernel holds: they run
in the pipelined kernel (two CTAs per SM: jac_get_trace names the CTAs of the last
call), longer ones in the resident kernel, in any order on one context, with
the iterates, counts and stops of a context pinned to the pipelined kernel.

Test values: both kernels add the same n squares, in different orders, so each
sum carries at most n roundings of it: relative difference <= 2 n u.
"""
import numpy as np
import pytest

from paper_2112_02377_gb300 import jacobi as J
from paper_2112_02377_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53

# the longest call that takes the pipelined kernel, by a CTA's shared memory
MATRICES = {"small": (lambda: W.laplace7(16), 0), "middle": (lambda: W.laplace7(48), 1),
            "large": (lambda: W.laplace7((71, 70, 69)), 2), "fe": (lambda: W.fe27_deleted(44, seed=4), 2)}


def _ctas(s):
    return len(J.jac_get_trace(s.ctx)[0])


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("name", ["middle", "large", "fe"])
def test_solves_of_large_systems_stop_at_the_same_sweep(name, local):
    """Decisions are read three sweeps late in the middle one, two in the others."""
    A = MATRICES[name][0]()
    b = np.random.default_rng(6).uniform(-1, 1, A.n)
    kw = dict(norm=0, stop=J.JAC_STOP_LOCAL, history=2048) if local else dict(history=2048)
    with J.Solver(A, b, "bandrow", 4, **kw) as a, \
            J.Solver(A, b, "bandrow", 4, variant=2, ctas_per_sm=2, lanes_per_row=a.stats()["lanes_per_row"], **kw) as p:
        assert a.stats()["ctas_per_sm"] == 1
        p.sweep(40)
        h = p.history()                           # test values of x^0 .. x^39: each ends a solve of its own
        tols = [1.0001 * h[k] for k in (0, 1, 2, 3, 4, 5, 17)]
        for maxit, tol in [(1000, t) for t in tols] + [(m, 0.0) for m in (4, 5, 511, 512, 513, 514)]:
            a.set_x(), p.set_x()
            ka, kp = a.solve(tol, maxit), p.solve(tol, maxit)
            assert ka[0] == kp[0] and ka[2] == kp[2] and np.array_equal(a.x(), p.x())
            ha, hp = a.history(), p.history()
            assert len(ha) == len(hp) == ka[0] + 1 and np.all(np.abs(ha - hp) <= 2 * A.n * U * hp)
            assert a.stats()["stop_part"] == p.stats()["stop_part"]


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("name", list(MATRICES))
def test_short_calls_take_the_pipelined_kernel(name, local):
    make, most = MATRICES[name]
    A = make()
    b = np.random.default_rng(5).uniform(-1, 1, A.n)
    kw = dict(norm=0, stop=J.JAC_STOP_LOCAL) if local else {}
    kw.update(history=64, debug=1)
    with J.Solver(A, b, "bandrow", 3, **kw) as a, \
            J.Solver(A, b, "bandrow", 3, variant=2, ctas_per_sm=2, lanes_per_row=a.stats()["lanes_per_row"], **kw) as p:
        sms = a.stats()["ctas"]
        assert a.stats()["ctas_per_sm"] == 1

        def same():
            assert np.array_equal(a.x(), p.x())
            sa, sp = a.stats(), p.stats()
            assert (sa["k"], sa["sweeps_total"], sa["last_resinf"]) == (sp["k"], sp["sweeps_total"], sp["last_resinf"])
            ha, hp = a.history(), p.history()
            assert len(ha) == len(hp) and np.all(np.abs(ha - hp) <= 2 * A.n * U * hp)

        for k in (1, 7, 2, 1, 3, 1, 1, 12, 2, 5):   # every buffer of the rotation as a start of either kernel
            a.sweep(k), p.sweep(k)
            assert _ctas(a) == (2 * sms if k <= most else sms)
            same()
        for maxit in (0, 1, 2, 0, 3):               # a solve of maxit sweeps evaluates maxit + 1 iterates
            a.set_x(), p.set_x()
            ka, kp = a.solve(0.0, maxit), p.solve(0.0, maxit)
            assert _ctas(a) == (2 * sms if maxit + 1 <= most else sms)
            assert ka[0] == kp[0] == maxit and ka[2] == kp[2] == J.JAC_ENOTCONV
            same()
        scale = 2 * a.history().max()
        for maxit in (3, 100):                      # passes at once, at k = 3: one iterate, in either kernel
            ka, kp = a.solve(scale, maxit), p.solve(scale, maxit)
            assert _ctas(a) == (2 * sms if maxit == 3 and most else sms)
            assert ka[0] == kp[0] == 3 and ka[2] == kp[2] == J.JAC_OK
            same()
        assert a.solve(0.0, 40)[0] == p.solve(0.0, 40)[0] == 40
        same()
