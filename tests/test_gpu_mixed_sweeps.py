"""jac_sweep on a mixed context is FP64 sweeps: they run in the geometry that suits
those (jac_get_trace names the CTAs of the last call) where the context's cycles
take a third CTA per SM, with the iterates of an FP64 context, and the cycles
after and between them are those of a context pinned to their own geometry.
"""
import numpy as np
import pytest

from paper_2112_02377_gb300 import jacobi as J
from paper_2112_02377_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("dims,split,per_sm", [((64, 64, 64), "bandrow", 2), ((64, 65, 66), "substruct", 2),
                                               ((96, 90, 91), "bandrow_nnz", 2), ((100, 100, 101), "bandrow", 2)])
def test_fp64_sweeps_of_a_mixed_context(dims, split, per_sm):
    A = W.laplace7(dims)
    b = np.random.default_rng(7).uniform(-1, 1, A.n)
    kw = dict(subdomains=(2, 2, 2)) if split == "substruct" else {}
    with J.Solver(A, b, split, 3, precision=J.JAC_MIXED, debug=1, **kw) as a, \
            J.Solver(A, b, split, 3, precision=J.JAC_MIXED, variant=2, ctas_per_sm=3, **kw) as p, \
            J.Solver(A, b, split, 3, variant=2, lanes_per_row=1, **kw) as f:
        sms = a.stats()["ctas"] // 3
        assert a.stats()["ctas_per_sm"] == 3
        for k in (1, 2, 70):
            ra, rf = a.sweep(k), f.sweep(k)
            assert len(J.jac_get_trace(a.ctx)[0]) == per_sm * sms
            assert np.array_equal(a.x(), f.x()) and abs(ra - rf) <= 2 * A.n * U * rf
        p.sweep(73)
        for _ in range(2):                        # whole cycles, then FP64 sweeps again
            ka, kp = a.solve(1e-30, a.stats()["k"] + 256), p.solve(1e-30, p.stats()["k"] + 256)
            assert ka[0] == kp[0] and ka[2] == kp[2] and len(J.jac_get_trace(a.ctx)[0]) == 3 * sms
            assert np.array_equal(a.x(), p.x())
            a.sweep(3), p.sweep(3)
            assert np.array_equal(a.x(), p.x())


def _fifteen_points(edge):
    """The faces' and corners' neighbours on edge^3 nodes (diagonal 14, others -1)."""
    n = edge ** 3
    g = np.arange(n)
    node = (g % edge, g // edge % edge, g // edge ** 2)
    offs = [(a, c, e) for e in (-1, 0, 1) for c in (-1, 0, 1) for a in (-1, 0, 1) if abs(a) + abs(c) + abs(e) in (0, 1, 3)]
    ok = np.stack([np.all([(node[q] + o[q] >= 0) & (node[q] + o[q] < edge) for q in range(3)], axis=0) for o in offs], 1)
    col = np.stack([g + o[0] + edge * (o[1] + edge * o[2]) for o in offs], 1)
    val = np.tile([14.0 if o == (0, 0, 0) else -1.0 for o in offs], (n, 1))
    ptr = np.concatenate([[0], np.cumsum(ok.sum(1))])
    return W.CSR(n=n, rowptr=ptr.astype(np.int32), col=col[ok].astype(np.int32), val=val[ok])


@pytest.mark.parametrize("edge,per_sm", [(60, 2), (86, 3)])    # two large stages below 600,000 rows
def test_fp64_sweeps_of_longer_rows(edge, per_sm):
    A = _fifteen_points(edge)
    b = np.random.default_rng(8).uniform(-1, 1, A.n)
    with J.Solver(A, b, precision=J.JAC_MIXED) as a, J.Solver(A, b, variant=2, ctas_per_sm=2, lanes_per_row=1) as f:
        sms = a.stats()["ctas"] // 3
        assert a.stats()["ctas_per_sm"] == 3
        for k in (1, 4):
            ra, rf = a.sweep(k), f.sweep(k)
            assert len(J.jac_get_trace(a.ctx)[0]) == per_sm * sms
            assert np.array_equal(a.x(), f.x()) and abs(ra - rf) <= 2 * A.n * U * rf
