"""The geometry that an open jac_opts gives, on both sides of the sizes where it
changes, against a pinned one: iterates bit for bit.

Test values: both add the same n squares, in different orders, so each sum
carries at most n roundings of it: relative difference <= 2 n u.
"""
import numpy as np
import pytest

from paper_2112_02377_gb300 import jacobi as J
from paper_2112_02377_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _check(a, p, n, per_sm, stages):
    try:
        sa = J.jac_stats(a)
        assert (sa["ctas_per_sm"], sa["stages"]) == (per_sm, stages)
        for k in (1, 6):
            ra, rp = J.jac_sweep(a, k), J.jac_sweep(p, k)
            assert np.array_equal(J.jac_get_x(a, None, n), J.jac_get_x(p, None, n))
            assert abs(ra - rp) <= 2 * n * U * rp
    finally:
        J.jac_free(a)
        J.jac_free(p)


@pytest.mark.parametrize("make,lanes,per_sm,stages", [
    (lambda: W.laplace7((85, 84, 84)), 0, 2, 2),            # 599,760 rows
    (lambda: W.laplace7((100, 75, 80)), 0, 2, 4),           # 600,000
    (lambda: W.fe27_deleted(50, seed=1), 1, 2, 2)])         # one lane, rows longer than a small stage's share
def test_open_geometry_sweeps_are_the_pinned_ones(make, lanes, per_sm, stages):
    A = make()
    b = np.random.default_rng(1).uniform(-1, 1, A.n)
    a = J.jac_setup(A, b, J.JAC_BANDROW, 3, J.opts(lanes_per_row=lanes))
    p = J.jac_setup(A, b, J.JAC_BANDROW, 3, J.opts(lanes_per_row=J.jac_stats(a)["lanes_per_row"], variant=2,
                                                   ctas_per_sm=3))
    _check(a, p, A.n, per_sm, stages)


@pytest.mark.parametrize("edge,sub,per_sm,stages", [(5, 2, 2, 2), (24, 3, 2, 2), (83, 2, 2, 2), (84, 4, 2, 4),
                                                    (101, 2, 3, 3)])
def test_open_split_geometry_sweeps_are_the_pinned_ones(edge, sub, per_sm, stages):
    n = edge ** 3
    b = np.random.default_rng(2).uniform(-1, 1, n)
    loc = W.cell_box_locals("laplace7", edge, (sub,) * 3)
    a = J.jac_setup_local(n, loc, b, J.opts())
    p = J.jac_setup_local(n, loc, b, J.opts(variant=2, lanes_per_row=1, ctas_per_sm=2, stages=4 if per_sm == 3 else 3))
    _check(a, p, n, per_sm, stages)
