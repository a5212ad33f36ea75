"""The geometry that an open jac_opts gives mixed contexts, on both sides of the
sizes where it changes, against a pinned one: whole cycles bit for bit (an FP32
sweep's sums do not depend on tiles or CTAs, and its FP64 pass keeps each row's).

Test values: both add the same n squares, in different orders, so each sum
carries at most n roundings of it: relative difference <= 2 n u."""
import numpy as np
import pytest

from paper_2112_02377_gb300 import jacobi as J
from paper_2112_02377_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _check(A, per_sm, stages, inner, split=J.JAC_BANDROW, **kw):
    b = np.random.default_rng(1).uniform(-1, 1, A.n)
    kw.update(precision=J.JAC_MIXED, inner_sweeps=inner)
    a = J.jac_setup(A, b, split, 3, J.opts(**kw))
    s = J.jac_stats(a)
    other = 2 if per_sm == 3 else 3
    p = J.jac_setup(A, b, split, 3, J.opts(lanes_per_row=s["lanes_per_row"], variant=2, ctas_per_sm=other, **kw))
    try:
        assert (s["ctas_per_sm"], s["stages"]) == (per_sm, stages)
        for _ in range(2):
            k = J.jac_stats(a)["k"] + 2 * inner
            ra, rp = J.jac_solve(a, 1e-30, k), J.jac_solve(p, 1e-30, k)
            assert ra[0] == rp[0] and ra[2] == rp[2] and abs(ra[1] - rp[1]) <= 2 * A.n * U * rp[1]
            assert np.array_equal(J.jac_get_x(a, None, A.n), J.jac_get_x(p, None, A.n))
    finally:
        J.jac_free(a)
        J.jac_free(p)


@pytest.mark.parametrize("dims,inner,per_sm", [
    ((50, 50, 50), 128, 2),                   # 2 rounds of tiles with two CTAs per SM, 2 with three
    ((54, 54, 54), 128, 3),                   # 3 and 2
    ((48, 48, 48), 128, 2),                   # 2 and 1, the one 95 % full
    ((47, 47, 48), 128, 3),                   # 2 and 1, 91 %
    ((46, 46, 46), 128, 2), ((46, 46, 46), 132, 3),      # rows times the cycle's sweeps
    ((16, 16, 16), 4096, 2), ((40, 40, 40), 512, 2),     # long cycles, one round either way
    ((74, 73, 74), 32, 2), ((74, 74, 74), 32, 3)])       # short ones
def test_open_mixed_geometry_one_lane(dims, inner, per_sm):
    _check(W.laplace7(dims), per_sm, 3 if per_sm == 3 else 4, inner)


def _plane(edge, corners):
    """A plane's 5- or 9-point operator on edge x edge nodes (diagonal 4 or 8, others -1)."""
    n = edge * edge
    i, j = np.arange(n) % edge, np.arange(n) // edge
    offs = [(a, c) for c in (-1, 0, 1) for a in (-1, 0, 1) if corners or a == 0 or c == 0]
    ok = np.stack([(i + a >= 0) & (i + a < edge) & (j + c >= 0) & (j + c < edge) for a, c in offs], 1)
    col = np.stack([i + a + edge * (j + c) for a, c in offs], 1)
    val = np.tile([float(len(offs) - 1) if a == c == 0 else -1.0 for a, c in offs], (n, 1))
    ptr = np.concatenate([[0], np.cumsum(ok.sum(1))])
    return W.CSR(n=n, rowptr=ptr.astype(np.int32), col=col[ok].astype(np.int32), val=val[ok])


@pytest.mark.parametrize("edge,corners,per_sm", [(450, False, 2), (700, False, 3), (500, True, 2), (980, True, 3)])
def test_open_mixed_geometry_of_planes(edge, corners, per_sm):
    _check(_plane(edge, corners), per_sm, 3 if per_sm == 3 else 4, 128)


@pytest.mark.parametrize("corners,per_sm,stages", [(False, 3, 3), (True, 2, 4)])
def test_open_fp64_geometry_of_planes(corners, per_sm, stages):
    A = _plane(1740, corners)                 # 3,027,600 rows
    b = np.random.default_rng(2).uniform(-1, 1, A.n)
    a = J.jac_setup(A, b, J.JAC_BANDROW, 1, J.opts())
    p = J.jac_setup(A, b, J.JAC_BANDROW, 1, J.opts(variant=2, ctas_per_sm=5 - per_sm))
    try:
        s = J.jac_stats(a)
        assert (s["ctas_per_sm"], s["stages"]) == (per_sm, stages)
        for k in (1, 6):
            ra, rp = J.jac_sweep(a, k), J.jac_sweep(p, k)
            assert np.array_equal(J.jac_get_x(a, None, A.n), J.jac_get_x(p, None, A.n))
            assert abs(ra - rp) <= 2 * A.n * U * rp
    finally:
        J.jac_free(a)
        J.jac_free(p)


@pytest.mark.parametrize("edge", [111, 113, 114, 115])     # entries kept in L2 or not; interface rows cost more from 1,500,000
def test_open_mixed_geometry_of_boxes(edge):
    _check(W.laplace7(edge), 3, 3, 32, J.JAC_SUBSTRUCT, grid=(edge,) * 3, subdomains=(2, 2, 2))


def _box_rows(edge, reach):
    """Every node of a box of +-reach around a node of edge^3 (diagonal the entries less one, others -1)."""
    n = edge ** 3
    g = np.arange(n)
    node = (g % edge, g // edge % edge, g // edge ** 2)
    offs = [(a, c, e) for e in range(-reach[2], reach[2] + 1) for c in range(-reach[1], reach[1] + 1)
            for a in range(-reach[0], reach[0] + 1)]
    ok = np.stack([np.all([(node[q] + o[q] >= 0) & (node[q] + o[q] < edge) for q in range(3)], axis=0) for o in offs], 1)
    col = np.stack([g + o[0] + edge * (o[1] + edge * o[2]) for o in offs], 1)
    val = np.tile([float(len(offs) - 1) if o == (0, 0, 0) else -1.0 for o in offs], (n, 1))
    ptr = np.concatenate([[0], np.cumsum(ok.sum(1))])
    return W.CSR(n=n, rowptr=ptr.astype(np.int32), col=col[ok].astype(np.int32), val=val[ok])


@pytest.mark.parametrize("edge,reach,lanes,stages", [
    (48, (1, 2, 2), 8, 2), (54, (1, 2, 2), 8, 4),     # 75-point rows, in L2 and past it
    (48, (2, 2, 2), 8, 2),                            # 125-point rows
    (70, (1, 1, 1), 2, 2), (71, (1, 1, 1), 2, 3)])    # 27-point rows on both sides of 350,000
def test_open_mixed_geometry_several_lanes(edge, reach, lanes, stages):
    A = _box_rows(edge, reach)
    with J.Solver(A, None, precision=J.JAC_MIXED) as s:
        assert s.stats()["lanes_per_row"] == lanes
    _check(A, 2, stages, 32)
