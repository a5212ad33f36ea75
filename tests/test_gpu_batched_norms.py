"""Per-(system, right-hand side) norms and decisions of a batched context: every
system against a single context of its own, for one, two and four right-hand
sides, both tile sizes and both norms, over systems of one row, around a tile's
edge, several in a CTA and one over many CTAs.

The rows' arithmetic is the same in both kernels, so iterates, counts and
infinity norms agree bit for bit; sums of n squares added in different orders
differ by at most 2 n u of the sum.
"""
import numpy as np
import pytest

from paper_2112_02377_gb300 import jacobi as J
from paper_2112_02377_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
EDGES = [(1, 1, 1), (95, 1, 1), (97, 1, 1), (14, 16, 1), (225, 1, 1), (9, 8, 7), (33, 32, 31), (2, 2, 2), (12, 12, 12)]


def _systems(nrhs, seed):
    rng = np.random.default_rng(seed)
    mats = [W.laplace7(e) for e in EDGES]
    # right-hand sides of different sizes: the largest residual is not always in the first one
    return mats, [rng.uniform(-1, 1, (A.n, nrhs)) * 10.0 ** rng.integers(-2, 3, nrhs) for A in mats]


def _check(ctx, mats, rhs, nrhs, norm, call):
    sweeps, rel = J.jac_get_batch_results(ctx, len(mats) * nrhs)
    x, at = J.jac_get_x(ctx), 0
    for s, (A, b) in enumerate(zip(mats, rhs)):
        for q in range(nrhs):
            with J.Solver(A, b[:, q].copy(), variant=2, ctas_per_sm=2, lanes_per_row=1, norm=norm) as one:
                k, r = call(one)
                assert sweeps[s * nrhs + q] == k, (s, q)
                tol = 0.0 if norm == 0 else 2 * A.n * U * r
                assert abs(rel[s * nrhs + q] - r) <= tol, (s, q)
                assert np.array_equal(x[at:at + A.n * nrhs].reshape(A.n, nrhs)[:, q], one.x()), (s, q)
        at += A.n * nrhs


@pytest.mark.parametrize("norm", [0, 2])
@pytest.mark.parametrize("nrhs,rows", [(1, 224), (2, 224), (4, 224), (2, 96), (4, 96)])
def test_batched_decisions_are_each_systems_own(nrhs, rows, norm):
    mats, rhs = _systems(nrhs, 3 * nrhs + norm)
    ctx = J.jac_setup_batched(mats, rhs, J.opts(nrhs=nrhs, tile_rows=rows, norm=norm))
    try:
        J.jac_sweep(ctx, 65)                         # fixed sweeps: the test value of x^64, over two launches

        def sweep(one):
            return 64, one.sweep(65)

        _check(ctx, mats, rhs, nrhs, norm, sweep)
        J.jac_set_x(ctx)
        tol, maxit = (1e-6, 400) if norm == 2 else (1e-4, 400)       # some converge, some reach the limit
        J.jac_solve(ctx, tol, maxit)

        def solve(one):
            k, r, _ = one.solve(tol, maxit)
            return k, r

        _check(ctx, mats, rhs, nrhs, norm, solve)
    finally:
        J.jac_free(ctx)


def test_batched_reports_a_diverging_right_hand_side():
    mats, rhs = _systems(4, 5)
    rng = np.random.default_rng(6)
    M = rng.uniform(-1, 1, (30, 30))
    np.fill_diagonal(M, 0.05)
    mats.insert(3, W.dense_to_csr(M))
    rhs.insert(3, np.concatenate([np.zeros((30, 3)), np.ones((30, 1))], 1))   # only the fourth one grows
    ctx = J.jac_setup_batched(mats, rhs, J.opts(nrhs=4))
    try:
        with pytest.raises(J.JacobiError) as e:
            J.jac_solve(ctx, 1e-8, 20000)
        assert e.value.status == J.JAC_ENUMERIC
    finally:
        J.jac_free(ctx)
