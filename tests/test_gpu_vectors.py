"""Vectors in and out of a context: device memory is read and written in place,
host memory and unaligned views go through a staged copy, and ||b|| comes from
the kernel that gathers b.  Sizes around its blocks (256 rows, four rows a
thread and step), every row order, and the gradient's output over its inputs.

From x = 0 the residual is b itself: relres = ||r|| / ||b||, two sums of the
same n squares in different orders, is 1 within 2 n u.
"""
import numpy as np
import pytest

from paper_2112_02377_gb300 import jacobi as J
from paper_2112_02377_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _context(kind, n):
    if kind == "split":
        return W.laplace7(9), J.jac_setup_local(729, W.cell_box_locals("laplace7", 9, (2, 2, 2)))
    A = W.laplace7((n, 1, 1)) if kind == "band" else W.laplace7(n)
    o = J.opts(grid=A.grid, subdomains=(2, 2, 2)) if kind == "boxes" else J.opts()
    return A, J.jac_setup(A, None, J.JAC_SUBSTRUCT if kind == "boxes" else J.JAC_BANDROW, 1, o)


@pytest.mark.parametrize("kind,n", [("band", 1), ("band", 255), ("band", 256), ("band", 257), ("band", 1025),
                                    ("band", 400000), ("boxes", 7), ("boxes", 40), ("split", 9)])
def test_vectors_in_place_equal_staged_ones(kind, n):
    import torch
    A, ctx = _context(kind, n)
    rng = np.random.default_rng(n)
    b, x = rng.uniform(-1, 1, A.n), rng.uniform(-1, 1, A.n)
    b[rng.integers(0, A.n, 3)] = 0.0
    dev = lambda a: torch.from_numpy(a).cuda()
    try:
        got = []
        for bb, xx in ((b, x), (dev(b), dev(x)), (dev(np.append(0.0, b))[1:], dev(np.append(0.0, x))[1:])):
            J.jac_set_b(ctx, bb)
            J.jac_set_x(ctx)
            rel = J.jac_sweep(ctx, 1)
            assert abs(rel - (1.0 if b.any() else 0.0)) <= 2 * (A.n + 1) * U      # (b = 0: ||r|| itself)
            J.jac_set_x(ctx, xx)
            assert J.jac_stats(ctx)["k"] == 0
            J.jac_sweep(ctx, 3)
            out = torch.empty(A.n + 1, dtype=torch.float64, device="cuda")[1:]
            assert np.array_equal(J.jac_get_x(ctx, out).cpu().numpy(), J.jac_get_x(ctx))
            got.append((rel, out.cpu().numpy()))
        for rel, out in got[1:]:
            assert rel == got[0][0] and np.array_equal(out, got[0][1])
        d = A.scipy().diagonal()
        J.jac_set_x(ctx, dev(x))
        assert np.all(np.abs(J.jac_get_x(ctx) - x) <= 2 * U * np.abs(x) * (1 + 1e-15))   # one multiply, one division
        J.jac_set_b(ctx, None)                      # b = 0: the test value is ||r|| itself, 0 from x = 0
        J.jac_set_x(ctx)
        assert J.jac_sweep(ctx, 1) == 0.0 and d.size == A.n
    finally:
        J.jac_free(ctx)


def test_gradient_written_over_its_inputs():
    import torch
    A = W.convection7(9)
    rng = np.random.default_rng(2)
    lam, x = rng.uniform(-1, 1, A.n), rng.uniform(-1, 1, A.n)
    ctx = J.jac_setup(A, np.ones(A.n))
    try:
        host = J.jac_adjoint_grad(ctx, lam, x, np.empty(A.nnz))
        rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
        assert np.array_equal(host, -(lam[rows] * x[A.col]))
        for at in (0, A.nnz - A.n, A.nnz // 2):     # lambda in the output's place; x apart from it
            buf = torch.zeros(A.nnz, dtype=torch.float64, device="cuda")
            buf[at:at + A.n] = torch.from_numpy(lam).cuda()
            J.jac_adjoint_grad(ctx, buf[at:at + A.n], torch.from_numpy(x).cuda(), buf)
            assert np.array_equal(buf.cpu().numpy(), host)
        dA = torch.empty(A.nnz, dtype=torch.float64, device="cuda")
        J.jac_adjoint_grad(ctx, torch.from_numpy(lam).cuda(), torch.from_numpy(x).cuda(), dA)
        assert np.array_equal(dA.cpu().numpy(), host)
    finally:
        J.jac_free(ctx)
