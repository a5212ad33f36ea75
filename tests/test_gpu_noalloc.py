"""The allocation-free sweep's staged kernel at the sizes where its blocks and
rounds end: n around multiples of 256 rows, blocks of more entries than one
staged round (7 per row), rows longer than a round, the diagonal anywhere in a
row, arrays with no more than their types' alignment, a CSR whose rowptr
starts past zero, and the ends of the quotient's fast range; against the CPU
oracle's sweeps.

Tolerance, from the rounding of one sweep: each side sums len_i terms and
divides, so x'_i carries at most (len_i + 3) roundings of the row's magnitude
scale_i = (|b_i| + sum_j |a_ij x_j|) / |a_ii|; both sides together
2 (len_i + 3) u scale_i, doubled here for the second-order terms.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2112_02377_gb300 import jacobi as J
from paper_2112_02377_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _laplace_rows(n):
    """n rows of a tridiagonal operator."""
    A = W.laplace7((n, 1, 1))
    return A


@pytest.mark.parametrize("name", ["n1", "n255", "n256", "n257", "n513", "fe27", "irregular", "long_row", "offset", "scale-300",
                                  "scale-101", "scale99", "scale300", "zeros"])
def test_noalloc_staged_rounds(name):
    import torch
    if name[0] == "n":
        A = _laplace_rows(int(name[1:]))
    elif name == "fe27":
        A = W.fe27_deleted(12, seed=5)            # 27-entry rows: four rounds a block
    elif name == "irregular":
        A = W.random_irregular(700, seed=3, long_rows=2, long_len=600)
    elif name == "long_row":
        A = W.random_irregular(5000, seed=4, long_rows=1, long_len=4000)   # a row of three rounds
    else:
        A = W.diffusion7((11, 10, 9), seed=6)
    rng = np.random.default_rng(11)
    if name.startswith("scale"):                   # diagonals inside and outside the quotient's fast range
        A.val[:] = A.val * 2.0 ** int(name[5:])
    b, x0 = rng.uniform(-1, 1, A.n), rng.uniform(-1, 1, A.n)
    rp, cl, vl = A.rowptr.copy(), A.col, A.val
    if name.startswith("scale"):
        b = b * 2.0 ** int(name[5:])
    if name == "zeros":                            # rows whose b_i - s_i is zero
        b[::3], x0[:] = 0.0, 0.0
    shift = 3 if name == "offset" else 0
    if shift:                                      # entries before the first row, and 8 / 4-byte aligned arrays
        rp = rp + shift
        cl, vl = np.concatenate([np.zeros(shift, np.int32), cl]), np.concatenate([np.zeros(shift), vl])

    def dev(a):
        t = torch.empty(len(a) + 1, dtype=torch.from_numpy(a[:1]).dtype, device="cuda")
        t[1:] = torch.from_numpy(np.ascontiguousarray(a)).cuda()
        return t[1:]                               # one element past the allocation's alignment

    drp, dcl, dvl, db, dx = (dev(v) for v in (rp, cl, vl, b, x0))
    Mo, S = O.prepare(A), abs(A.scipy())
    d = np.abs(A.scipy().diagonal())
    lens = np.diff(A.rowptr)
    x = x0
    for k in (1, 2):                               # the last sweep alone, and after one that keeps no sums
        out = dev(np.zeros(A.n))
        rel = J.jac_sweep_noalloc(drp, dcl, dvl, db, dx, out, k)
        y, bound = x0, np.zeros(A.n)
        for _ in range(k):
            prev, pb = y, bound
            mag = np.abs(b) + S @ np.abs(prev) - d * np.abs(prev)
            bound = 4 * (lens + 3) * U * mag / d + (S @ pb - d * pb) / d
            y, ss, _ = O.sweep(Mo, b, prev)
        err = np.abs(out.cpu().numpy() - y)
        assert np.all(err <= bound), float(np.max(err / (bound + 1e-300)))
        # the test value: r_i of x^{k-1}, (len_i + 3) roundings of |b| + |A||x|, and the sums' own n u
        rmag = np.abs(b) + S @ np.abs(prev)
        tol = np.linalg.norm(4 * (lens + 3) * U * rmag + S @ pb) + 2 * A.n * U * np.sqrt(ss)
        assert abs(rel - np.sqrt(ss) / np.linalg.norm(b)) * np.linalg.norm(b) <= tol + 4 * A.n * U * np.sqrt(ss)
