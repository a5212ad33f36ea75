"""The resident kernel (matrix kept in shared memory, one CTA per SM) against the
pipelined kernel, which the same context runs with a pinned geometry: iterates,
counts and stopping sweeps bit for bit, at the row counts where its slices and
CTA ranges end, around its launch length (512 sweeps), in both lane counts, from
rows of one entry to a matrix near the capacity limit and one past it.

Test values: both kernels add the same n squares, in different orders, so each
sum carries at most n roundings of it: relative difference <= 2 n u.
"""
import numpy as np
import pytest

from paper_2112_02377_gb300 import jacobi as J
from paper_2112_02377_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _matrix(name):
    if name.startswith("line"):
        return W.laplace7((int(name[4:]), 1, 1))
    return {"lap": lambda: W.laplace7((19, 17, 13)), "diff": lambda: W.diffusion7((41, 40, 39), seed=3),
            "fe": lambda: W.fe27_deleted(17, seed=2), "q1": lambda: W.q1_laplace(20)[0],
            "irregular": lambda: W.random_irregular(900, seed=5, long_rows=0),
            "large": lambda: W.laplace7((71, 70, 69)), "too_large": lambda: W.laplace7((80, 80, 80))}[name]()


def _pair(A, b, split="bandrow", nparts=3, **kw):
    lanes = kw.pop("lanes_per_row", 0)
    nparts = min(nparts, A.n)
    a = J.Solver(A, b, split, nparts, lanes_per_row=lanes, **kw)
    L = a.stats()["lanes_per_row"]
    return a, J.Solver(A, b, split, nparts, variant=2, ctas_per_sm=2, lanes_per_row=L, **kw)


def _same(a, p, n):
    assert np.array_equal(a.x(), p.x())
    sa, sp = a.stats(), p.stats()
    assert sa["k"] == sp["k"] and sa["sweeps_total"] == sp["sweeps_total"]
    assert sa["last_resinf"] == sp["last_resinf"]
    assert abs(sa["last_relres"] - sp["last_relres"]) <= 2 * n * U * sp["last_relres"]


@pytest.mark.parametrize("name", ["line1", "line31", "line33", "line152", "line4863", "line4865", "lap", "diff", "fe",
                                  "q1", "irregular", "large", "too_large"])
def test_resident_sweeps_are_the_pipelined_ones(name):
    A = _matrix(name)
    b = np.random.default_rng(1).uniform(-1, 1, A.n)
    a, p = _pair(A, b, history=64)
    with a, p:
        assert (a.stats()["ctas_per_sm"] == 1) == (name != "too_large")
        for k in (1, 2, 3, 40):
            ra, rp = a.sweep(k), p.sweep(k)
            _same(a, p, A.n)
            ha, hp = a.history(), p.history()
            assert len(ha) == len(hp) == k
            assert np.all(np.abs(ha - hp) <= 2 * A.n * U * hp) and ra == ha[-1] and rp == hp[-1]


@pytest.mark.parametrize("k", [511, 512, 513, 1025])
def test_resident_launch_boundaries(k):
    A = _matrix("lap")
    b = np.random.default_rng(2).uniform(-1, 1, A.n)
    a, p = _pair(A, b)
    with a, p:
        a.sweep(k), p.sweep(k)
        _same(a, p, A.n)


@pytest.mark.parametrize("name,split,norm,lanes", [("lap", "bandrow_nnz", 2, 0), ("lap", "substruct", 0, 2),
                                                   ("fe", "substruct", 2, 0), ("q1", "bandrow", 0, 1)])
def test_resident_solves_stop_at_the_same_sweep(name, split, norm, lanes):
    A = _matrix(name)
    b = np.random.default_rng(3).uniform(-1, 1, A.n)
    a, p = _pair(A, b, split, lanes_per_row=lanes, norm=norm, history=4096,
                 **(dict(subdomains=(2, 2, 2)) if split == "substruct" else {}))
    with a, p:
        scale = np.abs(b).max() if norm == 0 else 1.0
        for tol in (0.5, 1e-3, 1e-9):               # within the first sweeps; mid-launch; over several launches
            a.set_x(), p.set_x()
            ka, kp = a.solve(tol * scale, 20000), p.solve(tol * scale, 20000)
            assert ka[0] == kp[0] and ka[2] == kp[2] == J.JAC_OK
            _same(a, p, A.n)
            assert len(a.history()) == len(p.history()) == min(ka[0] + 1, 4096)
        for maxit in (0, 1, 2, 3, 513):             # the limit ends the run at every distance from a launch's end
            a.set_x(), p.set_x()
            ka, kp = a.solve(0.0, maxit), p.solve(0.0, maxit)
            assert ka[0] == kp[0] == maxit and ka[2] == kp[2] == J.JAC_ENOTCONV
            _same(a, p, A.n)


@pytest.mark.parametrize("name,split,parts,lanes", [("line33", "bandrow", 33, 0), ("lap", "bandrow_nnz", 200, 0),
                                                    ("lap", "substruct", (3, 3, 2), 2), ("q1", "substruct", (2, 2, 2), 0),
                                                    ("diff", "bandrow", 1, 1), ("fe", "bandrow", 64, 0)])
def test_resident_local_stop_is_the_pipelined_one(name, split, parts, lanes):
    """Stopping on local convergence (integer maxima: nothing here may differ)."""
    A = _matrix(name)
    b = np.random.default_rng(6).uniform(-1, 1, A.n)
    kw = dict(subdomains=parts) if split == "substruct" else dict(nparts=parts)
    a, p = _pair(A, b, split, lanes_per_row=lanes, norm=0, stop=J.JAC_STOP_LOCAL, history=4096, **kw)
    zero_part = np.where(np.arange(A.n) < A.n // 2, b, 0.0)     # a partition that passes at once, where there are several

    def check(tol, maxit):
        ka, kp = a.solve(tol, maxit), p.solve(tol, maxit)
        assert ka == kp
        _same(a, p, A.n)
        sa, sp = a.stats(), p.stats()
        assert sa["stop_part"] == sp["stop_part"] and sa["stop_local"] == sp["stop_local"]
        assert np.array_equal(a.history(), p.history())
        return ka[2]

    with a, p:
        assert a.stats()["ctas_per_sm"] == 1
        for tol in (0.5, 1e-2, 1e-5, 1e-9):
            a.set_x(), p.set_x()
            assert check(tol, 20000) == J.JAC_OK
            assert check(tol, 20000) == J.JAC_OK    # the returned iterate passes again
            assert check(tol / 2, 20000) == J.JAC_OK    # and the solve goes on from it
        for maxit in (0, 1, 2, 3, 513):
            a.set_x(), p.set_x()
            assert check(0.0, maxit) == J.JAC_ENOTCONV or maxit > 3     # (a residual may become exactly 0)
        a.set_b(zero_part), p.set_b(zero_part)
        a.set_x(), p.set_x()
        assert check(1e-5, 20000) == J.JAC_OK
        assert a.sweep(7) == p.sweep(7)             # sweeps without a test raise the maxima too
        a.set_x(), p.set_x()
        assert check(1e-7, 20000) == J.JAC_OK


def test_resident_reports_divergence_and_a_missing_cta():
    rng = np.random.default_rng(4)
    M = rng.uniform(-1, 1, (40, 40))
    np.fill_diagonal(M, 0.05)
    with J.Solver(W.dense_to_csr(M), np.ones(40)) as s:
        with pytest.raises(J.JacobiError) as e:
            s.sweep(20000)
        assert e.value.status == J.JAC_ENUMERIC
    A = _matrix("lap")
    with J.Solver(A, np.ones(A.n), fault_skip_cta=1, timeout_cycles=20_000_000) as s:
        with pytest.raises(J.JacobiError) as e:
            s.sweep(5)
        assert e.value.status == J.JAC_ETIMEOUT


def test_contexts_of_one_kernel_and_different_sizes_live_together():
    big, small = _matrix("large"), _matrix("line33")
    with J.Solver(big, np.ones(big.n)) as a, J.Solver(small, np.ones(small.n)) as c:
        c.sweep(2)
        a.sweep(2)                                  # the larger one's first launch, after the smaller one's set-up
        assert a.stats()["k"] == c.stats()["k"] == 2
