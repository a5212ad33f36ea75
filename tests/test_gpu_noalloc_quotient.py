"""x'_i = (b_i - s_i) / a_ii of the allocation-free sweep is the correctly rounded
quotient: rows that hold nothing but their diagonal give b / d, compared bit for bit
with IEEE division.  The cases a shorter algorithm gets wrong are quotients next to a
midpoint of two doubles: for an odd 53-bit integer d and a small odd m, the integer
Q with Q d = -m (mod 2^53) makes t = (Q d + m) / 2^53 an integer whose quotient by d
lies m / (2 d) of an ulp from the midpoint Q / 2.
"""
import numpy as np
import pytest

from paper_2112_02377_gb300 import jacobi as J

pytestmark = pytest.mark.gpu


def _near_midpoints(rng, count):
    t, d = [], []
    while len(t) < count:
        dd = int(rng.integers(1 << 52, 1 << 53)) | 1
        inv = pow(dd, -1, 1 << 53)
        for m in (1, -1, 3, -3):
            Q = ((-m * inv) % (1 << 53)) | (1 << 53)
            tt = Q * dd + m
            assert tt % (1 << 53) == 0
            tt >>= 53
            if (1 << 52) <= tt < (1 << 53):
                t.append(tt)
                d.append(dd)
    return np.array(t[:count], dtype=np.float64), np.array(d[:count], dtype=np.float64)


def _signed(rng, v):
    return v * rng.choice([-1.0, 1.0], v.size)


def _cases(name):
    rng = np.random.default_rng(3)
    n = 20000
    if name == "midpoints":                       # over the whole range of the short form
        t, d = _near_midpoints(rng, n)
        return _signed(rng, np.ldexp(t, rng.integers(-870, 720, n))), _signed(rng, np.ldexp(d, rng.integers(-150, 48, n)))
    if name == "random":
        m = lambda: 1.0 + rng.random(n)
        return _signed(rng, np.ldexp(m(), rng.integers(-823, 778, n))), _signed(rng, np.ldexp(m(), rng.integers(-100, 101, n)))
    if name == "ends":                            # one step inside and outside the short form's exponents
        et, ed = np.meshgrid([-1022, -900, -825, -824, -823, -822, 776, 777, 778, 779, 900], [-102, -101, -100, -99, 99, 100, 101, 102])
        t, d = np.ldexp(1.0 + rng.random(et.size), et.ravel()), np.ldexp(1.0 + rng.random(et.size), ed.ravel())
        keep = np.abs(np.log2(t) - np.log2(d)) < 1000      # an overflow is reported as NaN
        return t[keep], d[keep]
    if name == "powers":                          # quotients at and next to a power of two
        z = np.nextafter(1.0, rng.choice([0.0, 1.0, 2.0], n))
        d = 1.0 + rng.random(n)
        return np.nextafter(z * d, rng.choice([0.0, 4.0], n)), d
    if name == "small":                           # integers, zeros among them
        t, d = np.meshgrid(np.arange(-60, 61) * 0.125, np.arange(1, 80).astype(np.float64))
        return t.ravel(), d.ravel()


@pytest.mark.parametrize("name", ["midpoints", "random", "ends", "powers", "small"])
def test_the_quotient_is_the_division(name):
    import torch
    t, d = _cases(name)
    n = t.size
    ptr = torch.arange(n + 1, dtype=torch.int32, device="cuda")
    col = torch.arange(n, dtype=torch.int32, device="cuda")
    val, b = torch.from_numpy(d).cuda(), torch.from_numpy(t).cuda()
    with np.errstate(all="ignore"):
        want = t / d
    for k in (1, 2):                              # the last sweep's kernel, and both
        out = torch.empty(n, dtype=torch.float64, device="cuda")
        try:
            J.jac_sweep_noalloc(ptr, col, val, b, torch.zeros_like(b), out, k)
        except J.JacobiError as e:                # the sums of the largest t overflow; x_out is written all the same
            assert e.status == J.JAC_ENUMERIC
        got = out.cpu().numpy()
        assert np.array_equal(got.view(np.int64), want.view(np.int64)), int((got != want).sum())
