"""The explicit residual in 128-bit integers, against exact rational
arithmetic: the solver's relative residual of a given x without iterations.

b is A x rounded to double, so a residual entry is only the rounding of b
(2^-53 of it) and an error of 2^-80 of a row's products would be seen.  Rows of
0 to 70 entries with zeros, subnormals, wide exponent ranges and cancellation;
one row of 20,000 entries, which the floating-point form takes (with its
warp).  Tolerance: the residual carries at most 2^-96 of a row's largest
product per entry, the norms 1e-15 per addition over 2,000 rows in a tree:
1e-12 of the exact value."""

import math
from fractions import Fraction

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _system(mean, long_row, seed):
    rng = np.random.default_rng(seed)
    N = 2003
    x = rng.standard_normal(N) * 2.0 ** rng.integers(-40, 41, N)
    x[::17] = 0.0
    x[5::101] = 5e-324
    cols, vals, rp = [], [], [0]
    for i in range(N):
        k = int(rng.integers(0, 2 * mean + 1))
        if long_row and i == 777:
            k = 20_000
        c = rng.integers(0, N, k).astype(np.int32)
        v = rng.standard_normal(k) * 2.0 ** rng.integers(-40, 41, k)
        if k > 4:
            v[0] = 0.0
            c[2], v[2] = c[1], -v[1]  # cancels
            v[3] = -5e-324 if i % 3 else v[3]
        cols.append(c)
        vals.append(v)
        rp.append(rp[-1] + k)
    rp, col, val = np.array(rp, np.int64), np.concatenate(cols), np.concatenate(vals)
    b = np.zeros(N)
    r2 = b2 = Fraction(0)
    for i in range(N):
        s = sum((Fraction(float(v)) * Fraction(float(x[c])) for c, v in zip(cols[i], vals[i])), Fraction(0))
        b[i] = float(s)
        r = Fraction(float(b[i])) - s
        r2 += r * r
        b2 += Fraction(float(b[i])) ** 2
    return N, rp, col, val, x, b, math.sqrt(r2 / b2)


@pytest.mark.parametrize("mean,long_row", [(3, False), (20, False), (20, True), (56, False)])
def test_residual_matches_exact(mean, long_row):
    from paper_2107_03632_gb300 import rbffd as r

    N, rp, col, val, x, b, want = _system(mean, long_row, 11 + mean)
    dev = lambda a: torch.from_numpy(a).cuda()
    A = r.CsrMatrix(dev(rp), dev(col), dev(val))
    opts = r.make_opts(tol=1e-300, max_iter=0, jacobi=False)
    _, info = r.rbffd_solve(A, dev(b), dev(x), opts, raise_on_error=False)
    assert want > 1e-20
    assert abs(info["rel_residual"] - want) <= 1e-12 * want, (info["rel_residual"], want)


@pytest.mark.parametrize("bad", [math.inf, -math.inf, math.nan])
def test_non_finite_stays_non_finite(bad):
    from paper_2107_03632_gb300 import rbffd as r

    N, rp, col, val, x, b, _ = _system(20, False, 5)
    x[col[100]] = bad
    val[100] = 1.0
    dev = lambda a: torch.from_numpy(a).cuda()
    A = r.CsrMatrix(dev(rp), dev(col), dev(val))
    opts = r.make_opts(tol=1e-300, max_iter=0, jacobi=False)
    _, info = r.rbffd_solve(A, dev(b), dev(x), opts, raise_on_error=False)
    assert not math.isfinite(info["rel_residual"])
