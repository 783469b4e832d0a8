"""Accuracy of the refined FP64 weight solve against that of the FP64
elimination of every stencil (RBFFD_WEIGHTS=ns64), both measured against
weights in 180-bit fixed point.

The refined solve's residual is formed from kernel values known to 2^-54 of
their range and monomials to 2^-59 and summed exactly, the elimination rounds
every entry and operation to 2^-53 of its size.  So over the sampled rows of
an even or evenly stretched set neither the largest nor the median error may
be above the elimination's, from n = s + 1 to three times s."""

import math
from fractions import Fraction

import numpy as np
import pytest
import torch
from scipy.linalg import lu_factor, lu_solve

from fixtures import disk_nodes

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
BITS = 180


def exact_weights(pts, centre, m):
    """Laplacian weights of one stencil as (integers, exponent): w_j = int_j 2^exponent.

    The coordinates are scaled by a power of two, so the system's entries are
    the given doubles' to 2^-180; its double-precision LU refines the solution."""
    d = pts - centre  # (rounded as the solver rounds it)
    k = -math.frexp(np.abs(d).max())[1]
    X = [[int(Fraction(v) * Fraction(2) ** (k + BITS)) for v in p] for p in d.tolist()]
    ex = [(a - i, i) for a in range(m + 1) for i in range(a + 1)]
    n, s = len(X), len(ex)
    A = np.zeros((n + s, n + s), object)
    b = np.zeros(n + s, object)

    def radius(x, y):  # 2^BITS |(x, y)|
        return math.isqrt(x * x + y * y)

    for i, (x, y) in enumerate(X):
        for j in range(i):
            r = radius(x - X[j][0], y - X[j][1])
            A[i, j] = A[j, i] = r * r * r >> 2 * BITS
        px, py = [1 << BITS], [1 << BITS]
        for _ in range(m):
            px.append(px[-1] * x >> BITS)
            py.append(py[-1] * y >> BITS)
        for c, (u, v) in enumerate(ex):
            A[i, n + c] = A[n + c, i] = px[u] * py[v] >> BITS
        b[i] = 9 * radius(x, y)
    for c, e in enumerate(ex):
        b[n + c] = (2 << BITS) if e in ((2, 0), (0, 2)) else 0
    b = np.array([v << BITS for v in b], object)
    to_float = lambda v, bits: np.array([math.ldexp(float(t >> max(t.bit_length() - 60, 0)),
                                                    max(t.bit_length() - 60, 0) - bits) for t in v])
    lu = lu_factor(np.array([to_float(row, BITS) for row in A]))
    x = np.zeros(n + s, object)
    for _ in range(40):
        dx = lu_solve(lu, to_float(b - A.dot(x), 2 * BITS))
        x = x + np.array([int(Fraction(v) * 2 ** BITS) for v in dx], object)
        if np.abs(dx).max() <= 1e-26 * np.abs(to_float(x, BITS)).max():
            return x[:n], 2 * k - BITS
    raise AssertionError("no convergence of the reference")


def error(w, exact):
    """max |w - exact| / max |exact| of one stencil."""
    x = [Fraction(t) * Fraction(2) ** exact[1] for t in exact[0]]
    return float(max(abs(Fraction(v) - t) for v, t in zip(w.tolist(), x)) / max(abs(t) for t in x))


@pytest.mark.parametrize("m,n", [(1, 9), (2, 7), (2, 12), (3, 11), (4, 16), (4, 30), (4, 45), (5, 22), (6, 29), (6, 34),
                                 (6, 56)])
@pytest.mark.parametrize("stretch", [1.0, 4.0])
def test_refined_at_least_as_accurate_as_the_elimination(lib, monkeypatch, m, n, stretch):
    from paper_2107_03632_gb300 import rbffd

    pts = disk_nodes(0.08).xy * np.array([1.0, 1.0 / stretch])
    xy = torch.from_numpy(pts).to(DEV)
    idx = rbffd.rbffd_stencils(xy, n)
    w, st = rbffd.rbffd_weights(xy, idx, m)
    monkeypatch.setenv("RBFFD_WEIGHTS", "ns64")
    w64, st64 = rbffd.rbffd_weights(xy, idx, m)
    assert torch.equal(st, st64)
    rows = torch.nonzero((w != w64).any(dim=1) & (st == 0))[:, 0].cpu().numpy()
    rows = rows[:: max(1, len(rows) // 24)][:24]
    assert len(rows) >= 20  # (refined ones)
    idx, w, w64 = idx.cpu().numpy(), w.cpu().numpy(), w64.cpu().numpy()
    exact = [exact_weights(pts[idx[i]], pts[i], m) for i in rows]
    got = np.array([error(w[i], e) for i, e in zip(rows, exact)])
    elim = np.array([error(w64[i], e) for i, e in zip(rows, exact)])
    assert got.max() <= elim.max() and np.median(got) <= np.median(elim), (got, elim)
