"""Whole BiCGSTAB iterations in one launch (small FP64 systems without
multigrid) against the separate kernels, which the profiling switch selects:
one row, fewer rows than a block's share, one block more than full shares,
rows of 400 entries (more than a block holds in shared memory), and a system
just past the line.  Both must meet the tolerance; the solutions then differ
by at most 2 tol |A^-1| |b|: the systems are diagonally dominant by a factor
of 2 with |A^-1| <= 2 / min |a_ii|."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _system(N, per_row, seed):
    rng = np.random.default_rng(seed)
    k = min(per_row, N)
    col = np.empty((N, k), np.int32)
    col[:, 0] = np.arange(N)
    if k > 1:  # distinct columns, away from the diagonal
        step = rng.integers(1, N, (N, 1)) if N <= k else 1 + rng.integers(0, max(1, (N - 1) // (k - 1)), (N, 1))
        col[:, 1:] = (np.arange(N)[:, None] + step * np.arange(1, k)) % N
    val = rng.standard_normal((N, k))
    off = np.abs(val[:, 1:]).sum(axis=1)
    val[:, 0] = (2.0 * off + 1.0) * np.where(rng.random(N) < 0.5, -1.0, 1.0)
    rp = np.arange(N + 1, dtype=np.int64) * k
    return rp, col.reshape(-1), val.reshape(-1), rng.standard_normal(N)


@pytest.mark.parametrize("N,per_row", [(1, 1), (31, 5), (33, 9), (152 * 32 + 1, 15), (10_007, 15), (700, 400),
                                       (83_000, 15), (84_000, 15)])
@pytest.mark.parametrize("jacobi", [True, False])
def test_matches_separate_kernels(N, per_row, jacobi):
    from paper_2107_03632_gb300 import rbffd as r

    rp, col, val, b = _system(N, per_row, N + per_row)
    dev = lambda a: torch.from_numpy(a).cuda()
    A = r.CsrMatrix(dev(rp), dev(col), dev(val))
    tol = 1e-10
    opts = r.make_opts(tol=tol, jacobi=jacobi)
    x, info = r.rbffd_solve(A, dev(b), None, opts)
    r.rbffd_profile_enable(True)
    try:
        y, ref = r.rbffd_solve(A, dev(b), None, opts)
    finally:
        r.rbffd_profile_enable(False)
        r.rbffd_profile_read(reset=True)
    assert info["status_code"] == 0 and ref["status_code"] == 0
    x, y = x.cpu().numpy(), y.cpu().numpy()
    for z in (x, y):
        res = b - np.add.reduceat(val * z[col], rp[:-1])
        assert np.linalg.norm(res) <= 1.01 * tol * np.linalg.norm(b)
    diag = np.abs(val.reshape(N, -1)[:, 0]).min()
    assert np.abs(x - y).max() <= 2 * tol * (2.0 / diag) * np.linalg.norm(b)


@pytest.mark.parametrize("budget", [1, 2, 7])
def test_iteration_budget(budget):
    from paper_2107_03632_gb300 import rbffd as r

    rp, col, val, b = _system(5_000, 15, 3)
    dev = lambda a: torch.from_numpy(a).cuda()
    A = r.CsrMatrix(dev(rp), dev(col), dev(val))
    _, info = r.rbffd_solve(A, dev(b), None, r.make_opts(tol=1e-300, max_iter=budget), raise_on_error=False)
    assert info["iters"] <= budget and info["status_code"] != 0


def test_repeats_bit_for_bit():
    """A stale or early read of another block's values would show as a
    difference between runs."""
    from paper_2107_03632_gb300 import rbffd as r

    rp, col, val, b = _system(10_007, 15, 9)
    dev = lambda a: torch.from_numpy(a).cuda()
    A = r.CsrMatrix(dev(rp), dev(col), dev(val))
    bd = dev(b)
    opts = r.make_opts(tol=1e-13)
    x0, i0 = r.rbffd_solve(A, bd, None, opts)
    for _ in range(50):
        x, i = r.rbffd_solve(A, bd, None, opts)
        assert i["iters"] == i0["iters"] and torch.equal(x, x0)


def test_solves_from_several_threads_and_streams():
    """Launches whose blocks wait on one another, from four streams at once."""
    import threading

    from paper_2107_03632_gb300 import rbffd as r

    dev = lambda a: torch.from_numpy(a).cuda()
    systems = []
    for seed in range(4):
        rp, col, val, b = _system(10_007, 15, 20 + seed)
        A, bd = r.CsrMatrix(dev(rp), dev(col), dev(val)), dev(b)
        x, info = r.rbffd_solve(A, bd, None, r.make_opts(tol=1e-13))
        systems.append((A, bd, x, info["iters"]))
    torch.cuda.synchronize()
    wrong = []

    def work(A, bd, x0, iters):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(25):
                x, info = r.rbffd_solve(A, bd, None, r.make_opts(tol=1e-13))
                torch.cuda.current_stream().synchronize()
                if info["iters"] != iters or not torch.equal(x, x0):
                    wrong.append((info["iters"], iters))

    threads = [threading.Thread(target=work, args=s) for s in systems]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
