"""Kernels whose dynamic shared memory depends on the call, launched by several
threads with different sizes: no valid call fails, and every result has the
bits of the call alone.  Weights: pairs of (n, m) that share a kernel (the
refined solve of one degree, and the elimination of what it leaves; n > 64:
the elimination alone).  Solves: systems whose rows per block differ."""

import threading

import numpy as np
import pytest
import torch

from fixtures import disk_nodes

pytestmark = pytest.mark.gpu


def _run(jobs, repeats, burst):
    """Each job () -> tensors from its own thread and stream, `repeats` bursts of calls."""
    alone = [job() for job in jobs]
    torch.cuda.synchronize()
    wrong = []

    def work(job, ref):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(repeats):
                    for _ in range(burst):
                        got = job()
                    torch.cuda.current_stream().synchronize()
                    if not all(torch.equal(a, b) for a, b in zip(got, ref)):
                        wrong.append("bits")
        except Exception as e:
            wrong.append(str(e))

    threads = [threading.Thread(target=work, args=a) for a in zip(jobs, alone) for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong[:3]


@pytest.mark.parametrize("a,b", [((6, 28), (6, 64)), ((2, 12), (6, 56)), ((5, 70), (6, 100)), ((0, 7), (0, 40))])
def test_weights_of_two_sizes_from_several_threads(lib, a, b):
    from paper_2107_03632_gb300 import rbffd

    xy = torch.from_numpy(disk_nodes(0.1).xy).cuda()
    jobs = []
    for m, n in (a, b):
        idx = rbffd.rbffd_stencils(xy, n)
        jobs.append(lambda m=m, idx=idx: rbffd.rbffd_weights(xy, idx, m))
    _run(jobs, 40, 150)


def test_one_launch_solves_of_two_sizes_from_several_threads(lib):
    from paper_2107_03632_gb300 import rbffd as r

    jobs = []
    for N in (900, 60_000):
        k = np.arange(5)
        col = ((np.arange(N)[:, None] + k * 7) % N).astype(np.int32)
        val = np.where(k == 0, 9.0, -1.0) * np.ones((N, 1))
        A = r.CsrMatrix(*(torch.from_numpy(x).cuda() for x in (np.arange(N + 1, dtype=np.int64) * 5, col.ravel(),
                                                               val.ravel())))
        b = torch.from_numpy(np.random.default_rng(N).standard_normal(N)).cuda()
        jobs.append(lambda A=A, b=b: (r.rbffd_solve(A, b, None, r.make_opts(tol=1e-12))[0],))
    _run(jobs, 40, 1)
