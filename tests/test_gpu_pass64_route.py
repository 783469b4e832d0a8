"""Which kernels a small FP64 solve runs: at most a launch or two per chunk of
iterations up to the line (152 SMs x 8,192 entries on this chip), five per
iteration past it.  The line follows the device's SM count."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _band(N, per_row):
    """Row sums of 0.05 on a periodic band: hundreds to thousands of iterations."""
    k = np.arange(per_row)
    col = ((np.arange(N)[:, None] + k) % N).astype(np.int32)
    val = np.where(k == 0, per_row - 1 + 0.05, -1.0) * np.ones((N, 1))
    return np.arange(N + 1, dtype=np.int64) * per_row, col.ravel(), val.ravel()


@pytest.mark.parametrize("past", [False, True])
@pytest.mark.parametrize("per_row", [9, 15])
def test_route_at_the_line(lib, per_row, past):
    from paper_2107_03632_gb300 import rbffd as r

    sms = min(torch.cuda.get_device_properties(0).multi_processor_count, 160)
    N = sms * 8192 // per_row + (1 if past else 0)
    A = r.CsrMatrix(*(torch.from_numpy(x).cuda() for x in _band(N, per_row)))
    b = torch.from_numpy(np.random.default_rng(2).standard_normal(N)).cuda()
    r.rbffd_profile_read(reset=True)
    _, info = r.rbffd_solve(A, b, None, r.make_opts(tol=1e-10))
    launches = r.rbffd_profile_read(reset=True)["launches"]
    assert info["iters"] >= 20
    if past:
        assert launches >= 5 * info["iters"]
    else:
        assert launches < 2 * info["iters"]


def test_waits_for_another_stream_do_not_shorten_the_launches(lib):
    """Beside another stream's long kernels that leave no place on the SMs a
    launch waits for one of them to end, so a solve must not split into many."""
    import threading

    from fixtures import disk_nodes
    from paper_2107_03632_gb300 import rbffd as r

    xy = torch.from_numpy(np.ascontiguousarray(np.tile(disk_nodes(0.02).xy, (1, 1)))).cuda()
    idx = r.rbffd_stencils(xy, 56).repeat(12, 1)  # 12 copies of the stencils: several ms of weights
    many = xy.repeat(12, 1)
    A = r.CsrMatrix(*(torch.from_numpy(x).cuda() for x in _band(20_000, 15)))
    b = torch.from_numpy(np.random.default_rng(2).standard_normal(20_000)).cuda()
    stop, calls = threading.Event(), [0]

    def load():
        with torch.cuda.stream(torch.cuda.Stream()):
            while not stop.is_set():
                r.rbffd_weights(many, idx, 6)
                calls[0] += 1
                torch.cuda.current_stream().synchronize()

    r.rbffd_weights(many, idx, 6)  # (its modules loaded)
    r.rbffd_solve(A, b, None, r.make_opts(tol=1e-12))
    torch.cuda.synchronize()
    t = threading.Thread(target=load)
    t.start()
    try:
        while calls[0] < 2:
            pass
        with torch.cuda.stream(torch.cuda.Stream()):
            r.rbffd_profile_read(reset=True)
            before = calls[0]
            _, info = r.rbffd_solve(A, b, None, r.make_opts(tol=1e-12))
            launches = r.rbffd_profile_read(reset=True)["launches"] - 2 * (calls[0] - before)
    finally:
        stop.set()
        t.join()
    # the setup and the last residual; per pass (kept or undone) its residual,
    # one launch and one more per 512 iterations; and two where a weight call's
    # two launches fell on either side of the counting
    passes = info["outer_sweeps"] + info["restarts"]
    assert info["iters"] >= 40
    assert launches <= 4 + 2 * (passes + 1) + info["iters"] / 512, (launches, info)
