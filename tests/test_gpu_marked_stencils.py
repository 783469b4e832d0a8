"""The FP64 eliminations: of the stencils that the refined solve leaves, and of
every stencil at n > 64, in all their group sizes (a quarter, half, one, two,
four warps per stencil)."""

import numpy as np
import pytest
import torch

import oracle
from fixtures import disk_nodes, splitmix64, uniform01

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

FORMS = [("null-space", 1), ("null-space", 4), ("null-space-2warp", 2), ("null-space-4warp", 4), ("null-space-half", 1),
         ("null-space-half", 3), ("null-space-quarter", 1), ("null-space-quarter", 4)]


def _graded(N, power):
    """Spacing ratios that leave float32 no digits: all or most stencils are left."""
    u = uniform01(splitmix64(11, 2 * N)).reshape(N, 2) - 0.5
    return np.ascontiguousarray(np.sign(u) * (2.0 * np.abs(u)) ** power)


def _each_form(rbffd, xy, idx, m):
    """Weights and status of every form that fits in shared memory."""
    n = idx.shape[1]
    out = []
    try:
        for kernel, wpb in FORMS:
            try:
                rbffd.set_weights_config(n, m, kernel, wpb)
            except rbffd.RbffdError:
                continue
            out.append((kernel, wpb, *rbffd.rbffd_weights(xy, idx, m)))
    finally:
        rbffd.set_weights_config(n, m, None)
    return out


@pytest.mark.parametrize("m,n", [(1, 9), (2, 12), (3, 20), (4, 30), (5, 42), (6, 56)])
@pytest.mark.parametrize("N,power", [(40, 9), (67, 9), (1500, 5), (1500, 2)])
def test_left_stencils_in_every_form(lib, monkeypatch, m, n, N, power):
    """Sets that leave all, most or a part of their stencils, from a few groups'
    shares on: each form solves every one (no mark stays), with the same bits,
    and where a row differs from the elimination of all stencils it was refined."""
    from paper_2107_03632_gb300 import rbffd

    if n > N:
        pytest.skip("more nodes per stencil than nodes")
    xy = torch.from_numpy(_graded(N, power)).to(DEV)
    idx = rbffd.rbffd_stencils(xy, n)
    forms = _each_form(rbffd, xy, idx, m)
    assert len(forms) >= 4
    for kernel, wpb, w, st in forms:
        assert torch.isfinite(w).all(), (kernel, wpb)
        assert torch.equal(w, forms[0][2]) and torch.equal(st, forms[0][3]), (kernel, wpb)
    monkeypatch.setenv("RBFFD_WEIGHTS", "ns64")
    w64, st64 = rbffd.rbffd_weights(xy, idx, m)
    assert torch.equal(st64, forms[0][3])
    same = (w64 == forms[0][2]).all(dim=1)
    if power == 9:
        assert int(same.sum()) > 0  # (some were left)


@pytest.mark.parametrize("m,n", [(1, 65), (2, 66), (4, 80), (6, 90)])
def test_large_supports_in_every_form(lib, m, n):
    from paper_2107_03632_gb300 import rbffd

    d = disk_nodes(0.1)
    idx_ref = oracle.knn(d.xy, n)
    w_ref, _ = oracle.weights(d.xy, idx_ref, m)
    forms = _each_form(rbffd, torch.from_numpy(d.xy).to(DEV), torch.from_numpy(idx_ref).to(DEV), m)
    assert len(forms) >= 5
    bar = 1e-9 if m <= 4 else 1e-7
    for kernel, wpb, w, st in forms:
        assert int(st.sum()) == 0 and torch.equal(w, forms[0][2]), (kernel, wpb)
    w = forms[0][2].cpu().numpy()
    assert (np.abs(w - w_ref).max(axis=1) / np.abs(w_ref).max(axis=1)).max() <= bar


def test_left_stencils_are_shared_out(lib, monkeypatch):
    """A small set that leaves every stencil: the time of the attempt and of one
    elimination of all, not of 32 in a row.  The attempt costs less than the
    elimination and the default form less than one warp per stencil: at most
    twice RBFFD_WEIGHTS=ns64; three times leaves room for noise (one warp per 32
    consecutive stencils took 13 times)."""
    from paper_2107_03632_gb300 import rbffd

    xy = torch.from_numpy(_graded(2000, 5)).to(DEV)
    idx = rbffd.rbffd_stencils(xy, 56)

    def ms():
        out = []
        for _ in range(7):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            rbffd.rbffd_weights(xy, idx, 6)
            e1.record()
            torch.cuda.synchronize()
            out.append(e0.elapsed_time(e1))
        return sorted(out)[3]

    both = ms()
    monkeypatch.setenv("RBFFD_WEIGHTS", "ns64")
    assert both <= 3.0 * ms()
