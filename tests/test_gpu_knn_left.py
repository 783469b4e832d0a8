"""Queries that the fixed-point search leaves to the list search in sets large
enough that a warp looks at several (32,768 queries on): rows against brute
force, and the time of a set that leaves many."""

import math

import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _disk(N, power):
    """About N points of a jittered grid disk at radius r^power: crowded towards the centre."""
    g = torch.Generator(device=DEV)
    g.manual_seed(4)
    h = math.sqrt(math.pi / N)
    k = math.ceil(1.0 / h)
    a = torch.arange(-k, k + 1, device=DEV, dtype=torch.float64) * h
    j = (2.0 * torch.rand((2 * k + 1, 2 * k + 1, 2), generator=g, device=DEV, dtype=torch.float64) - 1.0) * 0.25 * h
    p = torch.stack([a[None, :] + j[..., 0], a[:, None] + j[..., 1]], dim=-1)
    p = p[a[None, :] ** 2 + a[:, None] ** 2 < 1.0]
    return (p * p.norm(dim=1, keepdim=True) ** (power - 1.0)).contiguous()


def _brute(xy, rows, n):
    out = []
    for q in rows.split(64):
        dx = xy[None, :, 0] - xy[q, None, 0]
        dy = xy[None, :, 1] - xy[q, None, 1]
        dx, dy = dx * dx, dy * dy  # (rounded one by one)
        out.append(torch.sort(dx + dy, dim=1, stable=True).indices[:, :n])
    return torch.cat(out).int()


@pytest.mark.parametrize("N,power,n", [(32_900, 4.0, 12), (66_000, 3.0, 45), (131_072, 2.0, 112), (600_001, 3.0, 6)])
def test_left_queries_of_large_sets(lib, N, power, n):
    from paper_2107_03632_gb300 import rbffd

    xy = _disk(N, power)
    idx = rbffd.rbffd_stencils(xy, n)
    assert int(idx.min()) >= 0 and int(idx.max()) < len(xy)
    assert torch.equal(idx[:, 0], torch.arange(len(xy), device=DEV, dtype=torch.int32))
    g = torch.Generator(device=DEV)
    g.manual_seed(1)
    near = torch.argsort((xy * xy).sum(dim=1))[:128]  # the crowded centre, and rows anywhere
    rows = torch.cat([near, torch.randint(len(xy), (128,), generator=g, device=DEV),
                      torch.tensor([0, len(xy) - 1], device=DEV)])
    assert torch.equal(idx[rows], _brute(xy, rows, n))


def test_left_queries_are_shared_out(lib):
    """The crowded half of the queries is left.  It takes the list search alone
    about twice the time of the even set's search of all, so three times in all;
    with neighbouring queries, which are left together, in one warp it took 5.5."""
    from paper_2107_03632_gb300 import rbffd

    def ms(xy):
        out = []
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            rbffd.rbffd_stencils(xy, 45)
            e1.record()
            torch.cuda.synchronize()
            out.append(e0.elapsed_time(e1))
        return sorted(out)[2]

    assert ms(_disk(1_000_000, 2.0)) <= 3.0 * ms(_disk(1_000_000, 1.0))
