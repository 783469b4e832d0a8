"""The select-then-sort stencil search (n <= 112) and what it leaves to the
list search, bit-exact against the oracle's brute force: support sizes at the
edges of its candidate counts (24 / 25, 56 / 57, 112 / 113), and node sets
with ties, gradings, lines, empty cells and non-finite coordinates."""

import numpy as np
import pytest
import torch

import oracle
from fixtures import disk_nodes, splitmix64, uniform01

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _sets():
    u = uniform01(splitmix64(3, 4000)).reshape(2000, 2)
    disk = disk_nodes(0.05).xy
    return {
        "disk": disk,
        "random": u,
        "lattice": disk_nodes(1.0 / 16.0, jitter=0.0).xy,
        "graded": np.sign(u - 0.5) * np.abs(u - 0.5) ** 5,
        "strip": u * np.array([1.0, 1e-3]),
        "line": np.stack([u[:, 0], np.zeros(2000)], axis=1),
        "clusters": np.concatenate([u[:900] * 1e-4, u[900:1800] * 1e-4 + 3.0, u[1800:]]),
        "duplicates": np.concatenate([disk[:600], disk[:600], disk[:40]]),
        "shifted": disk + 1e8,
        "scaled": disk * 1e-30,
        "one point": np.ones((300, 2)),
    }


@pytest.mark.parametrize("name", sorted(_sets()))
@pytest.mark.parametrize("n", [1, 12, 24, 25, 56, 57, 112, 113])
def test_search_bitexact(lib, name, n):
    from paper_2107_03632_gb300 import rbffd

    xy = np.ascontiguousarray(_sets()[name])
    idx = rbffd.rbffd_stencils(torch.from_numpy(xy).to(DEV), n).cpu().numpy()
    assert np.array_equal(idx, oracle.knn(xy, n))


def test_search_with_a_nan_point(lib):
    """The finite points' stencils are as without the point."""
    from paper_2107_03632_gb300 import rbffd

    xy = disk_nodes(0.1).xy.copy()
    ref = oracle.knn(xy, 12)
    with_nan = np.concatenate([xy, [[np.nan, 0.3]]])
    idx = rbffd.rbffd_stencils(torch.from_numpy(with_nan).to(DEV), 12).cpu().numpy()
    assert np.array_equal(idx[:-1], ref)


@pytest.mark.parametrize("bad", [np.inf, -np.inf])
def test_search_with_an_infinite_point_returns(lib, bad):
    """No grid holds such a set: the rows are indices, nothing more is promised."""
    from paper_2107_03632_gb300 import rbffd

    xy = np.concatenate([disk_nodes(0.1).xy, [[bad, 0.3]]])
    idx = rbffd.rbffd_stencils(torch.from_numpy(xy).to(DEV), 12).cpu().numpy()
    assert (idx >= 0).all() and (idx < len(xy)).all()
