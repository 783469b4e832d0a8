"""Stencils of node sets whose squared distances leave the normal FP64 range:
below it they underflow to equal keys, above it they overflow to infinity, and
the node index decides.  Bit-exact against the oracle's brute force, on both
sides of the lines where the fixed-point search begins and ends to apply."""

import numpy as np
import pytest
import torch

import oracle
from fixtures import disk_nodes

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("scale", [1e-320, 1e-300, 1e-165, 1e-161, 1e-155, 1e-140, 1e-138, 1e149, 1e151, 1e160, 1e300,
                                   8e307])
def test_search_bitexact_at_any_scale(lib, scale):
    from paper_2107_03632_gb300 import rbffd

    xy = disk_nodes(0.08).xy * scale
    x = torch.from_numpy(xy).to(DEV)
    for n in (1, 12, 45, 90, 113):
        with np.errstate(over="ignore", under="ignore"):
            ref = oracle.knn(xy, n)
        assert np.array_equal(rbffd.rbffd_stencils(x, n).cpu().numpy(), ref), n


def test_search_of_a_set_whose_span_overflows(lib):
    """Finite coordinates, infinite differences; a far pair beside an ordinary disk."""
    from paper_2107_03632_gb300 import rbffd

    disk = disk_nodes(0.1).xy
    far = np.array([[1.5e308, 0.0], [-1.5e308, 0.0]])
    for xy in (np.concatenate([disk, far]), np.concatenate([disk, far[:1]]), np.concatenate([far * 0.2, disk])):
        with np.errstate(over="ignore", under="ignore"):
            ref = oracle.knn(xy, 12)
        assert np.array_equal(rbffd.rbffd_stencils(torch.from_numpy(xy).to(DEV), 12).cpu().numpy(), ref)
