"""One application of the preconditioner where the finest level fills the chip
(32 rows per warp in the sweeps and the residual), against the same cycle in
torch float64 from the level views.  Node counts just above the line where
those kernels start and not a multiple of 32; rows of 1 entry (Dirichlet), 12,
30 and 56, and, in the adjoint, of mixed lengths.

Tolerance: a row of at most 64 entries is summed with an error of 64 u of its
terms; a sweep or transfer scales errors by a small factor and there are about
8 per level on at most 8 levels: 64 * 64 * 16 u = 7e4 u of the largest entry,
u = 2^-53 and, float32, 2^-24."""

import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def _cycle(views, l, b, nu=2):
    v = views[l]
    if v["minv"] is not None:
        return v["minv"] @ b
    A, w, n = v["A"], v["w"], v["n_nodes"]
    row = torch.repeat_interleave(torch.arange(n, device=b.device), A.row_ptr[1:] - A.row_ptr[:-1])
    col = A.col.long()

    def resid(x):
        return b - torch.zeros_like(b).index_add_(0, row, A.val * x[col])

    x = w * b
    for _ in range(nu - 1):
        x = x + w * resid(x)
    nc = views[l + 1]["n_nodes"]
    cm = views[l + 1]["is_dirichlet"].bool()
    p = v["p_idx"].long()
    if views[0]["adjoint"]:  # restrict with P^T; prolong with the scaled P (the view holds it)
        raw = views[l]["raw_p"]
        bc = torch.zeros(nc, dtype=b.dtype, device=b.device).index_add_(
            0, p.reshape(-1), (raw * resid(x)[:, None]).reshape(-1))
    else:
        bc = torch.zeros(nc, dtype=b.dtype, device=b.device).index_add_(
            0, p.reshape(-1), (v["p_val"] * resid(x)[:, None]).reshape(-1)) * (nc / n)
        bc = torch.where(cm, torch.zeros_like(bc), bc)
    e = _cycle(views, l + 1, bc, nu)
    x = x + (v["p_val"] * e[p]).sum(dim=1)
    for _ in range(nu):
        x = x + w * resid(x)
    return x


@pytest.mark.parametrize("m,n,adjoint", [(2, 12, False), (4, 30, False), (6, 56, False), (4, 30, True)])
def test_cycle_of_a_large_level(m, n, adjoint):
    from paper_2107_03632_gb300 import rbffd

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    k = math.isqrt(sms * 2048) + 2
    gen = torch.Generator(device="cuda").manual_seed(7 + n)
    g = (torch.arange(k, device="cuda", dtype=torch.float64) + 0.5) / k
    xy = torch.stack([g.repeat(k), g.repeat_interleave(k)], dim=1)
    mask = (xy.sub(0.5).abs().amax(dim=1) > 0.5 - 1.0 / k).to(torch.uint8)
    xy = (xy + (torch.rand(xy.shape, generator=gen, device="cuda", dtype=torch.float64) - 0.5) * (0.5 / k)).contiguous()
    N = xy.shape[0]
    assert N > sms * 2048 and N % 32 != 0
    idx = rbffd.rbffd_stencils(xy, n)
    w, status = rbffd.rbffd_weights(xy, idx, m)
    A = rbffd.rbffd_assemble(idx, w, mask, want_f32=True)
    mg = rbffd.Multigrid(xy, mask, A)
    fwd = mg
    if adjoint:
        mg = rbffd.Multigrid.adjoint_of(fwd, rbffd.rbffd_transpose(A, want_f32=True))
    views = [mg.level(l) for l in range(len(mg.levels()))]
    views[0]["adjoint"] = adjoint
    if adjoint:
        for l in range(len(views) - 1):
            views[l]["raw_p"] = fwd.level(l)["p_val"]
    b = torch.randn(N, generator=gen, device="cuda", dtype=torch.float64)
    if adjoint:  # (the application adds the Dirichlet back substitution; interior data leave it out)
        b = torch.where(mask.bool(), torch.zeros_like(b), b)
    want = _cycle(views, 0, b)
    inner = ~mask.bool()
    for fp32, u in ((False, 2.0**-53), (True, 2.0**-24)):
        got = mg.apply(b, fp32=fp32)
        err = ((got - want)[inner].abs().max() / want[inner].abs().max()).item()
        assert err <= 7e4 * u, (fp32, err)
