"""Field at the particles (mixed form: records fetched by whole warps; FP64 form: the centre
from the record) against the same expansion in FP64, at particle counts around those of
warps and blocks."""
import pytest
import torch

from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n,depth,c", [(33, 4, 1.0), (2016, 4, 0.5), (2047, 5, 0.3), (2048, 4, 0.5), (2049, 4, 0.5),
                                       (2305, 6, 0.1)])
def test_mixed_gather_is_the_leaf_expansion(n, depth, c):
    # FP32 terms: each passes at most 16 roundings (record, offset, products, sums) of 2^-24
    _check(n, depth, c, "mixed", 16 * 2.0 ** -24)


@pytest.mark.parametrize("n,depth,c", [(33, 4, 1.0), (2049, 4, 0.5), (2305, 6, 0.1)])
def test_fp64_gather_is_the_leaf_expansion(n, depth, c):
    # the same count of roundings, and up to 64 in the sums of the derivatives on either side
    _check(n, depth, c, "fp64", 80 * 2.0 ** -53, True)


def _check(n, depth, c, precision, tol, sums=False):
    from paper_1603_04039_gb300 import APCloud
    x, y, z, _ = inputs.beam_with_halo_device(n, 9, DEV)
    order = torch.randperm(n, device=DEV)
    p = torch.stack([x, y, z])[:, order].contiguous()
    ap = APCloud(max_depth=depth, c_refine=c, precision=precision)
    ap.build_octree(*p)
    ap.stencils()
    ap.deposit(rtol=1e-6)
    nodes, ni = ap.get_nodes(), ap.n_int
    xyz = nodes["xyz"]
    phi0 = torch.cos(3.0 * xyz[:, 0]) * torch.exp(xyz[:, 1]) + xyz[:, 2] ** 3
    ap.solve(phi0=phi0, max_iter=0)
    got = ap.gather_field()
    # node derivatives x y z xx xy xz yy yz zz
    st = ap.get_stencils()
    live = torch.arange(st["nbr"].shape[1], device=DEV) < st["m"][:, None]
    diff = torch.where(live, phi0[st["nbr"].long().clamp(min=0)] - phi0[:ni, None], 0.0)
    terms = torch.where(live[:, None, :], st["D"], 0.0) * diff[:, None, :]
    f, fa = terms.sum(2), terms.abs().sum(2)
    # every particle's leaf
    lev = nodes["level"][:ni].long()
    anchor = ap.get_leaves()["key"] << (3 * (depth - lev))
    key = torch.zeros(n, dtype=torch.int64, device=DEV)
    for d in range(3):
        cell = torch.clamp(torch.floor((p[d] + 1.0) * 2.0 ** (depth - 1)).long(), max=2 ** depth - 1)
        for b in range(depth):
            key |= (cell >> b & 1) << (3 * b + 2 - d)
    leaf = torch.searchsorted(anchor, key, right=True) - 1
    r = p.T - xyz[leaf]
    g, h = f[leaf][:, :3], f[leaf][:, [3, 4, 5, 4, 6, 7, 5, 7, 8]].reshape(-1, 3, 3)
    hr = (h * r[:, None, :]).sum(2)
    want = [phi0[leaf] + (g * r).sum(1) + 0.5 * (r * hr).sum(1)] + list((g + hr).T)
    if sums:
        g, h = fa[leaf][:, :3], fa[leaf][:, [3, 4, 5, 4, 6, 7, 5, 7, 8]].reshape(-1, 3, 3)
    ahr = (h.abs() * r.abs()[:, None, :]).sum(2)
    size = [(g.abs() * r.abs()).sum(1) + (r.abs() * ahr).sum(1)] + list((g.abs() + ahr).T)
    for k in range(4):
        assert torch.all((got[k] - want[k]).abs() <= tol * size[k] + 1e-13)
