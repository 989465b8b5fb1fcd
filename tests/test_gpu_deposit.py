"""Charge of every leaf, summed by a warp (few leaves) or a thread (many): empty
leaves, leaves of one to thousands of particles, against sums in FP64."""
import pytest
import torch

from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n,depth,c", [(40, 3, 0.5), (5000, 3, 3.0), (100000, 6, 1.0), (400000, 8, 0.1)])
def test_leaf_charges(n, depth, c):
    from paper_1603_04039_gb300 import APCloud
    x, y, z, _ = inputs.beam_with_halo_device(n, 9, DEV)
    q = torch.rand(n, device=DEV, dtype=torch.float64) - 0.25
    ap = APCloud(max_depth=depth, c_refine=c)
    ap.build_octree(x, y, z)
    lev, lv = ap.get_nodes()["level"][:ap.n_int].long(), ap.get_leaves()
    anchor = lv["key"] << (3 * (depth - lev))
    key = torch.zeros(n, dtype=torch.int64, device=DEV)
    for d, p in enumerate((x, y, z)):
        cell = torch.clamp(torch.floor((p + 1.0) * 2.0 ** (depth - 1)).long(), max=2 ** depth - 1)
        for b in range(depth):
            key |= (cell >> b & 1) << (3 * b + 2 - d)
    leaf = torch.searchsorted(anchor, key, right=True) - 1
    zero = torch.zeros(ap.n_int, dtype=torch.float64, device=DEV)
    want, size = zero.index_add(0, leaf, q), zero.index_add(0, leaf, q.abs())
    ap.stencils()
    ap.deposit(q=q, rtol=1e-6)
    got = ap.get_rho_m()[:ap.n_int] * (2.0 * 0.5 ** lev.double()) ** 3
    # two sums of count terms each, and three more roundings
    assert torch.all((got - want).abs() <= (2 * lv["count"] + 3) * 2.0 ** -53 * size)
    assert int(lv["count"].max()) > 2 and (n > 100000 or ap.n_int < 9000) and (n < 400000 or ap.n_int > 10000)
