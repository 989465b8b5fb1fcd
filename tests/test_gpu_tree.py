"""The tree's own branches: 32- and 64-bit keys, integer key arithmetic on and
beside cell boundaries in other domains, a set of cells that outgrows its first
table, and the three ways the particle-to-leaf maps are stored."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


def _same_tree(x, y, z, depth, c, lo=-1.0, hi=1.0):
    from paper_1603_04039_gb300 import APCloud
    ap = APCloud(lo=lo, hi=hi, max_depth=depth, c_refine=c)
    counts = ap.build_octree(*(torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (x, y, z)))
    o = oracle.Oracle(lo=(lo,) * 3, hi=(hi,) * 3, max_depth=depth, c_refine=c)
    o.build(x, y, z)
    assert counts == (o.n_int, o.n_bnd)
    g, (key, first, count) = ap.get_leaves(), o.leaves()
    assert np.array_equal(g["key"].cpu().numpy().astype(np.uint64), key)
    assert np.array_equal(g["first"].cpu().numpy(), first)
    assert np.array_equal(g["count"].cpu().numpy(), count)
    assert np.array_equal(ap.get_nodes()["xyz"].cpu().numpy(), o.nodes()["xyz"])


# depth 0: nothing to sort; 10 and 11: 32- and 64-bit keys; 300 lone particles
# refined to depth 15: the balance opens about seven times the cells the
# criterion does, more than the first table takes
@pytest.mark.parametrize("n,depth,c", [(50, 0, 1.0), (1, 3, 1e-9), (20000, 10, 0.2), (20000, 11, 0.2), (300, 15, 1e-9)])
def test_tree_sizes(n, depth, c):
    x, y, z, _ = inputs.uniform_box(n, 7) if depth == 15 else inputs.beam_with_halo(n, 6)
    _same_tree(x, y, z, depth, c)


# power-of-two extents take the integer keys where lo is a whole number of
# their units; the others, and lo past the units' range, the FP64 ones
@pytest.mark.parametrize("lo,hi", [(-1.0, 1.0), (0.0, 1.0), (-1e-3, 1.999), (-0.5, 1.5), (0.0, 3.0), (100.0, 104.0),
                                   (0.0, 2.0 ** -30), (-2.0 ** -10, 2.0 - 2.0 ** -10)])
def test_keys_on_cell_boundaries(lo, hi):
    rng = np.random.default_rng(3)
    ext = hi - lo
    p = lo + rng.integers(0, 2 ** 14 + 1, size=(3, 6000)) * (ext * 2.0 ** -14)
    p[:, :50], p[:, 50:100] = lo, hi
    for k, (steps, to) in enumerate([(0, 0), (1, math.inf), (1, -math.inf), (2, math.inf), (2, -math.inf)]):
        s = slice(1000 * k, 1000 * (k + 1))
        for _ in range(steps):
            p[:, s] = np.nextafter(p[:, s], to)
    tiny = np.array([0.0, -0.0, 5e-324, -5e-324, 1e-300, -1e-300] + [s * 2.0 ** -e for e in (53, 55, 60, 61, 62)
                                                                       for s in (1, -1)])
    p = np.clip(np.concatenate([p, np.tile(tiny, (3, 1))], axis=1), lo, hi)
    _same_tree(*p, 14, 0.1 * ext, lo, hi)


def test_positions_outside_the_domain_are_refused():
    from paper_1603_04039_gb300 import APCloud, APCloudError
    x = torch.zeros(1000, dtype=torch.float64, device=DEV)
    ap = APCloud(max_depth=5)
    for bad in (math.nextafter(1.0, 2.0), math.nextafter(-1.0, -2.0), math.nan, math.inf, -math.inf, 1e300):
        y = x.clone()
        y[777] = bad
        with pytest.raises(APCloudError) as e:
            ap.build_octree(x, y, x)
        assert e.value.status == -2


# straight stores; windows in shared memory (a ragged last one); windows in L2
@pytest.mark.parametrize("n", [8193, 13_200_000, 33_700_001])
def test_particle_maps(n):
    """Charges that differ from particle to particle, deposited leaf by leaf, and
    the leaves' field at the particles."""
    from paper_1603_04039_gb300 import APCloud
    depth = 5
    x, y, z, _ = inputs.beam_with_halo_device(n, 9, DEV)
    order = torch.randperm(n, device=DEV)
    x, y, z = x[order], y[order], z[order]
    q = torch.rand(n, device=DEV, dtype=torch.float64)
    ap = APCloud(max_depth=depth, c_refine=math.sqrt(n) * 2e-3)
    ap.build_octree(x, y, z)
    leaves, nodes = ap.get_leaves(), ap.get_nodes()
    lev = nodes["level"][:ap.n_int].long()
    anchor = leaves["key"] << (3 * (depth - lev))
    key = torch.zeros(n, dtype=torch.int64, device=DEV)
    for d, p in enumerate((x, y, z)):
        c = torch.clamp(torch.floor((p + 1.0) * 2.0 ** (depth - 1)).long(), max=2 ** depth - 1)
        for b in range(depth):
            key |= (c >> b & 1) << (3 * b + 2 - d)
    leaf = torch.searchsorted(anchor, key, right=True) - 1
    assert torch.equal(torch.bincount(leaf, minlength=ap.n_int), leaves["count"].long())
    ap.stencils()
    ap.deposit(q=q, rtol=1e-6)
    h = 2.0 * 0.5 ** lev.double()
    want = torch.zeros(ap.n_int, dtype=torch.float64, device=DEV).index_add_(0, leaf, q)
    got = ap.get_rho_m()[:ap.n_int] * h ** 3
    # both sums of up to n terms round: n eps of the sum at the very most
    assert torch.all((got - want).abs() <= 1e-9 * want)
    # potential and field of phi = x: the leaf's own expansion, so exactly x to rounding
    ap.solve(phi0=nodes["xyz"][:, 0].contiguous(), max_iter=0)
    phi, ex, _, _ = ap.gather_field()
    assert float((phi - x).abs().max()) <= 1e-11 and float((ex - 1.0).abs().max()) <= 1e-9
