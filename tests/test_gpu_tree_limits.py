"""Trees at the ends of the parameters' ranges."""
import numpy as np
import pytest
import torch

import oracle
from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


# thresholds of the deeper levels past 2^53 particles, the last two past every level's
@pytest.mark.parametrize("depth,c", [(21, 140.0), (21, 200.0), (12, 60.0), (8, 1e7), (21, 1e9), (21, 1e200)])
@pytest.mark.timeout(120)
def test_large_refinement_constants(depth, c):
    from paper_1603_04039_gb300 import APCloud
    x, y, z, _ = inputs.beam_with_halo(20000, 6)
    ap = APCloud(max_depth=depth, c_refine=c)
    counts = ap.build_octree(*(torch.from_numpy(a).to(DEV) for a in (x, y, z)))
    o = oracle.Oracle(max_depth=depth, c_refine=c)
    o.build(x, y, z)
    assert counts == (o.n_int, o.n_bnd)
    g, (key, first, count) = ap.get_leaves(), o.leaves()
    assert np.array_equal(g["key"].cpu().numpy().astype(np.uint64), key)
    assert np.array_equal(g["first"].cpu().numpy(), first)
    assert np.array_equal(g["count"].cpu().numpy(), count)


def test_many_particles_in_few_deep_cells():
    """Every particle opens its cells down to depth 21, but all of them the same few."""
    from paper_1603_04039_gb300 import APCloud
    g = torch.Generator(device=DEV).manual_seed(3)
    few = 2.0 * torch.rand(3, 8, generator=g, dtype=torch.float64, device=DEV) - 1.0
    res = []
    for n in (80, 100_000_000):
        at = torch.arange(n, device=DEV) % 8
        ap = APCloud(max_depth=21, c_refine=1e-9)
        res.append((ap.build_octree(*(p[at].contiguous() for p in few)), ap.get_leaves()["key"]))
        assert ap.get_leaves()["count"].sum().item() == n
    assert res[0][0] == res[1][0] and torch.equal(res[0][1], res[1][1])


# hi - lo rounds to a power of two, and the doubles past hi lie closer than the units of the
# integer keys
@pytest.mark.parametrize("lo,hi", [(-(1.0 - 2.0 ** -11), 2.0 ** -11 + 2.0 ** -60), (-(1.0 - 2.0 ** -20), 2.0 ** -20 + 2.0 ** -60),
                                   (-(1.0 - 2.0 ** -11), 2.0 ** -11)])
def test_the_last_bit_past_the_domain(lo, hi):
    from paper_1603_04039_gb300 import APCloud, APCloudError
    assert hi - lo == 1.0
    ap = APCloud(lo=lo, hi=hi, max_depth=5, c_refine=0.1)
    x = torch.full((1000,), 0.5 * (lo + hi), dtype=torch.float64, device=DEV)
    y = x.clone()
    y[777] = hi
    ap.build_octree(y, y, y)
    y[777] = np.nextafter(hi, 2.0)
    for k in range(3):
        with pytest.raises(APCloudError) as e:
            ap.build_octree(*(y if d == k else x for d in range(3)))
        assert e.value.status == -2
