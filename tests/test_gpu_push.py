"""Drift with reflection at the walls: positions inside, on, next to and past them,
signed zeros, infinities and NaN, in exact arithmetic."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("lo,hi", [(-1.0, 1.0), (0.0, 1.0), (-3.0, 0.0)])
def test_push_reflects_at_the_walls(lo, hi):
    from paper_1603_04039_gb300 import APCloud
    rng = np.random.default_rng(4)
    q = 2.0 ** -20   # sums and reflections of multiples of this are exact
    inside = lo + np.round(rng.random(5001) * (hi - lo) / q) * q
    step = np.round(rng.normal(size=5001) * np.where(rng.random(5001) < 0.5, 1e-2, 3.0) / q) * q
    edge = np.array([lo, hi, lo + q, hi - q, 0.0, -0.0, np.nextafter(hi, 9e9), np.nextafter(lo, -9e9), np.inf, -np.inf,
                     np.nan, 1e300, -1e300])
    p0 = np.concatenate([inside, edge])
    v0 = np.concatenate([2.0 * step, np.zeros(len(edge))])   # dt = 1/2
    p, v = p0 + 0.5 * v0, v0.copy()
    with np.errstate(all="ignore"):
        for wall, out in ((hi, lambda a: a > hi), (lo, lambda a: a < lo)):
            m = out(p)
            p[m], v[m] = 2.0 * wall - p[m], -v[m]
        p = np.where(np.isnan(p), lo, np.clip(p, lo, hi))
    ap = APCloud(lo=lo, hi=hi, max_depth=3)
    got = [torch.from_numpy(a.copy()).to(DEV) for a in (p0, p0, p0, v0, v0, v0)]
    ap.push_particles(*got, dt=0.5)
    for d in range(3):
        assert np.array_equal(got[d].cpu().numpy(), p)
        assert np.array_equal(got[3 + d].cpu().numpy(), v)
