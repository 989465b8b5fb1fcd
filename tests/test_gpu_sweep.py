"""Sweeps and products on the block-local copy of the matrix against the same ones
on the sliced ELL: the same entries in the same order, so the same bits."""
import numpy as np
import pytest
import torch

from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


def _cloud(beams, n, depth, c, **kw):
    """restart 32 keeps systems of any size off the resident solve."""
    from paper_1603_04039_gb300 import APCloud
    ap = APCloud(max_depth=depth, c_refine=c, precision="mixed", poly_degree=16, poly_omega=1.0, restart=32, **kw)
    sets = [inputs.beam_with_halo(n * (1 + 3 * i), 50 + i) for i in range(beams)]
    p = [torch.from_numpy(np.concatenate([s[k] for s in sets])).to(DEV) for k in range(3)]
    if beams == 1:
        ap.build_octree(*p)
    else:
        ap.build_octree_batched(*p, np.concatenate([[0], np.cumsum([len(s[0]) for s in sets])]))
    ap.stencils()
    return ap


# less than a block of rows; a few blocks and a ragged last slice; rows of up to
# 32 entries (every chunk in use) and of 16; a million rows (lines read evict-first);
# beams that converge one by one
@pytest.mark.parametrize("beams,n,depth,c,kw", [
    (1, 300, 2, 0.5, {}), (1, 20000, 5, 0.7, {}), (1, 100000, 8, 0.15, {}), (1, 60000, 7, 0.2, dict(m_target=32, ring_max=5)),
    (1, 60000, 7, 0.2, dict(stencil_slots=16)), (1, 10_000_000, 10, 0.043, {}), (3, 2000, 6, 0.2, {}), (9, 500, 5, 0.3, {})])
def test_block_local_copy_gives_the_bits_of_the_ell(beams, n, depth, c, kw):
    ap = _cloud(beams, n, depth, c, **kw)
    out = []
    for sorted_ in (0, 1):
        ap.set_launch_shape(256, 4, 4, sorted_)
        rho, i0 = ap.deposit(q_uniform=1.0 / n, rtol=1e-10)
        phi, i1 = ap.solve(rtol=1e-10)
        assert i0["status"] == 0 and i1["status"] == 0
        out.append((rho.clone(), phi.clone(), i0["iters"], i1["iters"]))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert out[0][2:] == out[1][2:] and out[0][3] > 0


def test_column_scaled_system():
    """The closed-form column scaling leaves a diagonal that is not 1."""
    from paper_1603_04039_gb300 import MPNN
    ap = _cloud(1, 30000, 6, 0.3)
    ap.deposit(q_uniform=1.0 / 30000, rtol=1e-10)
    net = MPNN(seed=1)
    out = []
    for sorted_ in (0, 1):
        ap.set_launch_shape(256, 4, 4, sorted_)
        plain, i0 = ap.solve(rtol=1e-10)
        scaled, i1 = ap.solve_learned(net, use=4, rtol=1e-10)
        again, i2 = ap.solve(rtol=1e-10)
        assert torch.equal(plain, again) and i0["status"] == 0 and i1["status"] == 0 and i1["iters"] > 0
        out.append((plain, scaled, i0["iters"], i1["iters"]))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert out[0][2:] == out[1][2:]
