"""A context that is used again replays a captured restart cycle only where everything
the capture fixed is the same: solves after a rebuild, or with other arguments, have the
bits and step counts of a fresh context."""
import numpy as np
import pytest
import torch

from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
MIXED = dict(precision="mixed", poly_degree=16, poly_omega=1.0, restart=32)   # restart 32: launched cycles


def _context(beams, form):
    from paper_1603_04039_gb300 import APCloud
    ap = APCloud(max_depth=6, c_refine=0.3, **form)
    sets = [inputs.beam_with_halo(40000 + 7000 * i, 31 + i)[:3] for i in range(beams)]
    return ap, sets


def _build(ap, sets, axes, sign):
    """The clouds seen along other axes: the same cells mirrored, in another order."""
    p = [np.concatenate([sign * s[a] for s in sets]) for a in axes]
    p = [torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in p]
    if len(sets) == 1:
        ap.build_octree(*p)
    else:
        ap.build_octree_batched(*p, np.concatenate([[0], np.cumsum([len(s[0]) for s in sets])]))
    ap.stencils()
    m = ap.get_stencils()["m"].long().cpu()
    m = torch.nn.functional.pad(m, (0, -len(m) % 32)).reshape(-1, 32).amax(dim=1)
    return ap.n_nodes, int(((m + 7) // 8).sum())   # chunks of eight entries in all 32-row slices


def _solve(ap, rtol):
    rho, i0 = ap.deposit(q_uniform=1e-5, rtol=rtol)
    phi, i1 = ap.solve(rtol=rtol, max_iter=2000)
    return rho.clone(), phi.clone(), i0["iters"], i1["iters"], i0["status"], i1["status"]


def _same(a, b):
    return a[2:] == b[2:] and torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("beams", [1, 3])
def test_rebuild_with_the_same_node_count(beams):
    views = [((0, 1, 2), 1.0), ((2, 0, 1), 1.0), ((1, 0, 2), -1.0)]
    used, sets = _context(beams, MIXED)
    shapes = []
    for axes, sign in views:
        shapes.append(_build(used, sets, axes, sign))
        got = _solve(used, 1e-10)
        fresh, _ = _context(beams, MIXED)
        assert _build(fresh, sets, axes, sign) == shapes[-1]
        want = _solve(fresh, 1e-10)
        assert want[4:] == (0, 0) and _same(got, want)
    assert used.graph_stats()["replays"] > 0
    assert len({n for n, _ in shapes}) == 1 and len({k for _, k in shapes}) > 1


@pytest.mark.parametrize("form", [dict(precision="fp64"), dict(precision="fp64", poly_degree=8, poly_omega=1.0),
                                  dict(precision="mixed"), MIXED])
def test_batch_with_another_tolerance(form):
    used, sets = _context(3, form)
    _build(used, sets, (0, 1, 2), 1.0)
    for rtol in (1e-3, 1e-9):
        got = _solve(used, rtol)
        fresh, _ = _context(3, form)
        _build(fresh, sets, (0, 1, 2), 1.0)
        want = _solve(fresh, rtol)
        assert want[4:] == (0, 0) and _same(got, want)
