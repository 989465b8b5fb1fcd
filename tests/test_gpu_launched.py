"""Single systems whose solves run as launched cycles: too large for one kernel (restart 12, the
single-reduction steps of the mixed form) or with a restart past its limit (32).  Graphs,
timers, launch shapes, cache hints and dependent launches change nothing but the time."""
import functools

import pytest
import torch

from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
SMALL = dict(n=60_000, depth=6, c=0.3, restart=32)
LARGE = dict(n=3_000_000, depth=9, c=0.063, restart=12)   # 2.5e5 nodes
FORMS = [(SMALL, dict(precision="fp64")), (SMALL, dict(precision="fp64", poly_degree=8, poly_omega=1.0)),
         (SMALL, dict(precision="mixed", poly_degree=16, poly_omega=1.0)), (LARGE, dict(precision="fp64")),
         (LARGE, dict(precision="mixed", poly_degree=16, poly_omega=1.0))]
STEPS = 60   # of a solve: several cycles (one for FP64 with the polynomial of degree 8)


@functools.lru_cache(maxsize=2)
def _particles(n):
    return inputs.beam_with_halo_device(n, 21, DEV)[:3]


def _context(size, form, setup=lambda ap: None):
    from paper_1603_04039_gb300 import APCloud
    ap = APCloud(max_depth=size["depth"], c_refine=size["c"], restart=size["restart"], **form)
    setup(ap)
    ap.build_octree(*_particles(size["n"]))
    ap.stencils()
    ap.deposit(q_uniform=1.0 / size["n"], rtol=1e-11, max_iter=STEPS)
    return ap


def _solve(ap):
    l0 = ap.launch_count()
    phi, info = ap.solve(rtol=1e-11, max_iter=STEPS)
    launches = ap.launch_count() - l0
    assert launches > info["iters"] > 0 and info["restarts"] > 0
    return phi.clone(), info["iters"], info["restarts"], launches


def _same(a, b):
    return a[1:] == b[1:] and torch.equal(a[0], b[0])


@pytest.mark.parametrize("size,form", FORMS)
def test_graphs_direct_launches_and_timers(size, form):
    direct = _context(size, form, lambda ap: ap.set_graphs(False))
    want = _solve(direct)
    direct.get_timing(reset=True)
    direct.set_timing(0xFFFF)
    timed = _solve(direct)
    t0 = direct.get_timing(reset=True)
    assert direct.graph_stats()["replays"] == 0
    graphs = _context(size, form)
    runs = [_solve(graphs) for _ in range(2)]   # captured, then replayed
    assert graphs.graph_stats()["replays"] > 0
    graphs.set_timing(0xFFFF)
    graphs.get_timing(reset=True)
    runs.append(_solve(graphs))
    t1 = graphs.get_timing(reset=True)
    # a replay counts the kernels that ran: its fixed nodes and the bodies of
    # the steps before the stopping test
    assert all(_same(r, want) for r in runs + [timed])
    for kind in ("spmv", "gmres_dots", "gmres_update_norm", "gmres_cycle_end"):
        assert t1[kind][0] > 0.0 and t1[kind][1:] == t0[kind][1:], kind


@pytest.mark.parametrize("size,form", FORMS)
def test_launch_shapes(size, form):
    want = None
    for shape in ((256, 4, 1, 0), (64, 2, 4, 1), (512, 8, 1, 1), (128, 4, 4, 0)):
        ap = _context(size, form, lambda ap: ap.set_launch_shape(*shape))
        got = _solve(ap)
        want = want or got
        assert _same(got, want)


@pytest.mark.parametrize("size,form", [f for f in FORMS if f[1]["precision"] == "mixed"])
def test_kept_lines_and_dependent_launches(size, form):
    ap = _context(size, form)
    want = _solve(ap)
    for graphs in (True, False):
        ap.set_graphs(graphs)
        for keep in (-1, 0, 1 << 20, 1 << 40):
            ap.set_sweep_l2_keep(keep)
            assert _same(_solve(ap), want)
        ap.set_sweep_l2_keep(-1)
        for pdl in (False, True):
            ap.set_dependent_launch(pdl)
            assert all(_same(_solve(ap), want) for _ in range(1 + 3 * pdl))
