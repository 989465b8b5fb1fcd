"""Solves that run as one cooperative kernel (matrix in shared memory): every
form at the sizes where the split into blocks and slices can go wrong."""
import numpy as np
import pytest
import torch

from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
FORMS = [dict(precision="fp64"), dict(precision="fp64", poly_degree=2, poly_omega=1.0),
         dict(precision="fp64", poly_degree=16, poly_omega=1.0), dict(precision="mixed"),
         dict(precision="mixed", poly_degree=2, poly_omega=1.0), dict(precision="mixed", poly_degree=16, poly_omega=1.0)]


def _system(n, depth, c, **form):
    from paper_1603_04039_gb300 import APCloud
    ap = APCloud(max_depth=depth, c_refine=c, **form)
    ap.build_octree(*(torch.from_numpy(a).to(DEV) for a in inputs.beam_with_halo(n, 41)[:3]))
    ap.stencils()
    return ap


def _check(ap, which, restart_launches, rtol=1e-9):
    """The reported residual is the FP64 residual of the stored system: the product
    recomputes it to ~1e-12 of ||b||, far inside the 1% left here."""
    g = torch.Generator().manual_seed(5)
    b = torch.randn(ap.n_nodes, generator=g, dtype=torch.float64).to(DEV)
    x0 = 0.1 * torch.randn(ap.n_nodes, generator=g, dtype=torch.float64).to(DEV)
    l0 = ap.launch_count()
    x, info = ap.solve_system(which, b, x0=x0, rtol=rtol, max_iter=20000)
    launches = ap.launch_count() - l0
    assert info["status"] == 0 and info["relres"] <= rtol
    r = b - ap.matvec(which, x)
    assert float(r.norm()) <= 1.01 * rtol * float(b.norm())
    assert (launches == 1) == restart_launches
    # the same call again: the same bits
    x2, info2 = ap.solve_system(which, b, x0=x0, rtol=rtol, max_iter=20000)
    assert torch.equal(x, x2) and info2["iters"] == info["iters"]
    return x, info


# 4 x 4 x 4 cells and fewer than one block's rows; a few blocks with a ragged
# last slice; every SM with several slices
@pytest.mark.parametrize("n,depth,c", [(500, 2, 0.5), (20000, 5, 0.7), (100000, 8, 0.15)])
@pytest.mark.parametrize("form", FORMS)
def test_resident_solve_residual(n, depth, c, form):
    ap = _system(n, depth, c, **form)
    for which in ("A", "B"):
        _check(ap, which, True)


@pytest.mark.parametrize("restart", [1, 2, 31, 32])
@pytest.mark.parametrize("form", [FORMS[0], FORMS[5]])
def test_resident_restart_lengths(restart, form):
    """Restart 31 fills the sums' slots; 32 takes the launched kernels.  The density
    system converges at every length."""
    ap = _system(20000, 5, 0.7, restart=restart, **form)
    _check(ap, "B", restart <= 31)


@pytest.mark.parametrize("form", [FORMS[0], FORMS[5]])
def test_resident_limits(form):
    """Zero right-hand side, a start that already solves the system, an iteration limit."""
    ap = _system(20000, 5, 0.7, **form)
    z = torch.zeros(ap.n_nodes, dtype=torch.float64, device=DEV)
    x, info = ap.solve_system("A", z)
    assert info["iters"] == 0 and info["status"] == 0 and not x.any()
    sol = torch.randn(ap.n_nodes, dtype=torch.float64, device=DEV)
    b = ap.matvec("A", sol)
    x, info = ap.solve_system("A", b, x0=sol, rtol=1e-9)
    assert info["iters"] == 0 and info["status"] == 0
    for limit in (0, 1, 7):
        x, info = ap.solve_system("A", b, rtol=1e-14, max_iter=limit)
        assert info["iters"] == limit and info["status"] == 1
        r = float((b - ap.matvec("A", x)).norm() / b.norm())
        assert abs(r - info["relres"]) <= 1e-10 + 1e-6 * info["relres"]


def test_systems_past_the_shared_memory():
    """A matrix that does not fit runs on the launched kernels, with the same outcome."""
    ap = _system(1_000_000, 8, 0.06, **FORMS[2])
    assert ap.n_nodes > 120_000
    _check(ap, "B", False)
