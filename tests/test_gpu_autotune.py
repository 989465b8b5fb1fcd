"""The autotuner times what differs and leaves the rest as it was."""
import pytest
import torch

from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


def _context(**kw):
    from paper_1603_04039_gb300 import APCloud
    ap = APCloud(max_depth=6, c_refine=0.3, **kw)
    ap.build_octree(*(torch.from_numpy(a).to(DEV) for a in inputs.beam_with_halo(60000, 24)[:3]))
    ap.stencils()
    return ap


@pytest.mark.parametrize("form,variants", [(dict(precision="fp64"), 8), (dict(precision="fp64", poly_degree=8, poly_omega=1.0), 8),
                                           (dict(precision="mixed", poly_degree=16, poly_omega=1.0), 16)])
def test_solves_in_one_kernel_keep_the_shapes(form, variants):
    """None of the shapes reaches such a solve, so none can be better than another."""
    for shape in ((128, 4, 4, 1), (512, 2, 1, 0)):
        ap = _context(**form)
        ap.set_launch_shape(*shape)
        t = ap.autotune(stencils=False)
        assert (t["spmv_block"], t["wls_warps"], t["spmv_unroll"], t["sweep_sorted"]) == shape
        assert len(t["spmv_ms"]) == variants and all(v > 0 for v in t["spmv_ms"].values())


def test_the_block_local_copy_is_one_shape():
    ap = _context(precision="mixed", poly_degree=16, poly_omega=1.0, restart=32)
    t = ap.autotune(stencils=False)
    ms = list(t["spmv_ms"].values())
    assert len(ms) == 16 and len(set(ms[8:])) == 1 and len(set(ms[:8])) > 1
    assert t["sweep_sorted"] == (1 if ms[8] < min(ms[:8]) else 0)
    best = min(range(8), key=lambda k: ms[k])
    assert (t["spmv_block"], t["spmv_unroll"]) == ((64, 128, 256, 512)[best & 3], (1, 4)[best >> 2])
