"""Mixed-form operators: four nodes per warp against the list kernel's warp per
node (a context whose candidate capacity every ring outgrows sends all nodes
there), which does the same FP32 operations in the same order."""
import pytest
import torch

from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


# node counts around the blocks of 16, coordinates of few and of many bits, the
# smallest stencils (most not certified in FP32) and the widest
@pytest.mark.parametrize("n,depth,c,kw", [
    (33, 3, 0.5, {}), (300, 3, 0.05, {}), (777, 4, 0.05, {}), (20000, 5, 0.3, {}), (1000, 20, 0.02, {}),
    (60000, 7, 0.2, dict(m_target=9, ring_max=2)), (60000, 7, 0.2, dict(m_target=32, ring_max=5)),
    (20000, 6, 0.3, dict(fp32_rcond_min=0.0))])
def test_four_nodes_per_warp_give_the_bits_of_one(n, depth, c, kw):
    from paper_1603_04039_gb300 import APCloud
    x, y, z, _ = inputs.beam_with_halo_device(n, 3, DEV)
    out = []
    for slots in (128, 16):
        ap = APCloud(max_depth=depth, c_refine=c, precision="mixed", stencil_slots=slots, **kw)
        ap.build_octree(x, y, z)
        ap.stencils()
        st = ap.get_stencils()
        out.append(([st[k] for k in ("nbr", "m", "lap", "lapd", "D")], ap.sizes()["fp64_stencils"]))
        assert int(st["m"].min()) >= 9
    for a, b in zip(out[0][0], out[1][0]):
        assert torch.equal(a, b)
    assert out[0][1] == out[1][1]
