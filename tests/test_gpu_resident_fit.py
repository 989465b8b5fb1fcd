"""A system of which one block's share outgrows the shared memory, though the average one
fits: found out once per operator set."""
import pytest
import torch

from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


def test_a_share_that_does_not_fit_is_remembered():
    from paper_1603_04039_gb300 import APCloud
    ap = APCloud(max_depth=8, c_refine=0.087)
    ap.set_graphs(False)
    ap.build_octree(*(torch.from_numpy(a).to(DEV) for a in inputs.beam_with_halo(1_000_000, 41)[:3]))
    for _ in range(2):
        ap.stencils()
        b = torch.ones(ap.n_nodes, dtype=torch.float64, device=DEV)
        runs = []
        for which in ("A", "B", "A"):
            l0, h0 = ap.launch_count(), ap.host_sync_count()
            x, info = ap.solve_system(which, b, rtol=1e-12, max_iter=3)
            assert info["iters"] == 3
            runs.append((ap.launch_count() - l0, ap.host_sync_count() - h0, x.clone()))
        assert runs[1][0] > 1
        # the first one asks the kernel, which reads the matrix, finds out and reports back
        assert runs[0][0] == runs[2][0] + 1 and runs[0][1] == runs[2][1] + 1
        assert torch.equal(runs[0][2], runs[2][2])
