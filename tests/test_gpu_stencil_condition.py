"""The condition estimate that the rank test decides on, min / max |R_ii| of the weighted
Vandermonde, in FP64."""
import math

import numpy as np
import pytest
import torch

from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


class _Doubles:
    def __init__(self, ptr, n):
        self.__cuda_array_interface__ = dict(shape=(n,), typestr="<f8", data=(ptr, False), version=3)


# well conditioned; few neighbours, and weights that all but drop the farthest (estimates
# down to 3e-4, the correction of the first factorisation at its largest)
@pytest.mark.parametrize("kw", [{}, dict(m_target=9), dict(m_target=12, weight_c=1.02)])
def test_condition_estimate(kw):
    from paper_1603_04039_gb300 import APCloud
    from paper_1603_04039_gb300._binding import TorchAllocator
    alloc = TorchAllocator(DEV)
    ap = APCloud(max_depth=7, c_refine=0.3, allocator=alloc, **kw)
    ap.build_octree(*(torch.from_numpy(a).to(DEV) for a in inputs.beam_with_halo(30000, 5)[:3]))
    before = len(alloc.live)
    ap.stencils()
    est = torch.as_tensor(_Doubles(list(alloc.live)[before + 6], ap.n_int), device=DEV).cpu().numpy()
    st, xyz = ap.get_stencils(), ap.get_nodes()["xyz"].cpu().numpy()
    nbr, m = st["nbr"].cpu().numpy(), st["m"].cpu().numpy()
    ec = math.exp(-kw.get("weight_c", 4.0))
    for j in range(0, ap.n_int, 7):
        off = xyz[nbr[j, :m[j]]] - xyz[j]
        r2 = (off ** 2).sum(1)
        w = (np.exp(-r2 / r2.max()) - ec) / (1 - ec)
        x, y, z = (off / np.abs(off).max()).T
        v = np.stack([x, y, z, x * x / 2, x * y, x * z, y * y / 2, y * z, z * z / 2], axis=1) * w[:, None]
        d = np.abs(np.diag(np.linalg.qr(v, mode="r")))
        # kappa (at most 1e4 here) times the 64 roundings of a column's sums, on either side
        assert abs(est[j] - d.min() / d.max()) <= 1e4 * 128 * 2.0 ** -53 * est[j]
