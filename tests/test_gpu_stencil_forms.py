"""Branches of the stencil build against the oracle: FP64 blocks that need the
full second Cholesky QR pass, rings that outgrow the candidate set, trees too
deep for the packed rank keys, mixed blocks sent to the list kernel."""
import numpy as np
import pytest
import torch

import oracle
from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n,depth,c,kw", [
    (3000, 7, 0.2, dict(m_target=9, ring_max=2)),       # small, badly conditioned stencils
    (3000, 7, 0.2, dict(m_target=32)),                  # the widest
    (3000, 7, 0.2, dict(stencil_slots=16)),             # nearly every ring outgrows the first pass
    (400, 21, 1e-4, dict()),                            # 64-bit keys cannot hold distance and index
    (3000, 7, 0.2, dict(precision="mixed", fp32_rcond_min=2.0)),   # every block redone in FP64
])
def test_stencils_match_oracle(n, depth, c, kw):
    from paper_1603_04039_gb300 import APCloud
    x, y, z, _ = inputs.beam_with_halo(n, 8)
    ap = APCloud(max_depth=depth, c_refine=c, **kw)
    ap.build_octree(*(torch.from_numpy(a).to(DEV) for a in (x, y, z)))
    o = oracle.Oracle(max_depth=depth, c_refine=c, m_target=kw.get("m_target", 20), ring_max=kw.get("ring_max", 5))
    o.build(x, y, z)
    ap.stencils()
    g, w = {k: v.cpu().numpy() for k, v in ap.get_stencils().items()}, o.stencils()
    assert np.array_equal(g["m"], w["m"]) and np.array_equal(g["nbr"], w["nbr"])
    # the parity tests' bound: 1e-11 of the row's largest entry
    scale = np.abs(w["lap"]).max(axis=1, keepdims=True)
    assert np.all(np.abs(g["lap"] - w["lap"]) <= 1e-11 * scale)
    dscale = np.abs(w["D"]).max(axis=2, keepdims=True)
    assert np.all(np.abs(g["D"] - w["D"]) <= 1e-11 * dscale)
    if "precision" in kw:
        assert ap.sizes()["fp64_stencils"] >= ap.n_int
