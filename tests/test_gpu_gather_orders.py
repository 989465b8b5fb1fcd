"""The mixed gather's two ways of fetching leaf records give the same bits: particles in
cell order (a record per lane) and the same ones shuffled, which on many leaves have their
records staged by whole warps."""
import pytest
import torch

from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


# leaves below and above the 32768 from which records are staged; a last warp of 1, 31 and 32
@pytest.mark.parametrize("n,depth,c,many", [(60001, 8, 0.15, False), (300031, 8, 0.06, True), (300032, 8, 0.06, True),
                                            (300001, 8, 0.06, True)])
def test_orders_agree(n, depth, c, many):
    from paper_1603_04039_gb300 import APCloud
    p = torch.stack(inputs.beam_with_halo_device(n, 9, DEV)[:3])
    cell = torch.floor((p + 1.0) * 2.0 ** (depth - 1)).long()
    key = torch.zeros(n, dtype=torch.int64, device=DEV)
    for d in range(3):
        for b in range(depth):
            key |= (cell[d] >> b & 1) << (3 * b + 2 - d)
    orders = [torch.argsort(key, stable=True), torch.randperm(n, generator=torch.Generator(device=DEV).manual_seed(4), device=DEV)]
    out = []
    for order in orders:
        ap = APCloud(max_depth=depth, c_refine=c, precision="mixed")
        ap.build_octree(*p[:, order].contiguous())
        assert (ap.n_int >= 32768) == many
        ap.stencils()
        ap.deposit(rtol=1e-6)
        xyz = ap.get_nodes()["xyz"]
        ap.solve(phi0=torch.cos(3.0 * xyz[:, 0]) * torch.exp(xyz[:, 1]) + xyz[:, 2] ** 3, max_iter=0)
        got = torch.empty(4, n, dtype=torch.float64, device=DEV)
        for k, f in enumerate(ap.gather_field()):
            got[k, order] = f
        out.append(got)
    assert torch.equal(out[0], out[1]) and bool(torch.isfinite(out[0]).all())
