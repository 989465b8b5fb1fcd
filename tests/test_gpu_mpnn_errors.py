"""A sort of the learned part that reports a time-out (here its report is written into the
context's error word by the test; nothing hangs) fails the call, and the next one recovers."""
import pytest
import torch

from paper_1603_04039_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
ERR_TIMEOUT = 16


class _Words:
    def __init__(self, ptr, n):
        self.__cuda_array_interface__ = dict(shape=(n,), typestr="<i4", data=(ptr, False), version=3)


@pytest.mark.parametrize("call", ["loss", "outputs", "solve"])
def test_a_sort_that_gave_up_is_reported(call):
    from paper_1603_04039_gb300 import APCloud, APCloudError, MPNN
    from paper_1603_04039_gb300._binding import TorchAllocator
    alloc = TorchAllocator(DEV)
    ap = APCloud(max_depth=5, c_refine=0.5, allocator=alloc)
    word = torch.as_tensor(_Words(next(iter(alloc.live)), 4), device=DEV)   # the context's first buffer
    net = MPNN(seed=1)
    run = {"loss": lambda: net.loss(ap, backward=True)["L"], "outputs": lambda: net.outputs(ap)["s"].clone(),
           "solve": lambda: ap.solve_learned(net, use=3, rtol=1e-9)[0].clone()}[call]
    ap.build_octree(*(torch.from_numpy(a).to(DEV) for a in inputs.beam_with_halo(20000, 5)[:3]))
    ap.stencils()
    ap.deposit(q_uniform=1.0 / 20000, rtol=1e-10)
    assert not word[0].item()
    want = run()
    word[0] = ERR_TIMEOUT
    with pytest.raises(APCloudError) as e:
        run()
    assert e.value.status == -6
    got = run()
    assert torch.equal(torch.as_tensor(got), torch.as_tensor(want))
