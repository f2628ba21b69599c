"""Memory from PyTorch's caching allocator: a block that torch's stream has not finished with yet may become a buffer of
the library, which works on a stream of its own."""
import pytest

import paper_2011_00287_gb300 as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [L.FP64, L.FP32], ids=["fp64", "fp32"])
def test_buffers_that_torch_still_writes(prec):
    import torch
    shape = (40, 24, 20)
    prm = L.default_params(shape, R=6.0, p0=12.0, precision=prec)

    def run():
        sim = L.Simulation([shape], [prm], seed=2)
        sizes = [t.numel() for t in sim._alloc.live.values()]
        sim.step(3)
        state = sim.get_state(0).tobytes()
        sim.close()
        return sizes, state

    sizes, ref = run()
    blocks = [torch.empty(n, dtype=torch.uint8, device="cuda:0") for n in sizes]
    torch.cuda._sleep(200_000_000)  # about a tenth of a second; the writes below wait behind it
    for b in blocks:
        b.fill_(255)
    del b, blocks
    assert run()[1] == ref
    torch.cuda.synchronize()
