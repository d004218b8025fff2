"""Outputs of a simulator on a stream of its own, read back under another stream.
The allocator may hand an output a block whose last owner is still being read by work
on the current stream; the library has to write it after that work. Values are
copied, so the comparisons are exact."""
import pytest
import torch

import scenes
from paper_2303_02346_gb300 import binding as B
from paper_2303_02346_gb300.simulator import Simulator

pytestmark = pytest.mark.gpu


def _pending_copy(shape):
    """(block, its copy): the block of a freed tensor that a copy on the current
    stream, behind about a tenth of a second of waiting, still has to read."""
    torch.cuda.empty_cache()
    copy = torch.zeros(shape, device="cuda")
    block = torch.full(shape, 7.0, device="cuda")
    torch.cuda.synchronize()
    ptr = block.data_ptr()
    torch.cuda._sleep(200_000_000)
    copy.copy_(block)
    return ptr, copy


# binding: without Simulator, the library orders its outputs after the default stream alone
@pytest.mark.parametrize("what,current", [("state", "default"), ("state", "side"), ("backward", "default"),
                                          ("backward", "side"), ("binding", "default")])
def test_outputs_wait_for_the_current_stream(what, current):
    # 3 N floats: more than a megabyte, so that the block is one of its own
    sc = scenes.small_block(5, 64, (scenes.LIQUID,), ppc=8, size_cells=28, n_steps=2)
    sim = Simulator(sc, checkpoint_every=2, stream=torch.cuda.Stream().cuda_stream)
    sim.reset()
    sim.step(2)
    want = sim.state()[0].cpu()
    sim.position_loss(sc.loss["target"])
    shape = (sim.N, 3)
    with torch.cuda.stream(torch.cuda.Stream() if current == "side" else torch.cuda.default_stream()):
        ptr, copy = _pending_copy(shape)
        if what == "state":
            outs = sim.state()
        elif what == "backward":
            outs = sim.backward()[:2]
        else:
            outs = [torch.empty(shape, device="cuda") for _ in range(2)]
            B.sim_get_state(sim.h, -1, -1, *outs)
        torch.cuda.synchronize()
        assert ptr in [o.data_ptr() for o in outs], "the freed block was not handed out again"
        assert bool((copy == 7.0).all())
        if what != "backward":
            assert torch.equal(outs[0].cpu(), want)
    sim.close()
