"""Gradient readback and the adjoint state's two buffers: an odd and an even
number of chunk boundaries, launched directly and replayed from the captured
graph, twice in a row on one handle, into device and host buffers, and either
output alone. Same kernels on the same inputs: only the order of FP32 atomics
differs between runs, so results agree to 1e-5 relative."""
import numpy as np
import pytest

import scenes
from gpu_util import oracle_grad, rel
from paper_2303_02346_gb300 import binding as B
from paper_2303_02346_gb300.simulator import Simulator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps,every", [(4, 4), (6, 3), (6, 2), (7, 2)])
@pytest.mark.parametrize("kinds", [(scenes.LIQUID,), (scenes.LIQUID, scenes.DRUCKER_PRAGER, scenes.RIGID)])
def test_gradients_by_chunks(steps, every, kinds):
    sc = scenes.small_block(5, 24, kinds, ppc=3, size_cells=5, v0=(0.1, -0.3, 0.0), spin=1.0, n_steps=steps)
    ref = oracle_grad(sc)
    N = sc.n_particles
    first = None
    for graphs in (False, True):
        sim = Simulator(sc, checkpoint_every=every, graphs=graphs)
        for _ in range(3):
            sim.reset()
            sim.step(steps)
            sim.position_loss(sc.loss["target"])
            gx, gv, _ = sim.backward()
            assert rel(gx.cpu(), ref["x0"]) <= 1e-3 and rel(gv.cpu(), ref["v0"]) <= 1e-3  # the parity bound
            first = (gx, gv) if first is None else first
            assert rel(gx.cpu(), first[0].cpu()) <= 1e-5 and rel(gv.cpu(), first[1].cpu()) <= 1e-5
        for hx, hv in ((np.zeros((N, 3), np.float32), np.zeros((N, 3), np.float32)),
                       (None, np.zeros((N, 3), np.float32))):
            sim.reset()
            sim.step(steps)
            sim.position_loss(sc.loss["target"])
            B.sim_backward(sim.h, hx, hv)
            assert hx is None or rel(hx, first[0].cpu()) <= 1e-5
            assert rel(hv, first[1].cpu()) <= 1e-5
        sim.close()
