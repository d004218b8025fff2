"""Action gradients of a tool scene of water, von Mises and sand between launch shapes,
separate and fused adjoint, and repeated runs. Contact starts and ends, and sticks or
slips, by the sign of FP32 numbers; where one of those is within rounding of zero, a
gradient has two values and the order of FP32 atomics chooses between them. This scene
has no such node in its steps, so its runs differ by rounding: contributions of some
hundred nodes a step, 1e-7 each, and 1e-5 of the whole leaves room for a hundred such."""
import pytest

import scenes
from gpu_util import rel
from paper_2303_02346_gb300 import binding as B
from paper_2303_02346_gb300.simulator import Simulator

pytestmark = pytest.mark.gpu

SHAPES = [(128, 3, 0), (128, 4, 0), (256, 3, 0), (256, 4, 0), (128, 3, 1), (128, 4, 1), (256, 3, 1)]


@pytest.mark.parametrize("grid,particles,steps,every", [(80, 10_034, 17, 17), (64, 30_098, 40, 12), (110, 60_000, 30, 7)])
def test_launch_shapes_agree(grid, particles, steps, every):
    sc = scenes.multi_material(1, scale=particles / 200_000, n_steps=steps, grid_n=grid, checkpoint_every=every)
    sim = Simulator(sc)
    first = None
    for threads, ctas, fuse in SHAPES:
        B.sim_set_launch(sim.h, threads, threads, 4, 8, fuse_adjoint=fuse, scatter_ctas=ctas)
        for _ in range(2):
            sim.reset()
            sim.step(steps)
            x, v = (t.cpu() for t in sim.state())
            loss = sim.grid_mass_loss(sc.loss["target_mass"], sc.loss["target_dist"], sc.loss["total_mass"])
            ga = sim.backward()[2].cpu()
            if first is None:
                first = (x, v, loss, ga)
                assert float(ga.norm()) > 0.0
            assert rel(x, first[0]) <= 1e-6 and rel(v, first[1]) <= 1e-5 and abs(loss - first[2]) <= 1e-5 * abs(first[2])
            assert rel(ga, first[3]) <= 1e-5, (threads, ctas, fuse)
    sim.close()
