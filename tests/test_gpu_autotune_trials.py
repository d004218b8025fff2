"""The autotuner scores the shapes of the separate adjoint kernels on those kernels,
whichever adjoint the handle runs when it is tuned. Counted in launches: of its
trials, ten come before the choice between fused and separate, and a fused trial of
10 steps in 2 chunks launches 8 kernels fewer. The trials after it (staged gather,
persistent forward) follow its choice, which may differ between the handles: at most
two trials of those 8."""
import numpy as np
import pytest

import scenes
from paper_2303_02346_gb300 import binding as B
from paper_2303_02346_gb300.simulator import Simulator

pytestmark = pytest.mark.gpu


def _launches(N, fuse):
    n = 24
    rng = np.random.default_rng(N)
    vp = (1.0 / n) ** 3 / 8
    sc = scenes.Scene(name="tune", grid_n=n, dt=1e-4, n_steps=10, materials=[scenes.water_material(vp)],
                      x=0.3 + 0.3 * rng.random((N, 3)), v=np.zeros((N, 3)), mat=np.zeros(N, np.uint8),
                      scene_counts=[N], checkpoint_every=5)
    sim = Simulator(sc)
    B.sim_set_launch(sim.h, 128, 128, 4, 8, fuse_adjoint=fuse)
    sim.reset()
    before = B.sim_kernel_launches(sim.h)
    B.sim_autotune(sim.h, 10)
    count = B.sim_kernel_launches(sim.h) - before
    sim.close()
    return count


def test_trials_do_not_depend_on_the_current_adjoint():
    assert abs(_launches(901, 0) - _launches(902, 1)) <= 2 * 8
