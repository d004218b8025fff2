"""The position loss's sums over scenes of a few to thousands of particles: exact
squares of FP32 differences in two FP32 words a thread. The low word holds at
most 24 terms of 2^-24 of the sum and rounds 24 times: 24 * 24 * 2^-48 = 2e-12,
so 1e-11."""
import numpy as np
import pytest

import scenes
from paper_2303_02346_gb300.simulator import Simulator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scene", [-1, 1])
@pytest.mark.parametrize("target", [(0.4, 0.3, 0.5), (1e20, 0.3, 0.5)])
def test_position_loss_sums(target, scene):
    parts = [scenes.small_block(31 + i, 16, [scenes.LIQUID], ppc=p, size_cells=s, lo_cell=(4, 4, 4), n_steps=1)
             for i, (p, s) in enumerate([(1, 1), (8, 7), (1, 3), (5, 5), (3, 1), (8, 8)])]
    sc = scenes.merge_scenes(parts)
    sim = Simulator(sc, checkpoint_every=1)
    sim.reset()
    sim.step(1)
    w = 0.75
    got = np.atleast_1d(np.asarray(sim.position_loss(target, w, scene=scene), np.float64))
    for i, s in enumerate(range(len(parts)) if scene < 0 else [scene]):
        d = sim.state(scene=s)[0].cpu().numpy() - np.asarray(target, np.float32)
        want = w * (d.astype(np.float64) ** 2).sum()
        assert abs(got[i] - want) <= 1e-11 * want, (s, got[i], want)
    sim.close()
