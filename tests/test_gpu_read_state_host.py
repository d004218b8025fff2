"""Host readback on both sides of the size (128 KB) up to which all outputs leave in one
copy: 1365 particles with four outputs need 131,040 bytes, 1366 need 131,136. Every
combination of outputs, against the device outputs; values are copied, so the
comparisons are exact."""
import itertools

import numpy as np
import pytest

import scenes
from paper_2303_02346_gb300 import binding as B
from paper_2303_02346_gb300.simulator import Simulator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [(3,), (1365,), (1366,), (700, 5000)])
def test_host_outputs(counts):
    n = 24
    rng = np.random.default_rng(len(counts) + counts[0])
    N = int(sum(counts))
    vp = (1.0 / n) ** 3 / 8
    sc = scenes.Scene(name="host", grid_n=n, dt=1e-4, n_steps=2, materials=[scenes.water_material(vp), scenes.von_mises_material(vp)],
                      x=(6 + 12 * rng.random((N, 3))) / n, v=rng.normal(size=(N, 3)), mat=rng.integers(0, 2, N).astype(np.uint8),
                      scene_counts=list(counts), checkpoint_every=2)
    sim = Simulator(sc)
    sim.reset()
    sim.step(2)
    for scene in range(-1, len(counts)):
        want = [t.cpu().numpy().reshape(t.shape[0], -1) for t in sim.state(scene=scene, with_CF=True)]
        for chosen in itertools.product((False, True), repeat=4):
            outs = [np.full_like(w, np.nan) if c else None for w, c in zip(want, chosen)]
            B.sim_get_state(sim.h, scene, -1, *outs)
            assert all(o is None or np.array_equal(o, w) for o, w in zip(outs, want))
    sim.close()
