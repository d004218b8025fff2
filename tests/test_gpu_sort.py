"""Particle sort and neighbour bins where they can go wrong: one particle, counts
around a warp and a CTA, empty scenes, grids that are not a power of two,
particles in the last cells of the grid and of every 4^3 block, and repeated
sorts (the bins of one must be gone in the next). The neighbour sums over the
bins are compared with brute force over all pairs.

Tolerance: 1e-5 relative as in the sharing tests; a sum has at most a few dozen
FP32 terms of one sign here (positive g), whose rounding is below 3e-6."""
import numpy as np
import pytest
import torch

import scenes
from gpu_util import rel
from oracle import sharing as osh
from paper_2303_02346_gb300.simulator import Simulator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 13, 32])
@pytest.mark.parametrize("counts", [(1,), (31, 0, 2), (257,), (640, 33)])
def test_neighbour_sums_and_order(n, counts):
    rng = np.random.Generator(np.random.PCG64(n + len(counts)))
    N = int(sum(counts))
    # stencil origins over every cell of the grid, the last ones included; half
    # of the particles crowd one corner block
    x = (0.5 + rng.random((N, 3)) * (n - 2.001)) / n
    x[::2] = (n - 2.501 + 0.999 * rng.random((len(x[::2]), 3))) / n
    mats = [scenes.water_material(1e-6), scenes.von_mises_material(1e-6)]
    sc = scenes.Scene(name="sort", grid_n=n, dt=1e-6, n_steps=3, materials=mats, x=x, v=np.zeros_like(x),
                      mat=rng.integers(0, 2, N).astype(np.uint8), scene_counts=[int(c) for c in counts],
                      gravity=(0.0, 0.0, 0.0), bound=0)
    ids = np.repeat(np.arange(len(counts)), counts)
    sim = Simulator(sc, checkpoint_every=0, resort_every=1)
    ell, g = rng.random(N).astype(np.float32), rng.random((N, 3)).astype(np.float32)
    sim.reset()
    for steps in (0, 1, 2):
        sim.step(steps)
        xs, _ = sim.state()
        assert np.abs(xs.cpu().numpy() - x).max() < 0.1 / n  # rows still are the caller's
        got = sim.share_gradients(ell, g, 0.9 / n, 0.5)
        want = osh.share_gradients(xs.cpu().double(), ids, ell, 0.9 / n, 0.5, g)
        assert rel(got.cpu(), want) <= 1e-5
        assert torch.equal(sim.share_gradients(ell, g, 0.9 / n, 0.5).argmax(0), got.argmax(0))
    sim.close()
