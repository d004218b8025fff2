"""Warp scatter of the P2G and G2P-adjoint kernels where it can go wrong: a lone
particle, partial and exactly full warps, a warp whose particles all share one
cell, a warp spread over 32 cells far apart, and warps that straddle scenes,
for every CTA size and residency, separate and fused adjoint.

Tolerances: the library's own parity bounds (1e-4 relative on x and v, 1e-3 on
gradients). Each node sum has at most a few hundred FP32 terms of mixed sign,
whose rounding is below 1e-5 relative, so the bounds leave an order of
magnitude."""
import numpy as np
import pytest

import scenes
from gpu_util import oracle_forward, oracle_grad, rel
from paper_2303_02346_gb300 import binding as B
from paper_2303_02346_gb300.simulator import Simulator

pytestmark = pytest.mark.gpu


def _scene(counts, layout, seed=11, n=24):
    rng = np.random.Generator(np.random.PCG64(seed))
    xs = []
    for c in counts:
        if layout == "one_cell":
            cell = np.full((c, 3), 9.6)
        elif layout == "spread":
            cell = 4.0 + 14.0 * rng.random((c, 3))
        else:
            cell = 8.0 + np.floor(3.0 * rng.random((c, 3)))
        xs.append((cell + 0.8 * rng.random((c, 3))) / n)
    x = np.concatenate(xs)
    N = len(x)
    vp = (1.0 / n) ** 3 / 8
    mats = [scenes.water_material(vp), scenes.von_mises_material(vp)]
    return scenes.Scene(name="scatter", grid_n=n, dt=1e-4, n_steps=4, materials=mats, x=x,
                        v=0.5 * rng.normal(size=(N, 3)), mat=(np.arange(N) % 3 == 2).astype(np.uint8),
                        scene_counts=[int(c) for c in counts], checkpoint_every=2,
                        loss={"kind": "position", "target": (0.4, 0.3, 0.5), "weight": 1.0}, seed=seed)


@pytest.mark.parametrize("layout", ["one_cell", "spread", "block"])
@pytest.mark.parametrize("counts", [(1,), (31, 1), (32,), (33, 0, 40), (130, 127)])
def test_scatter_against_oracle(counts, layout):
    sc = _scene(counts, layout)
    fwd = [oracle_forward(sc, scene_index=s) for s in range(sc.n_scenes) if counts[s]]
    ref = [oracle_grad(sc, scene_index=s) for s in range(sc.n_scenes) if counts[s]]
    x, v = (np.concatenate([f[k] for f in fwd]) for k in (0, 1))
    gx, gv = (np.concatenate([r[k] for r in ref]) for k in ("x0", "v0"))
    for threads, ctas, fuse in ((128, 3, 0), (128, 4, 0), (256, 3, 1), (256, 4, 0), (128, 3, 1)):
        sim = Simulator(sc)
        B.sim_set_launch(sim.h, threads, 256, 4, 8, fuse_adjoint=fuse, scatter_ctas=ctas)
        sim.reset()
        sim.step(sc.n_steps)
        hx, hv = sim.state()
        assert rel(hx.cpu(), x) <= 1e-4 and rel(hv.cpu(), v) <= 1e-4
        sim.position_loss(sc.loss["target"])
        hgx, hgv, _ = sim.backward()
        assert rel(hgx.cpu(), gx) <= 1e-3 and rel(hgv.cpu(), gv) <= 1e-3
        sim.close()
