"""Tool kinematics by whole actions, at the edges of their chunks, and contact at
the edge of the tool's reach. States and gradients to the parity bounds (1e-4,
1e-3: FP32 steps against FP64)."""
import math

import numpy as np
import pytest

import scenes
from gpu_util import oracle_forward, oracle_grad, rel
from paper_2303_02346_gb300.simulator import Simulator

pytestmark = pytest.mark.gpu


def tool_scene(steps, spa, **kw):
    sc = scenes.small_block(12, 16, [scenes.LIQUID, scenes.VON_MISES], ppc=2, size_cells=4, lo_cell=(5, 3, 5),
                            n_steps=steps, dt=5e-5, tool=True, **kw)
    sc.substeps_per_action = spa
    rng = np.random.default_rng(3)
    n_act = (steps + spa - 1) // spa
    sc.tool_actions = rng.uniform(-1, 1, (1, n_act, 6)) * [0.3, 0.3, 0.3, 6.0, 6.0, 6.0] + [0, -1.0, 0, 0, 0, 0]
    return sc


def check(sc, every):
    sim = Simulator(sc, checkpoint_every=every)
    sim.reset()
    sim.step(sc.n_steps)
    x, v = sim.state()
    xo, vo, _, _ = oracle_forward(sc)
    assert rel(x.cpu(), xo) < 1e-4 and rel(v.cpu(), vo) < 1e-4
    sim.position_loss(sc.loss["target"], 1.0, scene=0)
    gx, _, ga = sim.backward()
    ref = oracle_grad(sc, want_actions=True)
    assert np.abs(ref["actions"]).max() > 0
    assert rel(ga.cpu()[0], ref["actions"]) < 1e-3 and rel(gx.cpu(), ref["x0"]) < 1e-3
    sim.close()


# one step; one action a step; a ragged last action; 44 actions (two chunks of
# 32) over 131 steps (two chunks of 128); one action throughout
@pytest.mark.parametrize("steps,spa", [(1, 1), (5, 1), (20, 7), (131, 3), (131, 200)])
def test_actions_and_steps_by_chunks(steps, spa):
    check(tool_scene(steps, spa), 50)


def test_contact_at_the_corner_farthest_from_the_centre():
    sc = tool_scene(12, 5)
    dx = 1.0 / 16
    half = np.array([2.2, 0.4, 0.7]) * dx
    top = (3 + 4) * dx
    # the corner direction turned straight down: the contact shell's only part in reach
    d = half / np.linalg.norm(half)
    axis = np.cross(d, [0.0, -1.0, 0.0])
    ang = math.atan2(np.linalg.norm(axis), -d[1])
    axis /= np.linalg.norm(axis)
    q = np.concatenate([[math.cos(ang / 2)], math.sin(ang / 2) * axis])
    sc.tool_half = tuple(half)
    c = np.array([7.0 * dx, top + np.linalg.norm(half) + 0.3 * dx, 7.0 * dx])
    sc.tool_pose0 = np.array([[*c, *q]])
    check(sc, 12)
