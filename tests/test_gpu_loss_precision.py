"""The position loss against the exact sum of the squares of its FP32 differences, to
FP64's own rounding. All particles share one place, so that every thread's sum is
off by the same amount and nothing averages out. Roundings on the way: one a
thread's sum, one for the weight, five over a warp, eight over a CTA, one for the
total: 16 of 2^-53 each, 1.8e-15, so 2e-15."""
import math
from fractions import Fraction

import numpy as np
import pytest

import scenes
from paper_2303_02346_gb300.simulator import Simulator

pytestmark = pytest.mark.gpu

TARGETS = np.random.default_rng(1).uniform(0.0, 1.0, (12, 3)).astype(np.float32)


def _sim(N):
    n = 24
    sc = scenes.Scene(name="one place", grid_n=n, dt=1e-4, n_steps=1, materials=[scenes.water_material((1.0 / n) ** 3 / 8)],
                      x=np.tile([[0.43, 0.51, 0.37]], (N, 1)), v=np.tile([[0.3, -0.2, 0.1]], (N, 1)),
                      mat=np.zeros(N, np.uint8), scene_counts=[N], checkpoint_every=1)
    sim = Simulator(sc)
    sim.reset()
    sim.step(1)
    return sim


def _exact(x, target, w):
    d = x.astype(np.float32) - np.asarray(target, np.float32)
    return Fraction(float(np.float32(w))) * sum(Fraction(float(t)) ** 2 for t in d.ravel())


@pytest.mark.parametrize("N", [1, 511, 2048])
def test_rounded_as_fp64(N):
    sim = _sim(N)
    x = sim.state()[0].cpu().numpy()
    for target in TARGETS:
        want = _exact(x, target, 0.7)
        got = Fraction(float(sim.position_loss(target, 0.7)[0]))
        assert abs(got - want) <= want * Fraction(2e-15), (target, float((got - want) / want))
    sim.close()


def test_target_met_and_nearly_met():
    """Differences of 0, and of one step of FP32 in one coordinate."""
    sim = _sim(300)
    x = sim.state()[0].cpu().numpy()
    assert float(sim.position_loss(x[0])[0]) == _exact(x, x[0], 1.0)
    near = np.array([np.nextafter(x[0, 0], np.float32(1)), x[0, 1], x[0, 2]], np.float32)
    want = _exact(x, near, 1.0)
    assert abs(Fraction(float(sim.position_loss(near)[0])) - want) <= want * Fraction(2e-15)
    sim.close()


def test_many_particles():
    """Eight particles a thread (from 500,000 on): one more rounding for every CTA's
    total, of 2048 particles."""
    N = 600_001
    n = 64
    rng = np.random.default_rng(7)
    sc = scenes.Scene(name="many", grid_n=n, dt=1e-4, n_steps=1, materials=[scenes.water_material((1.0 / n) ** 3 / 8)],
                      x=0.2 + 0.6 * rng.random((N, 3)), v=np.zeros((N, 3)), mat=np.zeros(N, np.uint8), scene_counts=[N],
                      checkpoint_every=1)
    sim = Simulator(sc)
    sim.reset()
    sim.step(1)
    target = np.array([0.4, 0.1, 0.9], np.float32)
    d = (sim.state()[0].cpu().numpy() - target).astype(np.float64)
    want = math.fsum((d * d).ravel())  # squares of FP32 numbers are exact in FP64
    got = float(sim.position_loss(target)[0])
    assert abs(got - want) <= want * (16 + N / 2048 + 1) * 2.0 ** -53
    sim.close()
