"""The gas's sums over cells at both lengths of a thread's walk (4 planes below 64^3, 16
from there) and where the last walk is cut short, with obstacles. The projection
takes the mean of what it sums, so a cell left out or taken twice moves every
velocity. Against the FP64 oracle; the gas parity bounds (1e-4 on states, 1e-3 on
gradients; a sum in FP64 adds nothing to FP32's 1e-7). Velocities move points by half
a cell, away from the kinks of the back-trace at cell boundaries."""
import numpy as np
import pytest
import torch

from gpu_util import rel
from oracle import gas as G
from paper_2303_02346_gb300.gas import GasSolver

pytestmark = pytest.mark.gpu
DT = torch.float64


@pytest.mark.parametrize("n", [8, 13, 31, 63, 64, 65, 79])
def test_sums_against_oracle(n):
    r = np.random.default_rng(n)
    solid = np.zeros((n, n, n), dtype=bool)
    solid[n // 2:n // 2 + 2, 2:5, 1:6] = True
    solid[n - 1, :3] = True
    dt = 0.01
    u = ((0.5 + 0.2 * r.uniform(-1, 1, (3, n, n, n))) / (dt * n) * ~solid).astype(np.float32)
    d = (r.random((n, n, n)) * ~solid).astype(np.float32)
    w = r.normal(size=(4, n, n, n)).astype(np.float32)
    gs = GasSolver(n, dt, 0.5, 2, 1, solid)
    gs.set_state(u, d)
    gs.step(1)
    gu_, gd_ = gs.state()
    gs.add_grad(w[:3], w[3])
    gu, gd = gs.backward()
    gs.close()
    ut, dt_ = (torch.tensor(a, dtype=DT, requires_grad=True) for a in (u, d))
    u1, d1 = G.rollout(ut, dt_, solid, 1, dt, 0.5, 2)
    g = torch.autograd.grad((u1 * torch.tensor(w[:3], dtype=DT)).sum() + (d1 * torch.tensor(w[3], dtype=DT)).sum(), (ut, dt_))
    fluid = torch.tensor(~solid, dtype=DT)
    assert rel(gu_.cpu(), u1.detach()) <= 1e-4 and rel(gd_.cpu(), d1.detach()) <= 1e-4
    assert rel(gu.cpu(), g[0] * fluid) <= 1e-3 and rel(gd.cpu(), g[1] * fluid) <= 1e-3
