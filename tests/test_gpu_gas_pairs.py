"""Gas sweeps taken two at a time and the transposed advection's handed-over
corners, where they can go wrong: even and odd sweep counts, a single sweep, grids
whose strips and plane segments end anywhere (partial last strip, threads that
do not fill a warp), obstacles across strips, planes and row ends, solid
walls and none, smooth and rough velocities. Against the FP64 oracle, forward
and gradient.

Tolerances: the gas parity bounds (1e-4 relative on states, 1e-3 on gradients);
a sweep's FP32 rounding is about 1e-7 relative and does not grow with the
number of sweeps. The back-trace's derivative jumps where a traced point
crosses a cell boundary, which FP32 and FP64 may put on different sides, so
the initial velocity moves every point by 0.2 to 0.8 of a cell beyond whole
cells and the gradient is taken over one step."""
import numpy as np
import pytest
import torch

from gpu_util import rel
from oracle import gas as G
from paper_2303_02346_gb300.gas import GasSolver

pytestmark = pytest.mark.gpu
DT = torch.float64
DT_STEP, BETA = 0.01, 1.0  # buoyancy moves a point by at most n beta dt^2 = 0.016 cells


def _case(n, walls, rough, seed):
    r = np.random.default_rng(seed)
    solid = np.zeros((n, n, n), dtype=bool)
    if walls:
        solid[0] = solid[-1] = True
        solid[:, 0] = solid[:, -1] = solid[:, :, 0] = solid[:, :, -1] = True
    c = n // 2
    solid[c - 9:c + 12, c - 16:c + 3, c - 5:c + 30] = True
    solid[3:6, 11:17, 0:9] = True
    solid[n - 20:, 13:14, n - 3:] = True
    x = np.arange(n) / n
    X, Y, Z = np.meshgrid(x, x, x, indexing="ij")
    # displacement in cells: whole + 0.5 +- 0.25
    whole = np.array([1.0, -2.0, 0.0])[:, None, None, None]
    cells = whole + 0.5 + 0.15 * np.stack([np.sin(2 * np.pi * Y), np.cos(2 * np.pi * Z), np.sin(2 * np.pi * X)])
    if rough:
        cells = cells + r.uniform(-0.1, 0.1, cells.shape)
    u = cells / (DT_STEP * n)
    d = np.exp(-((X - 0.5) ** 2 + (Y - 0.3) ** 2 + (Z - 0.5) ** 2) / 0.02)
    w = np.stack([np.cos(2 * np.pi * (X + 0.1 * q)) * np.sin(2 * np.pi * (Y - 0.2 * q)) + Z for q in range(4)])
    return solid, (u * ~solid).astype(np.float32), (d * ~solid).astype(np.float32), w.astype(np.float32)


@pytest.mark.parametrize("n,K,walls,rough", [(160, 2, True, False), (160, 3, False, True), (164, 6, False, False),
                                             (172, 1, True, True), (188, 5, False, True), (40, 4, False, True)])
def test_pairs_against_oracle(n, K, walls, rough):
    solid, u0, d0, w = _case(n, walls, rough, n + K)
    gs = GasSolver(n, DT_STEP, BETA, K, 2, solid)
    for _ in range(2):  # the second time from the captured graphs
        gs.set_state(u0, d0)
        gs.step(1)
        gs.add_grad(w[:3], w[3])
        gu, gd = gs.backward()
    gs.set_state(u0, d0)
    gs.step(2)
    u, d = gs.state()
    gs.close()
    ut, dt_ = (torch.tensor(a, dtype=DT, requires_grad=True) for a in (u0, d0))
    u1, d1 = G.rollout(ut, dt_, solid, 1, DT_STEP, BETA, K)
    loss = (u1 * torch.tensor(w[:3], dtype=DT)).sum() + (d1 * torch.tensor(w[3], dtype=DT)).sum()
    g = torch.autograd.grad(loss, (ut, dt_))
    with torch.no_grad():
        uo, do = G.rollout(u1.detach(), d1.detach(), solid, 1, DT_STEP, BETA, K)
    fluid = torch.tensor(~solid, dtype=DT)
    assert rel(u.cpu(), uo) <= 1e-4 and rel(d.cpu(), do) <= 1e-4
    assert rel(gu.cpu(), g[0] * fluid) <= 1e-3 and rel(gd.cpu(), g[1] * fluid) <= 1e-3
