"""Gas sweeps in pairs on grids whose rows leave a CTA fewer than 16 rows of threads
(above 256^3): 15 rows at 260^3 with a last warp of 15 threads, 12 at 340^3, 8 at
512^3, the largest grid and the one that needs most shared memory. The FP64 oracle
runs on the GPU. Tolerances: the gas parity bounds (1e-4 relative on states, 1e-3 on
gradients), which leave FP32's 1e-7 a sweep much room; velocities move points by
half a cell, away from the kinks of the back-trace at cell boundaries."""
import numpy as np
import pytest
import torch

from oracle import gas as G
from paper_2303_02346_gb300.gas import GasSolver

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float((a.double() - b).norm() / b.norm())


@pytest.mark.parametrize("n,K,grad", [(260, 3, True), (340, 2, True), (512, 2, False)])
def test_large_grids_against_oracle(n, K, grad):
    solid = np.zeros((n, n, n), dtype=bool)
    solid[n // 2 - 9:n // 2 + 12, n // 2 - 16:n // 2 + 3, n // 2 - 5:n // 2 + 30] = True
    solid[3:6, 11:17, :9] = True
    solid[n - 20:, 13:14, n - 3:] = True
    dt = 0.004
    with torch.device("cuda"):
        g = torch.Generator("cuda").manual_seed(n)
        fluid = ~torch.as_tensor(solid)
        u = ((0.5 + 0.2 * (2 * torch.rand(3, n, n, n, generator=g) - 1)) / (dt * n)) * fluid
        d = torch.rand(n, n, n, generator=g) * fluid
        w = torch.randn(4, n, n, n, generator=g)
        gs = GasSolver(n, dt, 0.5, K, 1, solid)
        gs.set_state(u, d)
        gs.step(1)
        gu, gd = gs.state()
        if grad:
            gs.add_grad(w[:3], w[3])
            back = gs.backward()
        gs.close()
        ut, dt_ = u.double().requires_grad_(grad), d.double().requires_grad_(grad)
        with torch.set_grad_enabled(grad):
            u1, d1 = G.rollout(ut, dt_, solid, 1, dt, 0.5, K)
        assert _rel(gu, u1.detach()) <= 1e-4 and _rel(gd, d1.detach()) <= 1e-4
        if grad:
            want = torch.autograd.grad((u1 * w[:3]).sum() + (d1 * w[3]).sum(), (ut, dt_))
            assert _rel(back[0], want[0] * fluid) <= 1e-3 and _rel(back[1], want[1] * fluid) <= 1e-3
    torch.cuda.empty_cache()
