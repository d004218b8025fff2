"""Two gas solvers alive at once: creating one must not change what another can
launch. Each must give what it gives alone, the first time (graph capture) and from
the captured graphs. Same kernels on the same inputs: the only freedom is the order
of the FP64 sums of the forward (their FP32 mean can move by one rounding) and of
the FP32 atomics of the transposed advection, both of about 1e-7 relative."""
import numpy as np
import pytest
import torch

from gpu_util import rel
from paper_2303_02346_gb300.gas import GasSolver

pytestmark = pytest.mark.gpu


def _inputs(n):
    g = torch.Generator().manual_seed(n)
    u = 0.3 * torch.randn(3, n, n, n, generator=g)
    d = torch.rand(n, n, n, generator=g)
    solid = np.zeros((n, n, n), np.uint8)
    solid[n // 3:n // 2, n // 4:n // 2, n // 3:n // 2] = 1
    return solid, u.cuda(), d.cuda(), torch.randn(3, n, n, n, generator=g).cuda()


def _solver(n):
    return GasSolver(n, 0.005, 1.0, 3, 1, _inputs(n)[0])


def _pass(gs, n):
    _, u, d, w = _inputs(n)
    gs.set_state(u, d)
    gs.step(1)
    out = gs.state()
    gs.add_grad(w)
    return [t.cpu() for t in (*out, *gs.backward())]


# shared memory needed by a pair of sweeps, in bytes: 256: 188,416; 160: 117,760;
# 260: 179,920; 64 takes single sweeps
@pytest.mark.parametrize("first,second", [(256, 160), (260, 160), (160, 256), (256, 64)])
def test_solvers_side_by_side(first, second):
    alone = {}
    for n in (first, second):
        gs = _solver(n)
        alone[n] = _pass(gs, n)
        gs.close()
    solvers = [(n, _solver(n)) for n in (first, second)]
    for _ in range(2):
        for n, gs in solvers:
            for got, want in zip(_pass(gs, n), alone[n]):
                assert rel(got, want) <= 1e-5
    for _, gs in solvers:
        gs.close()
