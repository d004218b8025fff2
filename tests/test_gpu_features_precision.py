"""The feature transfer's adjoint on grids whose size is no power of two keeps the
precision of FP32: a particle's fractional position f = x n - base is rounded
once. Each weight then errs by about 2^-23 of itself, a product of three by
2e-7 with its own roundings, the sum over 27 nodes by as much again: 4e-7, and
7e-7 is asked for. Rounding x n before the subtraction errs by 1.4e-6 at n = 45."""
import pytest
import torch

from gpu_util import rel
from paper_2303_02346_gb300.surrogate import Surrogate

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 45, 50, 63, 64])
def test_adjoint_of_the_transfer(n):
    g = torch.Generator().manual_seed(n)
    N = 5000
    x = 0.2 + 0.6 * torch.rand(N, 3, generator=g)
    w = torch.randn(n ** 3, 8, generator=g)
    mat = torch.zeros(N, dtype=torch.uint8)
    sur = Surrogate(n, 1.0, 1.0, max_batch=1, blocks=1)
    zero = torch.zeros(N, 3, device="cuda")
    _, gv, gC = sur.features_vjp(x.cuda(), zero, torch.zeros(N, 9, device="cuda"), mat.cuda(), [1.0], w.cuda())
    xs = x.double() * n
    base = torch.floor(xs - 0.5)
    f, k = xs - base, base.long()
    W = (0.5 * (1.5 - f) ** 2, 0.75 - (f - 1.0) ** 2, 0.5 * (f - 0.5) ** 2)
    ev, eC = torch.zeros(N, 3).double(), torch.zeros(N, 3, 3).double()
    for o in torch.cartesian_prod(*[torch.arange(3)] * 3).tolist():
        i = ((k[:, 0] + o[0]) * n + k[:, 1] + o[1]) * n + k[:, 2] + o[2]
        t = (W[o[0]][:, 0] * W[o[1]][:, 1] * W[o[2]][:, 2])[:, None] * w[i, 1:4].double()
        ev += t
        eC += t[:, :, None] * ((torch.tensor(o).double() - f) / n)[:, None, :]
    assert rel(gv.cpu(), ev) <= 7e-7
    assert rel(gC.cpu().reshape(N, 3, 3), eC) <= 7e-7
    sur.close()
