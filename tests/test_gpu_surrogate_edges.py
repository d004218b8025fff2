"""Projection, lift backward and feature kernels at node counts that do not fill
a warp, a CTA or a grid stride (n^3 for odd n), single frames and batches
larger than one, against FP64 sums of the same BF16 inputs.

The network has one residual block with zero convolution weights and biases,
so h is the lifted frame exactly and every output is a sum over at most
2 x 29^3 nodes of products of BF16 values. Tolerance 1e-4 relative per block
of values: FP32 sums of n terms of mixed sign err by about sqrt(n) 6e-8 of
the terms' norm, below 2e-5 for these n; the BF16 rounding of h is applied to
the reference too, and FP32 and FP64 decide it differently for about 1.5e-5 of
the values, by 2^-8 each (1.5e-5 relative). Where a BF16-rounded gradient
enters as well: 1e-3."""
import numpy as np
import pytest
import torch

from gpu_util import rel
from paper_2303_02346_gb300.surrogate import Surrogate, param_count

pytestmark = pytest.mark.gpu


def _bf(t):
    return t.to(torch.bfloat16).double()


@pytest.mark.parametrize("n,batch", [(8, 1), (9, 3), (17, 2), (29, 2)])
def test_projection_and_lift_gradients(n, batch):
    g = torch.Generator().manual_seed(n)
    frames = torch.randn(2 * batch, n ** 3, 8, generator=g).to(torch.bfloat16)
    P = torch.zeros(param_count(blocks=1))
    P[:256] = torch.randn(256, generator=g) * 0.3
    P[256:288] = torch.randn(32, generator=g) * 0.3
    po = 288 + 2 * (27 * 1024 + 32)
    P[po:po + 96] = torch.randn(96, generator=g) * 0.3
    P[po + 96:] = torch.randn(3, generator=g)
    sur = Surrogate(n, 1.0, 1.0, max_batch=batch, blocks=1)
    sur.set_params(P.numpy())
    dev = frames.cuda().view(torch.int16)
    idx = torch.arange(batch, dtype=torch.int32, device="cuda")
    tgt = torch.arange(batch, 2 * batch, dtype=torch.int32, device="cuda")
    wl, bl, wp, bp = _bf(P[:256].reshape(32, 8)), P[256:288].double(), _bf(P[po:po + 96].reshape(3, 32)), P[po + 96:].double()
    f = frames[:batch].double()
    h = _bf((f @ wl.T + bl).float())
    pred = f[..., 1:4] + h @ wp.T + bp
    assert rel(sur.predict(dev, idx).cpu(), pred) <= 1e-4
    d = pred - frames[batch:].double()[..., 1:4]
    e = sur.eval(dev, idx, tgt)
    want = torch.sqrt((d ** 2).sum((1, 2)) / (frames[batch:].double()[..., 1:4] ** 2).sum((1, 2)))
    assert np.allclose(e, want.numpy(), rtol=1e-4)
    loss, grad, gf = sur.loss_grad(dev, idx, tgt, want_frame_grad=True)
    assert abs(loss - float((d ** 2).mean())) <= 1e-4 * float((d ** 2).mean())
    gp = 2 * d / d.numel()
    grad = grad.cpu().double()
    assert rel(grad[po:po + 96], torch.einsum("bvm,bvo->mo", gp, h).reshape(-1)) <= 1e-4
    assert rel(grad[po + 96:], gp.sum((0, 1))) <= 1e-3  # 3 sums that cancel to the mean difference
    gh = _bf((gp @ wp).float())
    assert rel(grad[:256], torch.einsum("bvo,bvq->oq", gh, f).reshape(-1)) <= 1e-3  # gh's own BF16 ties
    assert rel(gf.cpu()[..., :8], gh @ wl + torch.cat([torch.zeros_like(gp[..., :1]), gp, torch.zeros(batch, n ** 3, 4).double()], -1)) <= 1e-3
    w = torch.randn(batch, n ** 3, 3, generator=g)
    v = sur.vjp(dev, idx, w.cuda()).cpu()
    ref = _bf((w.double() @ wp).float()) @ wl
    ref[..., 1:4] += w.double()
    assert rel(v, ref) <= 1e-3
    sur.close()


@pytest.mark.parametrize("count,n", [(1, 8), (255, 9), (257, 16), (1000, 33)])
def test_features_and_adjoint(count, n):
    from oracle import surrogate as S
    r = np.random.default_rng(count)
    x = torch.tensor((1.0 + r.random((count, 3)) * (n - 3)) / n, dtype=torch.float32)
    v, C = torch.tensor(r.normal(size=(count, 3)), dtype=torch.float32), torch.tensor(r.normal(size=(count, 9)), dtype=torch.float32)
    mat = torch.tensor(r.integers(0, 4, count), dtype=torch.uint8)
    mm = [0.5, 1.0, 2.0, 3.0]  # the fourth material has no fraction channel
    sur = Surrogate(n, 0.7, 0.3, max_batch=1, blocks=1)
    mass = torch.tensor(mm)[mat.long()].double()
    for _ in range(2):  # the accumulation grid is clear again
        out = sur.empty_frames(1)
        sur.features(x.cuda(), v.cuda(), C.reshape(-1, 3, 3).cuda(), mat.cuda(), mm, out[0])
    got = out[0].view(torch.bfloat16).cpu().double()
    want = torch.as_tensor(S.grid_features(x.double(), v.double(), C.reshape(-1, 3, 3).double(), mat.long(), mass, n, 0.7, 0.3)).reshape(-1, 8)
    assert rel(got, want) <= 4e-3  # BF16 rounding: 2^-9 relative a value
    g = torch.tensor(r.normal(size=(n ** 3, 8)), dtype=torch.float32)
    gx, gv, gC = sur.features_vjp(x.cuda(), v.cuda(), C.reshape(-1, 3, 3).cuda(), mat.cuda(), mm, g.cuda())
    rx, rv, rC = S.features_vjp(x.double(), v.double(), C.reshape(-1, 3, 3).double(), mat.long(), mass, n, g.double(), 0.7, 0.3)
    assert rel(gx.cpu(), rx) <= 1e-4 and rel(gv.cpu(), rv) <= 1e-5 and rel(gC.cpu().reshape(-1), np.asarray(rC).reshape(-1)) <= 1e-4
    sur.close()
