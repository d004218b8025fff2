"""Lift and projection where their launches change form: as many nodes a frame as
threads (40^3) and more (41^3), a projection of one node a thread, of a few and of
eight, with cut-off last rounds. Networks whose convolutions are zero, weights and
frames of short binary fractions: every sum is exact in FP32, and the prediction
equals FP64's; the input gradient is rounded to BF16 on the way by the same rule, and
equals it too."""
import numpy as np
import pytest
import torch

from paper_2303_02346_gb300.surrogate import Surrogate

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [(8, 1), (13, 3), (40, 1), (40, 3), (41, 1), (47, 8), (64, 1), (64, 2)])
def test_exact_networks(n, batch):
    rng = np.random.default_rng(n + batch)
    short = lambda shape, unit, top: (rng.integers(-top, top + 1, shape) * unit).astype(np.float32)  # noqa: E731
    wl, bl, wp, bp = short((32, 8), 1 / 8, 4), short(32, 1 / 8, 4), short((3, 32), 1 / 16, 4), short(3, 1 / 16, 4)
    conv = np.zeros(2 * (27 * 1024 + 32), np.float32)
    sur = Surrogate(n, 1.0, 1.0, max_batch=batch, blocks=1)
    sur.set_params(np.concatenate([wl.ravel(), bl, conv, wp.ravel(), bp]))
    f = torch.tensor(short((batch, n ** 3, 8), 1 / 4, 4), device="cuda")
    frames = f.to(torch.bfloat16).view(torch.int16)
    idx = torch.arange(batch, dtype=torch.int32, device="cuda")
    wl, bl, wp, bp = (torch.tensor(a, dtype=torch.float64, device="cuda") for a in (wl, bl, wp, bp))
    h = (f.double() @ wl.T + bl).to(torch.bfloat16).double()
    want = f[..., 1:4].double() + h @ wp.T + bp
    assert torch.equal(sur.predict(frames, idx).double(), want)
    g = torch.tensor(short((batch, n ** 3, 3), 1 / 4, 4), device="cuda")
    gf = (g.double() @ wp).to(torch.bfloat16).double() @ wl
    gf[..., 1:4] += g.double()
    assert torch.equal(sur.vjp(frames, idx, g).double(), gf)
