"""The rounding of the projection's weight gradient. One frame with the same values at
every node, networks whose convolutions are zero: features, prediction and its
cotangent are the same at every node and exactly known (short binary fractions; the
cotangent is one FP32 product, repeated here), so that the sum over the nodes is all
that rounds, by the same amount in the same direction wherever it is a long chain.
n^3 nodes fit one CTA. Roundings on the way to an entry: 2 of products, 4 over 32
nodes, 8 of a warp's blocks, 8 over the CTA, 22 of 2^-24 in all."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2303_02346_gb300.surrogate import Surrogate

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 11, 12])
def test_sum_over_equal_nodes(n):
    rng = np.random.default_rng(n)
    f = np.array([0.5, -0.75, 1.25, 0.375, 1.0, 0.0, 0.0, 0.0], np.float32)
    t = np.array([0.0, 0.125, -0.5, 1.0, 0.0, 0.0, 0.0, 0.0], np.float32)
    wl = rng.integers(-8, 9, (32, 8)).astype(np.float32) / 8
    wp = rng.integers(-8, 9, (3, 32)).astype(np.float32) / 64
    h = torch.tensor(wl @ f).to(torch.bfloat16).float().numpy()  # products of short fractions: exact in FP32
    conv = np.zeros(27 * 1024 + 32, np.float32)
    sur = Surrogate(n, 1.0, 1.0, max_batch=1, blocks=1)
    sur.set_params(np.concatenate([wl.ravel(), np.zeros(32, np.float32), conv, conv, wp.ravel(), np.zeros(3, np.float32)]))
    both = torch.tensor(np.stack([f, t])).to(torch.bfloat16)[:, None].expand(2, n ** 3, 8).contiguous()
    idx = torch.tensor([0], dtype=torch.int32, device="cuda")
    _, grad, _ = sur.loss_grad(both.cuda().view(torch.int16), idx, idx + 1)
    got = grad.cpu().numpy()[-99:-3].reshape(3, 32)
    d = f[1:4] + wp @ h - t[1:4]
    assert np.array_equal(d, f[1:4].astype(np.float64) + wp.astype(np.float64) @ h - t[1:4])
    inv = np.float32(1) / (np.float32(1) * np.float32(n ** 3) * np.float32(3))
    gp = np.float32(2) * d * inv
    for m in range(3):
        for o in range(32):
            want = n ** 3 * Fraction(float(gp[m])) * Fraction(float(h[o]))
            assert abs(Fraction(float(got[m, o])) - want) <= abs(want) * 22 * Fraction(1, 2 ** 24), (m, o)
