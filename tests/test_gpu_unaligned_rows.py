"""Caller's device rows at addresses that are no multiple of 4: copies take them, kernels
do not, so they go through the library's own buffer. Values are those of aligned
rows; gradients differ by the order of FP32 atomics alone (1e-5, water)."""
import ctypes

import numpy as np
import pytest
import torch

import scenes
from gpu_util import rel
from paper_2303_02346_gb300 import binding as B
from paper_2303_02346_gb300.simulator import Simulator

pytestmark = pytest.mark.gpu


def _off(floats, shift, values=None):
    """(buffer, pointer into it `shift` bytes past a multiple of 4) for `floats` floats."""
    buf = torch.zeros(4 * floats + 8, dtype=torch.uint8, device="cuda")
    if values is not None:
        buf[shift:shift + 4 * floats] = values.contiguous().view(torch.uint8).reshape(-1)
    return buf, ctypes.c_void_p(buf.data_ptr() + shift)


def _back(buf, shift, floats):
    return buf[shift:shift + 4 * floats].clone().view(torch.float32).cpu().numpy()


@pytest.mark.parametrize("shift", [1, 2])
def test_rows_at_any_address(shift):
    sc = scenes.small_block(3, 24, (scenes.LIQUID,), ppc=4, size_cells=5, spin=1.0, n_steps=4)
    N = sc.n_particles
    x, v = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in (sc.x, sc.v))
    mat = torch.tensor(sc.mat, device="cuda")
    ref = Simulator(sc, checkpoint_every=2)
    ref.reset()
    ref.step(4)
    want = [t.cpu().numpy().ravel() for t in ref.state(with_CF=True)]
    ref.position_loss(sc.loss["target"])
    want_g = [t.cpu().numpy().ravel() for t in ref.backward()[:2]]
    lib = B.load()
    sim = Simulator(sc, checkpoint_every=2)
    xb, xp = _off(3 * N, shift, x)
    vb, vp = _off(3 * N, shift, v)
    assert lib.sim_set_particles(sim.h, -1, xp, vp, ctypes.c_void_p(mat.data_ptr()), 1) == 0
    x0 = sim.state(step=0)
    assert torch.equal(x0[0], x) and torch.equal(x0[1], v)
    sim.step(4)
    sizes = (3 * N, 3 * N, 9 * N, 9 * N)
    outs = [_off(k, shift) for k in sizes]
    assert lib.sim_get_state(sim.h, -1, -1, *(p for _, p in outs), 1) == 0
    aligned = [t.cpu().numpy().ravel() for t in sim.state(with_CF=True)]
    for (buf, _), k, a, w in zip(outs, sizes, aligned, want):
        got = _back(buf, shift, k)
        assert np.array_equal(got, a) and rel(got, w) <= 1e-5
    # one aligned and one not
    fine = torch.empty(N, 3, device="cuda")
    buf, p = _off(3 * N, shift)
    assert lib.sim_get_state(sim.h, -1, -1, ctypes.c_void_p(fine.data_ptr()), p, None, None, 1) == 0
    assert np.array_equal(fine.cpu().numpy().ravel(), aligned[0]) and np.array_equal(_back(buf, shift, 3 * N), aligned[1])
    sim.position_loss(sc.loss["target"])
    outs = [_off(3 * N, shift) for _ in range(2)]
    assert lib.sim_backward(sim.h, outs[0][1], outs[1][1], None, 1) == 0
    for (buf, _), w in zip(outs, want_g):
        assert rel(_back(buf, shift, 3 * N), w) <= 1e-5
    sim.close()
    ref.close()
