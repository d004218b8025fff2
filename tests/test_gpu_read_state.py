"""State readback kernel: rows in the caller's order, whole and per scene, to
device and host buffers, at particle counts around a CTA's edge. Every value
is copied, so the comparisons are exact."""
import numpy as np
import pytest
import torch

import scenes
from paper_2303_02346_gb300 import binding as B
from paper_2303_02346_gb300.simulator import Simulator

pytestmark = pytest.mark.gpu


def _scene(counts, seed=7):
    n = 24
    rng = np.random.Generator(np.random.PCG64(seed))
    N = int(sum(counts))
    x = (6 + 12 * rng.random((N, 3))) / n
    vp = (1.0 / n) ** 3 / 8
    mats = [scenes.water_material(vp), scenes.von_mises_material(vp), scenes.viscous_material(vp)]
    return scenes.Scene(name="read", grid_n=n, dt=1e-4, n_steps=4, materials=mats, x=x, v=rng.normal(size=(N, 3)),
                        mat=rng.integers(0, 3, N).astype(np.uint8), scene_counts=[int(c) for c in counts],
                        checkpoint_every=2)


@pytest.mark.parametrize("counts", [(1,), (255, 0, 1), (256, 257), (513, 31, 0, 700)])
def test_rows_in_caller_order(counts):
    sc = _scene(counts)
    N, dev = sc.n_particles, "cuda"
    sim = Simulator(sc)
    g = torch.Generator().manual_seed(3)
    x, v = (torch.tensor(a, dtype=torch.float32, device=dev) for a in (sc.x, sc.v))
    C = torch.randn(N, 9, generator=g).to(dev)
    F = (torch.eye(3).reshape(1, 9) + 0.1 * torch.randn(N, 9, generator=g)).to(dev)
    mat = torch.tensor(sc.mat, device=dev)
    B.sim_set_state(sim.h, -1, x, v, C, F, mat)
    want_F = F.clone()
    liquid = mat != 1
    want_F[liquid, 1:] = torch.eye(3, device=dev).reshape(-1)[1:]
    # step 0 (caller order in the library), then the same state after the library sorted it
    for _ in range(2):
        gx, gv, gC, gF = sim.state(with_CF=True, step=0)
        assert torch.equal(gx, x) and torch.equal(gv, v)
        assert torch.equal(gC.reshape(N, 9), C) and torch.equal(gF.reshape(N, 9), want_F)
        sim.step(3 if sim.current_step == 0 else 0)
    # a checkpoint and the current state: scenes are slices of the whole, host buffers equal device ones
    for step in (2, -1):
        whole = sim.state(with_CF=True, step=step)
        lo = 0
        for s, cnt in enumerate(counts):
            part = sim.state(scene=s, with_CF=True, step=step)
            for a, b in zip(part, whole):
                assert torch.equal(a, b[lo:lo + cnt])
            lo += cnt
        host = [np.zeros((N, 3), np.float32), None, np.zeros((N, 9), np.float32), np.zeros((N, 9), np.float32)]
        B.sim_get_state(sim.h, -1, step, *host)
        for a, b in zip(host, whole):
            if a is not None:
                assert np.array_equal(a.reshape(-1), b.cpu().numpy().reshape(-1))
    assert torch.equal(whole[3].reshape(N, 9)[liquid, 1:], want_F[liquid, 1:])
    sim.close()
