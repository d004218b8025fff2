"""Performance cases: the work that users of this library have it do, each
through the public entry points.

A case is a dict of plain values. `listed()` gives the fixed ones, `draw(rng)`
one more of the same ranges, `prepare(case, seed)` what a program holds before
the call, `run(state)` one pass, `work(case)` the bytes and operations a pass
cannot do without, and `exact(case, seed)` the same outputs in 64 bits by plain
torch.

Kinds:
  mpm       one optimisation iteration or rollout of the particle simulator: set
            the initial state (and tool), step, read the state, and with
            every > 0 a loss and the reverse sweep
  surrogate the convolutional grid operator: predict / parameter gradient /
            training step / input gradient
  features  particle state -> surrogate frame, and the adjoint of that transfer
  gas       the grid gas solver, forward and adjoint
  sharing   attraction loss (with its gradient carried through the step) and
            gradient sharing over the particles of a fluid body
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

import scenes
from paper_2303_02346_gb300 import binding
from paper_2303_02346_gb300.gas import GasSolver
from paper_2303_02346_gb300.simulator import Simulator, rollout
from paper_2303_02346_gb300.surrogate import Surrogate, frame_scales, init_params, param_count, particle_masses

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # smallest optimisation iteration: the 8,192-particle water cube pushed
        # onto the floor, through torch.autograd; launches and latency
        dict(name="water_8k_grad", kind="mpm", scene="water", grid=32, cells=8, ppc=16, steps=50, every=50),
        # one control frame of a candidate action: 10 substeps of a task-sized
        # scene (100k particles, 64^3), forward only, state read back
        dict(name="frame_100k", kind="mpm", scene="tool", grid=64, particles=100_000, steps=10, every=0),
        # every other material (von Mises, box yield, viscous, particle-made
        # rigid body) beside water, odd grid, short horizon, gradients
        dict(name="mixed_55k_grad", kind="mpm", scene="mixed", grid=50, cells=19, ppc=8, steps=30, every=10),
        # trajectory optimisation of the tool: 200k particles of three materials,
        # 200 steps, grid-mass loss, gradient w.r.t. the actions
        dict(name="tool_200k_grad", kind="mpm", scene="tool", grid=128, particles=200_000, steps=200, every=20),
        # many environments of uneven sizes in one handle, gradients
        dict(name="batch_64_grad", kind="mpm", scene="batch", grid=64, scenes=64, low=10_000, high=150_000,
             steps=40, every=20),
        # largest: 2M-particle dam break, four checkpoint intervals
        dict(name="dam_2m_grad", kind="mpm", scene="dam", grid=256, particles=2_000_000, steps=100, every=25),
        # the same scene rolled out without gradients (data generation, preview)
        dict(name="dam_2m_rollout", kind="mpm", scene="dam", grid=256, particles=2_000_000, steps=40, every=0),
        # surrogate inference for a batch of scenes
        dict(name="surrogate_predict", kind="surrogate", op="predict", grid=64, batch=8, blocks=4),
        # surrogate training: loss and parameter gradient of a minibatch
        dict(name="surrogate_grad", kind="surrogate", op="grad", grid=64, batch=8, blocks=4),
        # training data and warm starts: one frame of a task-sized scene and the
        # adjoint of the transfer
        dict(name="features_100k", kind="features", grid=64, particles=100_000),
        # gas: smoke simulation at the solver's usual size, and its adjoint
        dict(name="gas_256_grad", kind="gas", grid=256, sweeps=60, steps=4),
        # gradient sharing within a fluid body
        dict(name="sharing_195k", kind="sharing", grid=64, cells=29, ppc=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mpm", "mpm", "mpm", "surrogate", "features", "gas", "sharing"])
    if kind == "surrogate":
        return dict(kind=kind, op=rng.choice(["predict", "grad", "train", "vjp"]), grid=rng.randint(24, 64),
                    batch=rng.randint(1, 8), blocks=rng.randint(1, 4))
    if kind == "features":
        grid = rng.randint(32, 64)
        return dict(kind=kind, grid=grid, particles=_log_int(rng, 3000, 150_000 * (grid / 64) ** 3))
    if kind == "gas":
        return dict(kind=kind, grid=_log_int(rng, 24, 256), sweeps=rng.randint(10, 60), steps=rng.randint(1, 4))
    if kind == "sharing":
        grid = rng.randint(32, 72)
        return dict(kind=kind, grid=grid, cells=rng.randint(6, grid // 2), ppc=rng.choice([4, 8, 12]))
    scene = rng.choice(["water", "mixed", "tool", "batch", "dam"])
    steps = rng.randint(4, 100)
    every = rng.choice([0, steps, rng.randint(3, 25)])
    if every > 25 and scene in ("batch", "dam"):
        every = 25
    if scene in ("water", "mixed"):
        grid = rng.randint(24, 72)
        return dict(kind=kind, scene=scene, grid=grid, cells=rng.randint(6, grid // 2), ppc=rng.choice([2, 4, 8, 16]),
                    steps=min(steps, 40) if scene == "mixed" else steps, every=every)
    if scene == "tool":
        grid = rng.choice([64, 80, 96, 110, 128])
        return dict(kind=kind, scene=scene, grid=grid, particles=_log_int(rng, 8000, 200_000 * (grid / 128) ** 1.5),
                    steps=steps, every=every)
    if scene == "batch":
        low = _log_int(rng, 3000, 30_000)
        return dict(kind=kind, scene=scene, grid=64, scenes=_log_int(rng, 2, 48), low=low,
                    high=_log_int(rng, low, 120_000), steps=min(steps, 40), every=every)
    grid = rng.choice([64, 90, 128, 192, 256])
    most = 2_000_000 * (grid / 256) ** 3
    return dict(kind=kind, scene=scene, grid=grid, particles=_log_int(rng, most / 10, most), steps=steps, every=every)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
MIXED = (scenes.LIQUID, scenes.VON_MISES, scenes.BOX_YIELD, scenes.VISCOUS_LIQUID, scenes.RIGID)


def _scene(case, seed):
    n, what = case["grid"], case.get("scene", "tool")
    steps, every = case.get("steps", 1), case.get("every", 1)
    if what in ("water", "mixed"):
        lo = ((n - case["cells"]) // 2, 3, (n - case["cells"]) // 2)
        kinds = (scenes.LIQUID,) if what == "water" else MIXED
        sc = scenes.small_block(seed, n, kinds, ppc=case["ppc"], lo_cell=lo, size_cells=case["cells"],
                                v0=(0.2, -1.0, 0.1), spin=1.0, n_steps=steps)
        sc.checkpoint_every = every
        return sc
    if what == "tool":
        return scenes.multi_material(seed, scale=case["particles"] / 200_000, n_steps=steps, grid_n=n,
                                     checkpoint_every=every)
    if what == "batch":
        # the same sizes for every seed; placement and motion differ
        sc = scenes.batched_scenes(3, n_scenes=case["scenes"], grid_n=n, n_steps=steps, lo=case["low"], hi=case["high"])
        r = np.random.Generator(np.random.PCG64(seed))
        sc.x = sc.x + r.uniform(-0.3, 0.3, sc.x.shape) / n
        sc.tool_actions = sc.tool_actions * r.uniform(0.5, 1.0, (case["scenes"], 1, 6))
        return sc
    return scenes.dam_break(seed, scale=case["particles"] / 2_000_000, grid_n=n, n_steps=steps,
                            checkpoint_every=every)


def _dev(a, dtype=torch.float32):
    return torch.tensor(np.asarray(a), dtype=dtype, device=DEV).contiguous()


def _mpm_inputs(case, seed):
    sc = _scene(case, seed)
    s = dict(scene=sc, x=_dev(sc.x), v=_dev(sc.v), mat=_dev(sc.mat, torch.uint8))
    if sc.tool_enabled:
        s.update(pose=_dev(sc.tool_pose0), actions=_dev(sc.tool_actions))
    loss = sc.loss
    if loss["kind"] == "grid_mass":
        s.update(tm=_dev(loss["target_mass"]), td=_dev(loss["target_dist"]), total=float(loss["total_mass"]))
    else:
        s.update(target=tuple(float(t) for t in loss["target"]))
    return s


def _smooth_velocity(x, seed, amp=0.3):
    """Smooth velocity field at the points x and its gradient (the affine
    velocity of a particle in it)."""
    g = torch.Generator().manual_seed(seed)
    kv = (2 * math.pi * torch.randint(1, 3, (3, 3), generator=g)).to(x)
    ph = (2 * math.pi * torch.rand(3, generator=g)).to(x)
    arg = x @ kv.T + ph
    return amp * torch.sin(arg), amp * torch.cos(arg)[:, :, None] * kv[None]


def _layout(grid, particles, seed):
    sc = scenes.multi_material(seed, scale=particles / 200_000, n_steps=1, grid_n=grid)
    x = _dev(sc.x)
    v, C = _smooth_velocity(x, seed)
    return sc, x, v, C, _dev(sc.mat, torch.uint8)


def _surrogate_inputs(case, seed):
    """Frames of three-material scenes in smooth motion and, as targets, the
    frames of the same particles ten steps on."""
    n, batch = case["grid"], case["batch"]
    frames = torch.zeros(2 * batch, n ** 3, 8, dtype=torch.bfloat16, device=DEV)
    for b in range(batch):
        count = max(500, int(min(60_000, n ** 3 / 5) * (0.3 + 0.7 * (b + 1) / batch)))
        sc, x, v, C, mat = _layout(n, count, 1000 * seed + b)
        m_ref, v_ref = frame_scales(sc)
        later = (x + 1e-3 * v).clamp(1.6 / n, 1 - 2.6 / n)
        for k, xx in ((b, x), (batch + b, later)):
            frames[k] = _frame(xx.double(), v.double(), C.double(), mat.long(), particle_masses(sc), n, m_ref,
                               v_ref).to(torch.bfloat16)
    g = torch.Generator().manual_seed(seed)
    return dict(frames=frames, m_ref=m_ref, v_ref=v_ref, params=init_params(seed, blocks=case["blocks"]),
                idx=torch.arange(batch, dtype=torch.int32, device=DEV),
                tgt=torch.arange(batch, 2 * batch, dtype=torch.int32, device=DEV),
                g_pred=torch.randn(batch, n ** 3, 3, generator=g).to(DEV))


def _gas_inputs(case, seed):
    n = case["grid"]
    r = np.random.Generator(np.random.PCG64(seed))
    solid = np.zeros((n, n, n), np.uint8)
    a, b = int(0.4 * n), max(int(0.55 * n), int(0.4 * n) + 1)
    solid[a:b, a - n // 8:b - n // 8, a:b] = 1
    c = (torch.arange(n, device=DEV, dtype=torch.float32) + 0.5) / n
    x = torch.stack(torch.meshgrid(c, c, c, indexing="ij"), -1).reshape(-1, 3)
    u = _smooth_velocity(x, seed, 1.0)[0].T.reshape(3, n, n, n).contiguous()
    at = torch.tensor([0.5, 0.2, 0.5] + r.uniform(-0.05, 0.05, 3), dtype=torch.float32, device=DEV)
    d = torch.exp(-((x - at) ** 2).sum(-1) / 0.02).reshape(n, n, n).contiguous()
    gu = _smooth_velocity(x, seed + 1, 1.0)[0].T.reshape(3, n, n, n).contiguous()
    gd = _smooth_velocity(x, seed + 2, 1.0)[0][:, 0].reshape(n, n, n).contiguous()
    return dict(solid=solid, u=u, d=d, gu=gu, gd=gd, dt=0.01, buoyancy=2.0)


def _sharing_inputs(case, seed):
    s = _mpm_inputs(dict(case, scene="water", steps=1, every=1), seed)
    g = torch.Generator().manual_seed(seed)
    N = s["x"].shape[0]
    s.update(ell=torch.rand(N, generator=g).to(DEV), g=torch.randn(N, 3, generator=g).to(DEV),
             radius=0.8 / case["grid"], tau=0.5)
    return s


# ----------------------------------------------------------------------------
# preparation and one pass
# ----------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "mpm":
        s = _mpm_inputs(case, seed)
        s["sim"] = Simulator(s["scene"], checkpoint_every=case["every"], max_steps=case["steps"])
        if case["scene"] == "water":
            s["x"].requires_grad_(case["every"] > 0)
            s["v"].requires_grad_(case["every"] > 0)
    elif kind == "surrogate":
        s = _surrogate_inputs(case, seed)
        s["frames"] = s["frames"].view(torch.int16)
        s["sur"] = Surrogate(case["grid"], s["m_ref"], s["v_ref"], max_batch=case["batch"], blocks=case["blocks"])
        s["sur"].set_params(s["params"])
    elif kind == "features":
        sc, x, v, C, mat = _layout(case["grid"], case["particles"], seed)
        m_ref, v_ref = frame_scales(sc)
        g = torch.Generator().manual_seed(seed)
        s = dict(x=x, v=v, C=C, mat=mat, mass=particle_masses(sc), g=torch.randn(case["grid"] ** 3, 8, generator=g).to(DEV),
                 sur=Surrogate(case["grid"], m_ref, v_ref, max_batch=1))
    elif kind == "gas":
        s = _gas_inputs(case, seed)
        s["gas"] = GasSolver(case["grid"], s["dt"], s["buoyancy"], case["sweeps"], case["steps"], s["solid"])
    else:
        s = _sharing_inputs(case, seed)
        s["sim"] = Simulator(s["scene"], checkpoint_every=1, max_steps=1)
        s["sim"].set_particles(s["x"], s["v"], s["mat"])
        s["sim"].step(1)
    s["case"] = dict(case)
    return s


def run(s):
    return _RUN[s["case"]["kind"]](s)


def _run_mpm(s):
    case, sim, sc = s["case"], s["sim"], s["scene"]
    if case["scene"] == "water" and case["every"] > 0:
        # through torch.autograd
        x, v = rollout(sim, case["steps"], s["x"], s["v"])
        loss = ((x - torch.tensor(s["target"], device=DEV)) ** 2).sum()
        gx, gv = torch.autograd.grad(loss, (s["x"], s["v"]))
        return dict(x=x.detach(), v=v.detach(), loss=loss.detach(), gx=gx, gv=gv)
    sim.set_particles(s["x"], s["v"], s["mat"])
    if sc.tool_enabled:
        sim.set_tool(s["pose"], s["actions"])
    sim.step(case["steps"])
    x, v = sim.state()
    if case["every"] == 0:
        return dict(x=x, v=v)
    if "tm" in s:
        loss = binding.sim_grid_mass_loss(sim.h, 0, s["tm"], s["td"], s["total"])  # targets held on the device
    else:
        loss = torch.as_tensor(sim.position_loss(s["target"]), dtype=torch.float32)
    gx, gv, ga = sim.backward()
    return dict(x=x, v=v, loss=loss, gx=gx, gv=gv, ga=ga)


def _run_surrogate(s):
    sur, op = s["sur"], s["case"]["op"]
    if op == "predict":
        return dict(pred=sur.predict(s["frames"], s["idx"]))
    if op == "vjp":
        return dict(g_frames=sur.vjp(s["frames"], s["idx"], s["g_pred"]))
    if op == "grad":
        loss, grad, _ = sur.loss_grad(s["frames"], s["idx"], s["tgt"])
        return dict(loss=loss, grad=grad)
    sur.set_params(s["params"])
    loss = sur.train_step(s["frames"], s["idx"], s["tgt"], 1e-5)
    return dict(loss=loss, params=sur.get_params())


def _run_features(s):
    sur = s["sur"]
    frame = sur.empty_frames(1)
    sur.features(s["x"], s["v"], s["C"], s["mat"], s["mass"], frame[0])
    gx, gv, gC = sur.features_vjp(s["x"], s["v"], s["C"], s["mat"], s["mass"], s["g"])
    return dict(frame=frame[0].view(torch.bfloat16), gx=gx, gv=gv, gC=gC)


def _run_gas(s):
    gas = s["gas"]
    gas.set_state(s["u"], s["d"])
    gas.step(s["case"]["steps"])
    u, d = gas.state()
    gas.add_grad(s["gu"], s["gd"])
    gu, gd = gas.backward()
    return dict(u=u, d=d, gu=gu, gd=gd)


def _run_sharing(s):
    sim = s["sim"]
    loss = sim.attraction_loss(s["ell"], s["radius"], s["tau"])
    gx, gv, _ = sim.backward(want_actions=False)
    shared = sim.share_gradients(s["ell"], s["g"], s["radius"], s["tau"])
    return dict(loss=loss, gx=gx, gv=gv, shared=shared)


_RUN = dict(mpm=_run_mpm, surrogate=_run_surrogate, features=_run_features, gas=_run_gas, sharing=_run_sharing)


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
def _particles(case):
    if case.get("scene") == "batch":
        # mean of the log-uniform sizes
        lo, hi = case["low"], case["high"]
        return case["scenes"] * ((hi - lo) / math.log(hi / lo) if hi > lo else lo)
    return case["particles"] if "particles" in case else case["cells"] ** 3 * case["ppc"]


# share of particles that carry a whole deformation gradient
SOLID = dict(water=0.0, mixed=0.6, tool=0.5, batch=0.5, dam=0.3)


def work(case):
    """MPM, per particle and step: forward, x and J (solids: F) read and
    written (32 / 96 B); with gradients also the record the reverse sweep needs
    (x, v, C, J; solids F) written and read and the adjoint state (as the
    state) read and written. About 700 operations per particle and step
    forward (27 nodes, two transfers), 1,600 backward; solids 500 more."""
    kind, n = case["kind"], case["grid"]
    if kind == "mpm":
        N, f = _particles(case), SOLID[case["scene"]]
        b, o = 32 + 64 * f, 700 + 500 * f
        if case["every"]:
            b += 2 * (64 + 36 * f) + 32 + 64 * f
            o += 1600 + 500 * f
        return dict(bytes=N * case["steps"] * b + 50 * N, flops=N * case["steps"] * o)
    if kind == "surrogate":
        nodes, conv = case["batch"] * n ** 3, 2 * 27 * 32 * 32
        layers = 2 * case["blocks"]
        times = {"predict": 1, "vjp": 2, "grad": 3, "train": 3}[case["op"]]
        p = 4 * param_count(blocks=case["blocks"])
        io = 16 + {"predict": 12, "vjp": 12 + 32, "grad": 16, "train": 16}[case["op"]]
        return dict(bytes=nodes * io + p * (1 + (times == 3)), flops=nodes * (times * layers * conv + 700))
    if kind == "features":
        N = _particles(case)
        return dict(bytes=N * (61 + 61 + 60) + n ** 3 * (16 + 32), flops=N * 27 * 80)
    if kind == "gas":
        c = n ** 3 * case["steps"]
        return dict(bytes=2 * c * (32 + case["sweeps"] * 13), flops=2 * c * (200 + 12 * case["sweeps"]))
    N = _particles(case)
    near = 27 * case["ppc"]
    return dict(bytes=N * (28 + 16 + 24 + 28 + 12), flops=N * (2 * near * 15 + 2300))


# ----------------------------------------------------------------------------
# the same outputs in 64 bits
# ----------------------------------------------------------------------------
def exact(case, seed):
    return _EXACT[case["kind"]](case, seed)


def _spline(x, n):
    """Stencil origin, fractional position and quadratic B-spline weights."""
    xs = x * n
    base = torch.floor(xs - 0.5).detach()
    f = xs - base
    return base.long(), f, (0.5 * (1.5 - f) ** 2, 0.75 - (f - 1.0) ** 2, 0.5 * (f - 0.5) ** 2)


OFFSETS = [(a, b, c) for a in range(3) for b in range(3) for c in range(3)]


def _nodes(base, f, w, n):
    """For each of the 27 stencil nodes: weight, offset from the particle, index."""
    for o in OFFSETS:
        k = base + torch.tensor(o, device=base.device)
        yield (w[o[0]][:, 0] * w[o[1]][:, 1] * w[o[2]][:, 2], (torch.tensor(o, dtype=F64, device=f.device) - f) / n,
               (k[:, 0] * n + k[:, 1]) * n + k[:, 2])


def _momentum(x, v, C, mat, mass, n):
    m, p = mass[mat], torch.zeros(n ** 3, 4, dtype=F64, device=x.device)
    for W, d, i in _nodes(*_spline(x, n), n):
        p = p.index_add(0, i, (W * m)[:, None] * torch.cat([torch.ones_like(W)[:, None], v + torch.einsum("pij,pj->pi", C, d)], 1))
    return p


def _frame(x, v, C, mat, mass, n, m_ref, v_ref):
    mass = torch.tensor(mass, dtype=F64, device=x.device)
    p = _momentum(x, v, C, mat, mass, n)
    phi = torch.zeros(n ** 3, 3, dtype=F64, device=x.device)
    for W, _, i in _nodes(*_spline(x, n), n):
        phi.index_put_((i, mat), W.detach() * mass[mat], accumulate=True)
    phi = phi / p[:, :1].detach().clamp_min(1e-300)
    return torch.cat([p[:, :1] / m_ref, p[:, 1:] / (m_ref * v_ref), phi, torch.zeros_like(phi[:, :1])], 1)


def _svd(F):
    """U, sigma, V of 3x3 matrices of positive determinant, by Jacobi rotations
    of F^T F."""
    A, V = F.transpose(1, 2) @ F, torch.eye(3, dtype=F64, device=F.device).expand_as(F).clone()
    for _ in range(6):
        for p, q in ((0, 1), (0, 2), (1, 2)):
            d, e = A[:, q, q] - A[:, p, p], 2 * A[:, p, q]
            t = torch.where(d >= 0, e, -e) / (d.abs() + torch.sqrt(d * d + e * e)).clamp_min(1e-300)
            c = 1 / torch.sqrt(1 + t * t)
            s = t * c
            G = torch.eye(3, dtype=F64, device=F.device).repeat(F.shape[0], 1, 1)
            G[:, p, p], G[:, q, q], G[:, p, q], G[:, q, p] = c, c, s, -s
            A, V = G.transpose(1, 2) @ A @ G, V @ G
    sig = torch.sqrt(torch.diagonal(A, dim1=1, dim2=2).clamp_min(0))
    return (F @ V) / sig[:, None, :], sig, V


def _eig(U, d, W):
    return (U * d[:, None, :]) @ W.transpose(1, 2)


def _corotated(sig, mu, lam):
    J = sig.prod(1, keepdim=True)
    return 2 * mu * (sig - 1) * sig + lam * J * (J - 1)


def _stress(M, F, C, dt):
    """Projected F and Kirchhoff stress of one material's particles (F of a
    liquid: diag(J, 1, 1))."""
    eye = torch.eye(3, dtype=F64, device=F.device)
    if M.kind == scenes.LIQUID:
        J = F[:, 0, 0]
        return F, (M.bulk * J * (J - 1))[:, None, None] * eye
    if M.kind == scenes.RIGID:
        return F, torch.zeros_like(F)
    if M.kind == scenes.VISCOUS_LIQUID:
        G = eye + dt * C
        U, sig, _ = _svd((F[:, 0, 0] / torch.linalg.det(G)).pow(1 / 3)[:, None, None] * G)
        return F, _eig(U, _corotated(sig, M.shear, M.bulk), U)
    mu, lam = M.E / (2 * (1 + M.nu)), M.E * M.nu / ((1 + M.nu) * (1 - 2 * M.nu))
    U, sig, V = _svd(F)
    if M.kind == scenes.BOX_YIELD:
        s = sig.clamp(1 - M.crit_compress, 1 + M.crit_stretch)
        return _eig(U, s, V), _eig(U, _corotated(s, mu, lam), U)
    eps = torch.log(sig.clamp_min(1e-4))
    tr = eps.sum(1, keepdim=True)
    dev = eps - tr / 3
    nrm = dev.norm(dim=1, keepdim=True)
    u = dev / nrm.clamp_min(1e-300)
    if M.kind == scenes.VON_MISES:
        ky = M.yield_stress / (2 * mu)
        s = torch.where(nrm > ky, torch.exp(tr / 3 + ky * u), sig)
        return _eig(U, s, V), _eig(U, _corotated(s, mu, lam), U)
    sp = math.sin(math.radians(M.friction_deg))
    dg = nrm + math.sqrt(2 / 3) * 2 * sp / (3 - sp) * (3 * lam + 2 * mu) / (2 * mu) * tr
    ep = torch.where(dg <= 0, eps, torch.where((tr > 0) | (nrm == 0), torch.zeros_like(eps), eps - dg * u))
    return _eig(U, torch.where(dg <= 0, sig, torch.exp(ep)), V), _eig(U, 2 * mu * ep + lam * ep.sum(1, keepdim=True), U)


def _quat_mul(a, b):
    return torch.stack([a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3],
                        a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2],
                        a[0] * b[2] - a[1] * b[3] + a[2] * b[0] + a[3] * b[1],
                        a[0] * b[3] + a[1] * b[2] - a[2] * b[1] + a[3] * b[0]])


def _rotation(q):
    w, x, y, z = q
    return torch.stack([torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)]),
                        torch.stack([2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)]),
                        torch.stack([2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)])])


def _contact(sc, u, xi, pose, act):
    """Soft Coulomb contact of node velocities with the box tool."""
    R, half = _rotation(pose[3:]), torch.tensor(sc.tool_half, dtype=F64, device=u.device)
    r = xi - pose[:3]
    y = r @ R
    sgn = torch.where(y >= 0, 1.0, -1.0).to(F64)
    e = y.abs() - half
    ep = e.clamp_min(0)
    nrm = ep.norm(dim=1, keepdim=True)
    inside = torch.nn.functional.one_hot(e.argmax(1), 3).to(F64)
    out = nrm > 0
    phi = torch.where(out, nrm, e.max(1, keepdim=True).values)
    nn = torch.where(out, sgn * ep / nrm.clamp_min(1e-300), sgn * inside) @ R.T
    vT = act[:3] + torch.linalg.cross(act[3:].expand_as(r), r)
    vr = u - vT
    vn = (vr * nn).sum(1, keepdim=True)
    t = vr - vn * nn
    tn = t.norm(dim=1, keepdim=True)
    slide = torch.where(tn <= -sc.friction * vn, torch.zeros_like(t), t * (1 + sc.friction * vn / tn.clamp_min(1e-300)))
    alpha = torch.exp(-phi / sc.contact_soft).clamp_max(1.0)
    return torch.where((phi < sc.contact_eps) & (vn < 0), alpha * (vT + slide) + (1 - alpha) * u, u)


def _rollout(s, steps, x, v):
    """Positions and velocities after `steps` steps from (x, v) in 64 bits."""
    sc, mat = s["scene"], s["mat"].long()
    n, dt, S, dev = sc.grid_n, sc.dt, sc.n_scenes, x.device
    eye = torch.eye(3, dtype=F64, device=dev)
    own = torch.repeat_interleave(torch.arange(S, device=dev), torch.tensor(sc.scene_counts, device=dev)) * n ** 3
    mass = torch.tensor([m.rho * m.volume for m in sc.materials], dtype=F64, device=dev)[mat]
    vol = torch.tensor([m.volume for m in sc.materials], dtype=F64, device=dev)[mat]
    C, F = torch.zeros(len(x), 3, 3, dtype=F64, device=dev), eye.repeat(len(x), 1, 1)
    groups = [(M, torch.nonzero(mat == k)[:, 0]) for k, M in enumerate(sc.materials)]
    liquid = torch.zeros_like(mat, dtype=torch.bool)
    rest = {}
    for k, (M, at) in enumerate(groups):
        if M.kind in (scenes.LIQUID, scenes.VISCOUS_LIQUID):
            liquid[at] = True
        if M.kind == scenes.RIGID:
            rest[k] = x[at] - (mass[at][:, None] * x[at]).sum(0) / mass[at].sum()
    if sc.tool_enabled:
        pose, actions = s["pose"].to(F64).clone(), s["actions"].to(F64)
    gravity = torch.tensor(sc.gravity, dtype=F64, device=dev)
    for t in range(steps):
        Fp, tau = F, torch.zeros_like(F)
        for M, at in groups:
            if len(at):
                a, b = _stress(M, F[at], C[at], dt)
                Fp, tau = Fp.index_copy(0, at, a), tau.index_copy(0, at, b)
        A = (-dt * 4 * n * n) * vol[:, None, None] * tau + mass[:, None, None] * C
        p = torch.zeros(S * n ** 3, 4, dtype=F64, device=dev)
        stencil = _spline(x, n)
        for W, d, i in _nodes(*stencil, n):
            q = torch.cat([mass[:, None], mass[:, None] * v + torch.einsum("pij,pj->pi", A, d)], 1)
            p = p.index_add(0, i + own, W[:, None] * q)
        act = torch.nonzero(p[:, 0] > 0)[:, 0]
        u = p[act, 1:] / p[act, :1] + dt * gravity
        i = act % n ** 3
        ijk = torch.stack([i // (n * n), i // n % n, i % n], 1)
        if sc.tool_enabled:
            k = min(t // sc.substeps_per_action, actions.shape[1] - 1)
            for e in range(S):
                at = torch.nonzero(act // n ** 3 == e)[:, 0]
                u = u.index_copy(0, at, _contact(sc, u[at], ijk[at].to(F64) / n, pose[e], actions[e, k]))
                om, h = actions[e, k, 3:], 0.5 * dt
                th = h * om.norm()
                dq = torch.cat([torch.cos(th)[None], h * om * torch.sinc(th / math.pi)])
                turned = _quat_mul(dq, pose[e, 3:])
                pose[e] = torch.cat([pose[e, :3] + dt * actions[e, k, :3], turned / turned.norm()])
        wall = ((ijk < sc.bound) | (ijk >= n - sc.bound)).any(1, keepdim=True)
        grid = torch.zeros(S * n ** 3, 3, dtype=F64, device=dev).index_copy(0, act, torch.where(wall, torch.zeros_like(u), u))
        v, C = torch.zeros_like(v), torch.zeros_like(C)
        for W, d, i in _nodes(*stencil, n):
            wv = W[:, None] * grid[i + own]
            v, C = v + wv, C + 4 * n * n * wv[:, :, None] * d[:, None, :]
        x = x + dt * v
        G = eye + dt * C
        J = F[:, 0, 0] * torch.linalg.det(G)
        diag = torch.diag_embed(torch.stack([J, torch.ones_like(J), torch.ones_like(J)], 1))
        F = torch.where(liquid[:, None, None], diag, G @ Fp)
        for k, rb in rest.items():
            at = groups[k][1]
            m, M = mass[at][:, None], mass[at].sum()
            c, vb = (m * x[at]).sum(0) / M, (m * v[at]).sum(0) / M
            U, _, V = torch.linalg.svd((m * (x[at] - c)).T @ rb)
            fix = torch.diag(torch.stack([torch.ones((), dtype=F64, device=dev)] * 2 + [torch.linalg.det(U @ V)]))
            R = U @ fix @ V
            y = rb @ R.T
            inertia = (m * (y * y).sum(1, keepdim=True)).sum() * eye - (m * y).T @ y
            w = torch.linalg.solve(inertia, (m * torch.linalg.cross(y, v[at])).sum(0))
            K = torch.zeros(3, 3, dtype=F64, device=dev)
            K[0, 1], K[0, 2], K[1, 0], K[1, 2], K[2, 0], K[2, 1] = -w[2], w[1], w[2], -w[0], -w[1], w[0]
            x, v = x.index_copy(0, at, c + y), v.index_copy(0, at, vb + y @ K.T)
            C, F = C.index_copy(0, at, K.expand(len(at), 3, 3)), F.index_copy(0, at, R.expand(len(at), 3, 3))
    return x, v


def _exact_mpm(case, seed):
    """Forward outputs; gradients for water alone (the derivative of the plastic
    projections through torch's SVD does not exist where singular values
    coincide, as they do at rest)."""
    s = _mpm_inputs(case, seed)
    if s["x"].shape[0] * case["steps"] > 8e6:
        return None  # about 2.4 us per particle and step: more than 20 seconds
    grad = case["every"] > 0 and case["scene"] == "water"
    x0, v0 = s["x"].to(F64).requires_grad_(grad), s["v"].to(F64).requires_grad_(grad)
    if s["x"].shape[0] * case["steps"] > 2e6:
        grad = False  # the tape of a long rollout does not fit the time
    with torch.set_grad_enabled(grad):
        x, v = _rollout(s, case["steps"], x0, v0)
    out = dict(x=x.detach(), v=v.detach())
    if case["every"] == 0:
        return out
    sc = s["scene"]
    if "tm" in s:
        with torch.no_grad():
            m = _momentum(x, torch.zeros_like(x), torch.zeros(len(x), 3, 3, dtype=F64, device=DEV), s["mat"].long(),
                          torch.tensor(particle_masses(sc), dtype=F64, device=DEV), sc.grid_n)[:, 0]
            loss = ((m - s["tm"].to(F64)) ** 2).sum() / s["total"] ** 2 + (m * s["td"].to(F64)).sum() / s["total"]
    else:
        own = torch.repeat_interleave(torch.arange(sc.n_scenes, device=DEV), torch.tensor(sc.scene_counts, device=DEV))
        sq = ((x - torch.tensor(s["target"], dtype=F64, device=DEV)) ** 2).sum(1)
        loss = torch.zeros(sc.n_scenes, dtype=F64, device=DEV).index_add(0, own, sq)
    gx, gv = torch.autograd.grad(loss.sum(), (x0, v0)) if grad else (None, None)
    loss = loss.detach()
    out.update(loss=loss.sum() if case["scene"] == "water" else loss, gx=gx, gv=gv)
    return out


def _exact_surrogate(case, seed):
    s, n, B = _surrogate_inputs(case, seed), case["grid"], case["blocks"]
    P = torch.tensor(s["params"], dtype=F64, device=DEV).requires_grad_(case["op"] != "predict")

    def conv(h, at):
        pad = torch.nn.functional.pad(h.reshape(n, n, n, 32), (0, 0, 1, 1, 1, 1, 1, 1))
        W, out = P[at:at + 27 * 1024].reshape(27, 32, 32), P[at + 27 * 1024:at + 27 * 1024 + 32]
        for k, (a, b, c) in enumerate(OFFSETS):
            out = out + pad[a:a + n, b:b + n, c:c + n].reshape(-1, 32) @ W[k].T
        return out

    def net(f):
        h, at = f @ P[:256].reshape(32, 8).T + P[256:288], 288
        for _ in range(B):
            h = h + conv(torch.relu(conv(h, at)), at + 27 * 1024 + 32)
            at += 2 * (27 * 1024 + 32)
        return f[:, 1:4] + h @ P[at:at + 96].reshape(3, 32).T + P[at + 96:at + 99]

    batch = case["batch"]
    preds, gfs, grad, loss = [], [], torch.zeros_like(P), 0.0
    for b in range(batch):
        f = s["frames"][b].to(F64).requires_grad_(case["op"] == "vjp")
        with torch.set_grad_enabled(case["op"] != "predict"):
            pred = net(f)
        if case["op"] == "predict":
            preds.append(pred)
        elif case["op"] == "vjp":
            gfs.append(torch.autograd.grad(pred, f, s["g_pred"][b].to(F64))[0])
        else:
            one = ((pred - s["frames"][batch + b][:, 1:4].to(F64)) ** 2).sum() / (3 * batch * n ** 3)
            grad += torch.autograd.grad(one, P)[0]
            loss += float(one.detach())
    if case["op"] == "predict":
        return dict(pred=torch.stack(preds))
    if case["op"] == "vjp":
        return dict(g_frames=torch.stack(gfs))
    loss = torch.tensor(loss, dtype=F64)
    # an Adam step from rest moves every parameter by the sign of its gradient
    # almost alone, which the rounded activations leave open where it is small
    return dict(loss=loss, grad=grad) if case["op"] == "grad" else dict(loss=loss, params=None)


def _exact_features(case, seed):
    n = case["grid"]
    sc, x, v, C, mat = _layout(n, case["particles"], seed)
    g = torch.Generator().manual_seed(seed)
    w = torch.randn(n ** 3, 8, generator=g).to(DEV).to(F64)
    args = [a.to(F64).requires_grad_(True) for a in (x, v, C)]
    frame = _frame(*args, mat.long(), particle_masses(sc), n, *frame_scales(sc))
    gx, gv, gC = torch.autograd.grad((frame[:, :4] * w[:, :4]).sum(), args)
    return dict(frame=frame.detach(), gx=gx, gv=gv, gC=gC)


def _exact_gas(case, seed):
    s, n = _gas_inputs(case, seed), case["grid"]
    fluid = torch.tensor(s["solid"] == 0, device=DEV)
    ff, dx = fluid.to(F64), 1.0 / n

    def shift(a, axis, by, fill):
        """a at the neighbour `by` cells along `axis` (outside the grid: fill)."""
        r = torch.roll(a, -by, axis)
        r.narrow(axis, n - 1 if by > 0 else 0, 1).fill_(fill)
        return r

    nb = [(ax, by, shift(ff.clone(), ax, by, 0.0)) for ax in range(3) for by in (1, -1)]
    count = sum(m for _, _, m in nb).clamp_min(1.0)
    some = (sum(m for _, _, m in nb) > 0).to(F64)
    ijk = torch.stack(torch.meshgrid(*[torch.arange(n, device=DEV, dtype=F64)] * 3, indexing="ij"))

    def sweeps(p, rhs, k):
        for _ in range(k):
            q = sum(m * shift(p, ax, by, 0.0) for ax, by, m in nb)
            p = ff * (p / 3 + (2 / 3) * some * (q - dx * dx * rhs) / count)
        return p

    def step(u, d):
        ub = torch.stack([u[0], u[1] + s["dt"] * s["buoyancy"] * d, u[2]])
        X = (ijk - s["dt"] * n * ub).clamp(0.0, n - 1.0)
        b = torch.floor(X.detach()).clamp_max(n - 2)
        t, b = X - b, b.long()
        fields, new = torch.cat([ub, d[None]]).reshape(4, -1), 0.0
        for a in range(2):
            for c in range(2):
                for e in range(2):
                    w = (t[0] if a else 1 - t[0]) * (t[1] if c else 1 - t[1]) * (t[2] if e else 1 - t[2])
                    i = ((b[0] + a) * n + b[1] + c) * n + b[2] + e
                    new = new + w * fields[:, i.reshape(-1)].reshape(4, n, n, n)
        new = new * ff
        un = new[:3]
        div = ff * sum(by * m * shift(un[ax], ax, by, 0.0) for ax, by, m in nb) * (0.5 * n)
        rhs = ff * (div - div.sum() / ff.sum())
        p, left = torch.zeros_like(d), case["sweeps"]
        while left:
            k = min(10, left)
            p = torch.utils.checkpoint.checkpoint(sweeps, p, rhs, k, use_reentrant=False)
            left -= k
        parts = []
        for ax in range(3):
            hi, lo = [m * shift(p, ax, by, 0.0) + (1 - m) * p for a, by, m in nb if a == ax]
            parts.append(un[ax] - ff * (hi - lo) * (0.5 * n))
        return torch.stack(parts), new[3]

    u0, d0 = (s["u"].to(F64) * ff).requires_grad_(True), (s["d"].to(F64) * ff).requires_grad_(True)
    u, d = u0, d0
    for _ in range(case["steps"]):
        u, d = torch.utils.checkpoint.checkpoint(step, u, d, use_reentrant=False)
    gu, gd = torch.autograd.grad([u, d], [u0, d0], [s["gu"].to(F64), s["gd"].to(F64)])
    return dict(u=u.detach(), d=d.detach(), gu=gu * ff, gd=gd * ff)


def _exact_sharing(case, seed):
    s = _sharing_inputs(case, seed)
    x0, v0 = s["x"].to(F64).requires_grad_(True), s["v"].to(F64).requires_grad_(True)
    x1, _ = _rollout(s, 1, x0, v0)
    x, h = x1.detach(), s["radius"]
    c, g = torch.exp(-s["ell"].to(F64) / s["tau"]), s["g"].to(F64)
    N, loss = len(x), 0.0
    shared, gx = torch.zeros_like(x), torch.zeros_like(x)
    for a in range(0, N, 1024):
        diff = x[a:a + 1024, None] - x[None]
        at, of = torch.nonzero((diff * diff).sum(-1) < h * h, as_tuple=True)
        del diff
        e = x[a + at] - x[of]
        d = e.norm(dim=1)
        om = 1 - (d / h) ** 2
        shared.index_add_(0, a + at, (c[of] * om ** 3)[:, None] * g[of])
        k = d > 0
        at, of, e, d, om = at[k], of[k], e[k], d[k], om[k]
        loss += float((c[of] * d * om ** 3).sum())
        slope = om ** 3 - 6 * (d / h) ** 2 * om ** 2
        gx.index_add_(0, a + at, ((c[of] + c[a + at]) * slope / d)[:, None] * e)
    gx0, gv0 = torch.autograd.grad(x1, (x0, v0), gx)
    return dict(loss=torch.tensor(loss, dtype=F64), gx=gx0, gv=gv0, shared=shared)


_EXACT = dict(mpm=_exact_mpm, surrogate=_exact_surrogate, features=_exact_features, gas=_exact_gas,
              sharing=_exact_sharing)
