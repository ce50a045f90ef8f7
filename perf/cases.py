"""The work whose time counts: what a user of this library has it do, through its public calls.

Each case is one call pattern of a user's program, at sizes of the library's own workloads:

* ``forward``: a rollout of explicit steps from a saved state (``mpm_restore_state``,
  ``mpm_step``) and the whole particle state read back into device tensors
  (``mpm_get_particles_dev``);
* ``adjoint``: one evaluation of an inversion: restore, set the friction field, loss and
  gradient by the checkpointed adjoint (``mpm_step_adjoint``);
* ``infer``, ``train``: the warm-start network (``MLP.infer`` on host rows,
  ``MLP.train_step_async`` on resident mini-batches);
* ``gemm``: the tensor-core product ``mpm_gemm_bf16``.

The bodies are the workloads' bodies (water column, water block with two columns, sand
cylinder) in mid-flow: a smooth velocity field of the speeds those flows reach, its
gradient as the affine matrix, a slightly compressed density, a geostatic stress in the
sand.  Values are drawn from the seed and rounded to single precision.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2507_04192_gb300 import mpm

WATER = dict(kind=0, rho0=1000.0, bulk_K=2.0e5, gamma=7.0)
WATER_LINEAR = dict(kind=0, rho0=1000.0, bulk_K=1000.0 * 35.0 ** 2, gamma=1.0)
SAND = dict(kind=1, rho0=2000.0, E=1.0e6, nu=0.3, phi_deg=30.0)
SORT_EVERY = 32


def listed():
    return [
        # one held-out problem's observations through the warm-start network: the smallest call
        dict(name="infer_1", kind="infer", batch=1, n_in=640, hidden=256, n_out=32),
        # eight mini-batches of the network's training, batch 256, data resident on the GPU
        dict(name="train_256", kind="train", batch=256, n_in=640, hidden=256, n_out=32, steps=8),
        # the tensor-core product at the size of the benchmark's GEMM line
        dict(name="gemm_8192", kind="gemm", m=8192, n=2048, k=2048),
        # the small dam break (8,192 particles): interactive runs and tests, launch-bound
        dict(name="water2d_64", kind="forward", body="water2d", cells=64, batch=1, steps=32, fp64=False),
        # 256 dam breaks in one context (4.7M particles): the training data of the warm start
        dict(name="water2d_96_x256", kind="forward", body="water2d", cells=96, batch=256, steps=32, fp64=False),
        # the reduced sand cylinder (about 50,000 particles) over 4 x 4 floor patches
        dict(name="sand3d_64", kind="forward", body="sand3d", cells=64, batch=1, steps=32, fp64=False),
        # the 2.76M-particle sand collapse, the benchmark's workload
        dict(name="sand3d_256", kind="forward", body="sand3d", cells=256, batch=1, steps=32, fp64=False),
        # the 1.92M-particle 3D dam break with two rigid columns
        dict(name="water3d_200", kind="forward", body="water3d", cells=200, batch=1, steps=32, fp64=False),
        # the 1.36M-particle collapse in double precision: the accuracy mode
        dict(name="sand3d_192_fp64", kind="forward", body="sand3d", cells=192, batch=1, steps=8, fp64=True),
        # an evaluation of the 2D friction inversion (32,768 particles, 32 floor segments)
        dict(name="adjoint2d_128", kind="adjoint", body="water2d", cells=128, steps=100, every=50, fp64=False),
        # an evaluation of the reduced 3D friction inversion (4 x 4 floor patches)
        dict(name="adjoint3d_64", kind="adjoint", body="sand3d", cells=64, steps=60, every=20, fp64=False),
        # an evaluation of the 3D friction inversion at scale (1.36M particles, 16 x 16 patches)
        dict(name="adjoint3d_192", kind="adjoint", body="sand3d", cells=192, steps=40, every=20, fp64=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.random()
    if pick < 0.10:
        return dict(kind="infer", batch=_log(rng, 1, 512), n_in=8 * _log(rng, 8, 160), hidden=8 * _log(rng, 8, 64),
                    n_out=8 * _log(rng, 1, 32))
    if pick < 0.20:
        return dict(kind="train", batch=8 * _log(rng, 1, 64), n_in=8 * _log(rng, 8, 160), hidden=8 * _log(rng, 8, 64),
                    n_out=8 * _log(rng, 1, 32), steps=rng.randint(4, 8))
    if pick < 0.28:
        return dict(kind="gemm", m=_log(rng, 64, 8192), n=_log(rng, 8, 2048), k=8 * _log(rng, 8, 256))
    fp64 = rng.random() < 0.2
    if pick < 0.46:
        cells = _log(rng, 24, 160)
        batch = min(_log(rng, 1, 256), max(1, int(256 * (96 / cells) ** 2)))
        return dict(kind="forward", body="water2d", cells=cells, batch=1 if fp64 else batch,
                    steps=8 if fp64 else rng.choice([16, 32]), fp64=fp64)
    if pick < 0.62:
        return dict(kind="forward", body="sand3d", cells=_log(rng, 32, 160 if fp64 else 256), batch=1,
                    steps=8 if fp64 else rng.choice([16, 32]), fp64=fp64)
    if pick < 0.72:
        return dict(kind="forward", body="water3d", cells=20 * _log(rng, 3, 8 if fp64 else 10), batch=1,
                    steps=8 if fp64 else rng.choice([16, 32]), fp64=fp64)
    if pick < 0.86:
        return dict(kind="adjoint", body="water2d", cells=_log(rng, 32, 160), steps=10 * rng.randint(4, 10),
                    every=rng.choice([20, 25, 50]), fp64=fp64)
    return dict(kind="adjoint", body="sand3d", cells=_log(rng, 32, 96 if fp64 else 180), steps=4 * rng.randint(5, 10),
                every=rng.choice([10, 15, 20]), fp64=fp64)


# ---------------------------------------------------------------- inputs

class _Scene:
    """Grid, material, particles and boundary conditions of one simulated case."""

    def __init__(self, case, seed):
        body, g = case["body"], int(case["cells"])
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed))
        rand = lambda *s: torch.rand(*s, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
        self.batch = int(case.get("batch", 1))
        self.dim = 2 if body == "water2d" else 3
        d = self.dim
        if body == "water2d":
            self.cells, self.dx, self.dt, self.mat, ppc, speed = (g, g), 1.0 / g, 1.0e-4 * min(1.0, 128 / g), WATER, 4, 1.0
            hi = (0.25, 0.5)
            self.wall, self.seg = 2, (32, 1)
        elif body == "water3d":
            self.cells, self.dx, self.dt, self.mat, ppc, speed = (g, g // 2, 2 * g // 5), 1.0 / g, 1.0e-5, WATER_LINEAR, 2, 1.0
            hi = (0.3, self.cells[1] * self.dx, 0.2)
            self.wall = -1
        else:
            self.cells = (g, g, g // 2)
            self.dx, self.dt, self.mat, ppc, speed = 1.0 / 256.0, 1.0e-5, SAND, 2, 0.3
            if g < 128:                                   # the reduced problem's coarser grid and step
                self.dx, self.dt = 1.0 / 64.0, 4.0e-5
            r = 10 if g == 64 else (38 if g == 256 else 5 * g // 32)
            self.r, self.axis = r * self.dx, (0.5 * g * self.dx, 0.5 * g * self.dx)
            hi = (self.axis[0] + self.r, self.axis[1] + self.r, 2 * self.r)
            self.wall = 4
            self.seg = (4, 4) if g < 128 else (16, 16)
        self.gravity = (0.0,) * (d - 1) + (-9.81,)
        self.L = tuple(c * self.dx for c in self.cells)
        h = self.dx / ppc
        axes = [(torch.arange(min(c * ppc, math.ceil(top / h - 0.5)), device="cuda", dtype=torch.float64) + 0.5) * h
                for c, top in zip(self.cells, hi)]
        pts = torch.stack([m.reshape(-1) for m in torch.meshgrid(*axes[::-1], indexing="ij")[::-1]], 1)
        if body == "sand3d":
            pts = pts[((pts[:, 0] - self.axis[0]) ** 2 + (pts[:, 1] - self.axis[1]) ** 2 < self.r ** 2)]
        one = lambda t: t.float().double()  # noqa: E731
        self.per_sim = pts.shape[0]
        x = pts.repeat(self.batch, 1)
        self.sim = torch.arange(self.batch, device="cuda", dtype=torch.int32).repeat_interleave(self.per_sim)
        self.x = one(x + (rand(x.shape) - 0.5) * 0.5 * h).contiguous()
        self.n = x.shape[0]
        self.volume = self.dx ** d / ppc ** d
        # velocity: two sine waves per component over the body, and its gradient
        wave, phase, amp = 2.0 * math.pi * (rand(d, 2, d) - 0.5) / max(hi), 2.0 * math.pi * rand(d, 2), speed * (0.5 + rand(d, 2)) / 2
        v, C = torch.zeros_like(self.x), torch.zeros(self.n, d, d, device="cuda", dtype=torch.float64)
        for a in range(d):
            for j in range(2):
                arg = self.x @ wave[a, j] + phase[a, j]
                v[:, a] += amp[a, j] * torch.sin(arg)
                C[:, a] += (amp[a, j] * torch.cos(arg))[:, None] * wave[a, j]
        self.v, self.C = one(v).contiguous(), one(C).contiguous()
        depth = (hi[-1] - self.x[:, -1]).clamp_min(0.0)
        self.rho = one(self.mat["rho0"] * (1.0 + 2.0e-4 * torch.sin(self.x @ (2.0 * wave[0, 0]) + phase[0, 1])))
        self.sigma = None
        if self.mat["kind"] == 1:
            p = self.mat["rho0"] * 9.81 * depth + 50.0
            s = torch.zeros(self.n, 3, 3, device="cuda", dtype=torch.float64)
            s[:, 0, 0], s[:, 1, 1], s[:, 2, 2] = -0.6 * p, -0.55 * p, -p
            shear = 0.1 * p * torch.sin(self.x @ wave[1, 0] + phase[1, 1])
            s[:, 0, 2] = s[:, 2, 0] = shear
            s[:, 0, 1] = s[:, 1, 0] = 0.5 * shear
            self.sigma = one(s).contiguous()
        self.mu = None
        if self.wall >= 0:
            self.mu = (0.1 + 0.5 * rand(self.batch, self.seg[0] * self.seg[1]).float()).double().cpu().numpy()
        self.boxes = []
        if body == "water3d":
            for (cx, cy), side in (((0.5, 0.3), 0.04), ((0.6, 0.1), 0.06)):
                self.boxes.append(((cx - side / 2, cy - side / 2, 0.0), (cx + side / 2, cy + side / 2, self.L[2])))
        if case["kind"] == "adjoint":                     # tracked particles: their free flight, off by a hundredth of a cell
            steps = int(case["steps"])
            n_track = min(64 if d == 2 else 128, self.n)
            ids = torch.randperm(self.n, generator=gen, device="cuda")[:n_track]
            self.obs_steps = sorted({max(1, steps * (k + 1) // 10) for k in range(10)})
            z = []
            for s in self.obs_steps:
                t = s * self.dt
                z.append(self.x[ids] + t * self.v[ids] + 0.01 * self.dx * (2.0 * rand(n_track, d) - 1.0))
            self.ids, self.z = ids.cpu().numpy(), torch.stack(z).cpu().numpy()


def _forward_fields(scene):
    return ["x", "v", "C", "F", "rho"] + (["sigma", "eps"] if scene.mat["kind"] == 1 else ["sigma"])


@functools.lru_cache(maxsize=None)
def _stream():
    """The one stream of the program: passes on it follow each other."""
    return torch.cuda.Stream()


def _simulation(case, seed):
    sc = _Scene(case, seed)
    stream = _stream()
    prec = mpm.MPM_FP64 if case["fp64"] else mpm.MPM_FP32
    sim = mpm.Simulation(sc.dim, sc.cells, sc.dx, sc.dt, sc.gravity, sc.mat, prec, SORT_EVERY, sc.batch,
                         stream=stream.cuda_stream)
    torch.cuda.synchronize()
    mpm.mpm_load_particles_dev(sim.ctx, sc.n, sc.x.data_ptr(), sc.v.data_ptr(), sc.volume,
                               sc.sim.data_ptr() if sc.batch > 1 else None)
    sim.set_field("C", sc.C.cpu().numpy())
    sim.set_field("rho", sc.rho.cpu().numpy())
    if sc.sigma is not None:
        sim.set_field("sigma", sc.sigma.cpu().numpy())
    if sc.mu is not None:
        sim.set_friction(sc.wall, sc.seg, sc.mu.reshape(-1))
    if sc.boxes:
        sim.set_obstacles(sc.boxes)
    mpm.mpm_save_state(sim.ctx, 0)
    sim.synchronize()
    state = dict(kind=case["kind"], sim=sim, stream=stream, n=sc.n, dtype=torch.float64 if case["fp64"] else torch.float32,
                 np_dtype=np.float64 if case["fp64"] else np.float32, steps=int(case["steps"]))
    if case["kind"] == "forward":
        state["fields"] = _forward_fields(sc)
    else:
        mpm.mpm_set_observations(sim.ctx, sc.ids, sc.obs_steps, sc.z)
        state.update(every=int(case["every"]), wall=sc.wall, seg=sc.seg, mu=sc.mu.reshape(-1), dim=sc.dim, fields=["x", "v"])
    return state


def _network(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    widths = [case["n_in"], case["hidden"], case["hidden"], case["n_out"]]
    p = []
    for l in range(3):
        p.append(torch.randn(widths[l + 1] * widths[l], generator=gen, device="cuda") * math.sqrt(2.0 / widths[l]))
        p.append(0.05 * torch.randn(widths[l + 1], generator=gen, device="cuda"))
    rows = case["batch"] * case.get("steps", 1)
    x = torch.randn(rows, widths[0], generator=gen, device="cuda")
    t = 0.1 + 0.5 * torch.rand(rows, widths[-1], generator=gen, device="cuda")
    return widths, torch.cat(p), x, t


def prepare(case, seed):
    if case["kind"] in ("forward", "adjoint"):
        return _simulation(case, seed)
    if case["kind"] == "gemm":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed))
        m, n, k = case["m"], case["n"], case["k"]
        a = torch.randn(m, k, generator=gen, device="cuda").to(torch.bfloat16)
        b = torch.randn(n, k, generator=gen, device="cuda").to(torch.bfloat16)
        return dict(kind="gemm", a=a, b=b, c=torch.zeros(m, n, device="cuda"),
                    status=torch.zeros(1, dtype=torch.int32, device="cuda"), m=m, n=n, k=k)
    widths, params, x, t = _network(case, seed)
    stream = _stream()
    net = mpm.MLP(widths, (case["batch"] + 7) // 8 * 8, 0.1, 0.6, stream=stream.cuda_stream)
    net.set_params(params.cpu().numpy())
    state = dict(kind=case["kind"], net=net, stream=stream)
    if case["kind"] == "infer":
        state["x"] = x.cpu().numpy()
    else:
        b = case["batch"]
        state.update(batch=b, x=[x[i:i + b].contiguous() for i in range(0, len(x), b)],
                     t=[t[i:i + b].contiguous() for i in range(0, len(t), b)],
                     loss=torch.zeros(case["steps"], dtype=torch.float64, device="cuda"))
        torch.cuda.synchronize()
    return state


# ---------------------------------------------------------------- one pass

_WIDTH = {"x": lambda d: (d,), "v": lambda d: (d,), "C": lambda d: (d, d), "F": lambda d: (d, d), "rho": lambda d: (),
          "eps": lambda d: (), "sigma": lambda d: (3, 3)}


def _read_fields(state):
    """The particle state as tensors of the simulation's precision, on the context's stream."""
    out, sim = {}, state["sim"]
    with torch.cuda.stream(state["stream"]):
        for f in state["fields"]:
            t = torch.empty((state["n"],) + _WIDTH[f](sim.dim), dtype=torch.float64, device="cuda")
            mpm.mpm_get_particles_dev(sim.ctx, f, t.data_ptr())
            out[f] = t.to(state["dtype"])
    return out


def run(state):
    kind = state["kind"]
    if kind == "forward":
        sim = state["sim"]
        mpm.mpm_restore_state(sim.ctx, 0)
        sim.step(state["steps"])
        return _read_fields(state)
    if kind == "adjoint":
        sim = state["sim"]
        mpm.mpm_restore_state(sim.ctx, 0)
        sim.set_friction(state["wall"], state["seg"], state["mu"])
        loss, g = mpm.mpm_step_adjoint(sim.ctx, state["steps"], state["every"], state["wall"], len(state["mu"]))
        out = {"loss": np.asarray(loss, dtype=state["np_dtype"]), "dmu": g.astype(state["np_dtype"])}
        if state["dim"] == 2:                             # the initial-velocity inversion reads this too
            out["dv0"] = mpm.mpm_get_initial_adjoint(sim.ctx, "v").astype(state["np_dtype"])
        out.update(_read_fields(state))
        return out
    if kind == "infer":
        return state["net"].infer(state["x"])
    if kind == "train":
        net, loss = state["net"], state["loss"]
        for i, (x, t) in enumerate(zip(state["x"], state["t"])):
            net.train_step_async(state["batch"], x.data_ptr(), t.data_ptr(), 1e-3, loss.data_ptr() + 8 * i)
        return {"grad": net.get_params(1), "loss": loss.float()}
    mpm.mpm_gemm_bf16(state["m"], state["n"], state["k"], state["a"].data_ptr(), state["k"], state["b"].data_ptr(),
                      state["k"], state["c"].data_ptr(), state["n"], state["status"].data_ptr(),
                      torch.cuda.current_stream().cuda_stream)
    return state["c"]


# ---------------------------------------------------------------- what a pass cannot do without

def _count(case):
    body, g = case["body"], int(case["cells"])
    if body == "water2d":
        return int(case.get("batch", 1)) * (int(math.ceil(g - 0.5)) * int(math.ceil(2 * g - 0.5)))
    if body == "water3d":
        return int(math.ceil(0.6 * g - 0.5)) * 2 * (g // 2) * int(math.ceil(0.4 * g - 0.5))
    r = 10 if g == 64 else (38 if g == 256 else 5 * g // 32)
    return int(math.pi * r * r * 2 * r * 8)


def work(case):
    kind = case["kind"]
    if kind in ("infer", "train"):
        w = [case["n_in"], case["hidden"], case["hidden"], case["n_out"]]
        nw = sum(w[l] * w[l + 1] + w[l + 1] for l in range(3))
        b = case["batch"]
        if kind == "infer":                               # weights as bf16 operands once, rows in and out
            return dict(bytes=2 * nw + 4 * b * (w[0] + w[3]), flops=2 * b * nw)
        # per step: weights and two moments read and written in fp32, the gradient written, rows in
        return dict(bytes=case["steps"] * (28 * nw + 4 * b * (w[0] + w[3])), flops=case["steps"] * 6 * b * nw)
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(bytes=2 * (m * k + n * k) + 4 * m * n, flops=2 * m * n * k)
    n, real = _count(case), 8 if case["fp64"] else 4
    d = 2 if case["body"] == "water2d" else 3
    sand = case["body"] == "sand3d"
    words = 2 * d + 2 * d * d + 1 + (7 if sand else 0)    # x, v, C, F, rho [, sigma, eps]
    reads = 2 * d + d * d + 1 + (6 if sand else 0)        # what the reverse step needs of a state
    flops = 500 if d == 2 else (1800 if sand else 1500)   # P2G, G2P and the constitutive update of one particle
    if kind == "forward":                                 # per step the state once in and once out; then the fields
        return dict(bytes=case["steps"] * 2 * words * real * n + 3 * words * real * n, flops=case["steps"] * flops * n)
    # forward step, its state kept and read again, the adjoint state in and out
    return dict(bytes=case["steps"] * (2 * words + 4 * reads) * real * n, flops=case["steps"] * 3.5 * flops * n)


# ---------------------------------------------------------------- the same in 64 bits, plainly

def _safe_sqrt(t):
    ok = t > 0
    return torch.where(ok, torch.where(ok, t, torch.ones_like(t)).sqrt(), torch.zeros_like(t))


def _apply(A, u):
    """A u per particle."""
    return torch.stack([sum(A[:, a, b] * u[:, b] for b in range(u.shape[1])) for a in range(A.shape[1])], 1)


def _return_map(mat, L, dt, s, eps):
    """Drucker-Prager with tension cutoff and the Jaumann rate (corner return past the cutoff)."""
    K, G = mat["E"] / (3 * (1 - 2 * mat["nu"])), mat["E"] / (2 * (1 + mat["nu"]))
    sp = math.sin(math.radians(mat["phi_deg"]))
    q = 6 * sp / (math.sqrt(3.0) * (3 + sp))
    alpha = math.sqrt(1 + q * q) - q
    # cohesionless, no dilation: k = 0, the cutoff at 0
    de, w = 0.5 * dt * (L + L.transpose(1, 2)), 0.5 * dt * (L - L.transpose(1, 2))
    eye = torch.eye(3, dtype=s.dtype, device=s.device)
    tr = de.diagonal(dim1=1, dim2=2).sum(1)
    M = w @ s
    t = s + M + M.transpose(1, 2) + (K - 2 * G / 3) * tr[:, None, None] * eye + 2 * G * de
    sm = t.diagonal(dim1=1, dim2=2).sum(1) / 3
    dev = t - sm[:, None, None] * eye
    tau = _safe_sqrt(0.5 * (dev * dev).sum((1, 2)))
    fs, h = tau + q * sm, tau - alpha * sm
    one = (fs <= 0) & (sm < 0)
    two = ~one & (((fs > 0) & (sm < 0)) | ((h > 0) & (sm >= 0)))
    safe = torch.where(tau > 0, tau, torch.ones_like(tau))
    r2 = torch.where((tau > 0) & (sm <= 0), -q * sm / safe, torch.zeros_like(tau))      # corner: tau_P = 0
    m2 = torch.where(sm > 0, torch.zeros_like(sm), sm)
    r3 = torch.where(tau > 0, torch.zeros_like(tau), torch.ones_like(tau))
    s2 = r2[:, None, None] * dev + m2[:, None, None] * eye
    s3 = r3[:, None, None] * dev
    out = torch.where(one[:, None, None], t, torch.where(two[:, None, None], s2, s3))
    de2 = fs / G * math.sqrt(1.0 / 3.0)
    de3 = sm / K * (math.sqrt(2.0) / 3)
    zero = torch.zeros_like(eps)
    return out, eps + torch.where(one, zero, torch.where(two, de2, de3)).detach()


def _grid_update(sc, grid, mu):
    """Gravity, obstacles and walls on every node; grid: (batch, nodes, 1 + d), node axes x fastest."""
    d = sc.dim
    m = grid[..., 0]
    live = m > 1e-10 * sc.mat["rho0"] * sc.dx ** d
    v = grid[..., 1:] / torch.where(live, m, torch.ones_like(m))[..., None]
    g = torch.tensor(sc.gravity, dtype=grid.dtype, device=grid.device)
    v = torch.where(live[..., None], v + sc.dt * g, torch.zeros_like(v))
    ax = [torch.arange(c + 3, device=grid.device) - 1 for c in sc.cells]
    coord = [c.reshape(-1) for c in torch.meshgrid(*ax[::-1], indexing="ij")[::-1]]
    comp = list(v.unbind(-1))
    for lo, hi in sc.boxes:
        l = [math.ceil(a / sc.dx - 1e-9) for a in lo]
        u = [math.floor(a / sc.dx + 1e-9) for a in hi]
        inside = torch.ones_like(coord[0], dtype=torch.bool)
        best = torch.full_like(coord[0], -1)
        dist = torch.full_like(coord[0], 1 << 30)
        for a in range(d):
            inside = inside & (coord[a] >= l[a]) & (coord[a] <= u[a])
            for f, gap, face in ((2 * a, coord[a] - l[a], l[a] > 0), (2 * a + 1, u[a] - coord[a], u[a] < sc.cells[a])):
                if face:
                    near = gap < dist
                    best, dist = torch.where(near, f, best), torch.where(near, gap, dist)
        for f in range(2 * d):
            hit = inside & (best == f) & ((comp[f >> 1] < 0) if f & 1 else (comp[f >> 1] > 0))
            comp[f >> 1] = torch.where(hit, torch.zeros_like(comp[f >> 1]), comp[f >> 1])
    floor = 2 * (d - 1)
    for w in [q for q in range(2 * d) if q != floor] + [floor]:
        a, high = w >> 1, w & 1
        on = (coord[a] >= sc.cells[a]) if high else (coord[a] <= 0)
        vn = comp[a] if high else -comp[a]
        hit = on & (vn > 0)
        slid = [torch.zeros_like(c) if b == a else c for b, c in enumerate(comp)]
        if w == sc.wall:
            tang = [b for b in range(d) if b != a]
            seg = torch.zeros_like(coord[0])
            for k, b in reversed(list(enumerate(tang))):
                s = torch.div(coord[b].clamp_min(0) * sc.seg[k], sc.cells[b], rounding_mode="floor").clamp_max(sc.seg[k] - 1)
                seg = seg * sc.seg[k] + s
            m_ = mu[:, seg]
            vt = _safe_sqrt(torch.where(hit, sum(c * c for c in slid), torch.zeros_like(vn)))
            push = torch.where(hit, m_ * vn, torch.zeros_like(vn))
            slides = hit & (vt > push)
            scale = torch.where(slides, 1 - push / torch.where(slides, vt, torch.ones_like(vt)), torch.zeros_like(vt))
            slid = [torch.where(m_ > 0, c * scale, c) for c in slid]
        comp = [torch.where(hit, s, c) for s, c in zip(slid, comp)]
    return torch.stack(comp, -1)


def _exact_step(sc, x, v, C, F, rho, s, eps, mu):
    d, dx, dt, mat = sc.dim, sc.dx, sc.dt, sc.mat
    mass = mat["rho0"] * sc.volume
    cells = torch.tensor(sc.cells, device=x.device)
    base = torch.minimum((x.detach() / dx - 0.5).floor().long().clamp_min(-1), cells - 1)
    f = x / dx - base
    W = [0.5 * (1.5 - f) ** 2, 0.75 - (f - 1) ** 2, 0.5 * (f - 0.5) ** 2]
    dW = [(f - 1.5) / dx, -2 * (f - 1) / dx, (f - 0.5) / dx]
    size = [c + 3 for c in sc.cells]
    nodes = math.prod(size)
    vol = mass / rho
    if mat["kind"] == 0:
        p = mat["bulk_K"] / mat["gamma"] * ((rho / mat["rho0"]) ** mat["gamma"] - 1)
        force = (dt * vol * p)[:, None, None] * torch.eye(d, dtype=x.dtype, device=x.device)
    else:
        force = (-dt * vol)[:, None, None] * s[:, :d, :d]

    def stencil():
        for k in range(3 ** d):
            kk = [k % 3, (k // 3) % 3, k // 9][:d]
            idx, stride = sc.sim.long() * nodes, 1
            for a in range(d):
                idx = idx + (base[:, a] + 1 + kk[a]) * stride
                stride *= size[a]
            wt = W[kk[0]][:, 0]
            for a in range(1, d):
                wt = wt * W[kk[a]][:, a]
            gr = []
            for a in range(d):
                t = dW[kk[a]][:, a]
                for b in range(d):
                    if b != a:
                        t = t * W[kk[b]][:, b]
                gr.append(t)
            rel = (torch.tensor(kk, dtype=x.dtype, device=x.device) - f) * dx
            yield idx, wt, torch.stack(gr, 1), rel

    grid = torch.zeros(sc.batch * nodes, 1 + d, dtype=x.dtype, device=x.device)
    for idx, wt, gr, rel in stencil():
        mom = mass * wt[:, None] * (v + _apply(C, rel)) + _apply(force, gr)
        grid = grid.index_add_(0, idx, torch.cat([(mass * wt)[:, None], mom], 1))
    gv = _grid_update(sc, grid.reshape(sc.batch, nodes, 1 + d), mu).reshape(-1, d)
    vp, Bn, L = torch.zeros_like(v), torch.zeros_like(C), torch.zeros_like(C)
    for idx, wt, gr, rel in stencil():
        vi = gv.index_select(0, idx)
        wv = wt[:, None] * vi
        vp = vp + wv
        Bn = Bn + wv[:, :, None] * rel[:, None, :]
        L = L + vi[:, :, None] * gr[:, None, :]
    xn = x + dt * vp
    top = torch.tensor(sc.L, dtype=x.dtype, device=x.device)
    xn = torch.where(xn < 0, torch.zeros_like(xn), torch.where(xn > top, top.expand_as(xn), xn))
    Fn = F + dt * (L.detach() @ F)
    rn = rho / (1 + dt * L.diagonal(dim1=1, dim2=2).sum(1))
    if mat["kind"] == 1:
        s, eps = _return_map(mat, L, dt, s, eps)
    return xn, vp, Bn * (4 / dx ** 2), Fn, rn, s, eps


def _start_state(sc):
    n, d = sc.n, sc.dim
    F = torch.eye(d, dtype=torch.float64, device="cuda").repeat(n, 1, 1)
    s = sc.sigma if sc.sigma is not None else torch.zeros(n, 3, 3, dtype=torch.float64, device="cuda")
    return [sc.x, sc.v, sc.C, F, sc.rho, s, torch.zeros(n, dtype=torch.float64, device="cuda")]


def _exact_forward(case, seed):
    sc = _Scene(case, seed)
    S = _start_state(sc)
    mu = torch.as_tensor(sc.mu, device="cuda") if sc.mu is not None else None
    with torch.no_grad():
        for _ in range(int(case["steps"])):
            S = _exact_step(sc, *S, mu)
    x, v, C, F, rho, s, eps = S
    if sc.mat["kind"] == 0:
        p = sc.mat["bulk_K"] / sc.mat["gamma"] * ((rho / sc.mat["rho0"]) ** sc.mat["gamma"] - 1)
        s = -p[:, None, None] * torch.eye(3, dtype=p.dtype, device=p.device)
    got = dict(x=x, v=v, C=C, F=F, rho=rho, sigma=s, eps=eps)
    return {k: got[k] for k in _forward_fields(sc)}


def _exact_adjoint(case, seed):
    from torch.utils.checkpoint import checkpoint
    sc = _Scene(case, seed)
    if sc.n * int(case["steps"]) > 6.0e7:                 # over about 20 seconds
        return None
    S = _start_state(sc)
    mu = torch.as_tensor(sc.mu, device="cuda").requires_grad_()
    v0 = S[1].clone().requires_grad_()
    S[1] = v0
    ids, z = torch.as_tensor(sc.ids, device="cuda"), torch.as_tensor(sc.z, device="cuda")
    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    for t in range(1, int(case["steps"]) + 1):
        S = checkpoint(lambda *a: _exact_step(sc, *a), *S, mu, use_reentrant=False)
        if t in sc.obs_steps:
            loss = loss + ((S[0][ids] - z[sc.obs_steps.index(t)]) ** 2).sum()
    loss.backward()
    out = {"loss": loss.detach(), "dmu": mu.grad.reshape(-1)}
    if sc.dim == 2:
        out["dv0"] = v0.grad
    out.update(x=S[0].detach(), v=S[1].detach())
    return out


def _exact_network(case, seed):
    widths, params, x, t = _network(case, seed)
    p, at, layers = params.double(), 0, []
    for l in range(3):
        k = widths[l] * widths[l + 1]
        W = p[at:at + k].reshape(widths[l + 1], widths[l]).clone().requires_grad_()
        b = p[at + k:at + k + widths[l + 1]].clone().requires_grad_()
        layers.append((W, b))
        at += k + widths[l + 1]

    def net(rows):
        for l, (W, b) in enumerate(layers):
            rows = rows @ W.T + b
            rows = 0.5 * rows * (1 + torch.erf(rows / math.sqrt(2.0))) if l < 2 else 0.1 + 0.5 * torch.sigmoid(rows)
        return rows

    if case["kind"] == "infer":
        with torch.no_grad():
            return net(x.double())
    flat = [q for pair in layers for q in pair]
    opt = torch.optim.Adam(flat, lr=1e-3, betas=(0.9, 0.999), eps=1e-8)
    b, losses = case["batch"], []
    for i in range(0, len(x), b):
        opt.zero_grad()
        loss = ((net(x[i:i + b].double()) - t[i:i + b].double()) ** 2).mean()
        loss.backward()
        losses.append(loss.detach())
        opt.step()
    return {"grad": torch.cat([q.grad.reshape(-1) for q in flat]), "loss": torch.stack(losses)}


def exact(case, seed):
    if case["kind"] == "forward":
        return _exact_forward(case, seed)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    if case["kind"] == "gemm":
        s = prepare(case, seed)
        return s["a"].double() @ s["b"].double().T
    return _exact_network(case, seed)
