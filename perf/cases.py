"""What is measured of this simulator: one pass per case through its public entry points.

The cases are the work a user has it do: one control step of a small body on caller-owned arrays,
frames of a small cube read back by the host, lattices from cache-sized to larger than the
L2, an unstructured mesh, a swarm of worms, batches of robots rolled out together, the gradient of
a rollout, and the fitness surrogate (prediction, training, its product alone).  Geometry is
generated once per size and kept in a small cache; stiffness, rest lengths, actuation and states are
drawn from the seed.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1911_10274_gb300 import inputs
from paper_1911_10274_gb300 import titan as T

DEV = "cuda:0"
L2_BYTES = 129e6
GRAVITY = -9.81
GROUND_K, MU = 1e5, 0.5
WORM_OMEGA, WORM_PERIOD = 20.0, 1.0


def listed():
    return [
        # a hard-deadline control loop stepping one small body (the paper's 10^3 cube) on arrays it owns: the
        # smallest call there is, launches and host latency count
        dict(name="control_step", kind="control", a=10, b=10, c=10),
        # the paper's bouncing cube: a display loop that steps one frame and reads the state on the host
        dict(name="cube_frame", kind="frame", a=10, b=10, c=10, steps=50),
        # the paper's own 50^3 lattice (1,558,396 springs): fits the L2
        dict(name="lattice_50", kind="lattice", a=50, b=50, c=50, steps=20),
        # the 1M-mass lattice of the benchmark: larger than the L2, streamed from HBM every step
        dict(name="lattice_100", kind="lattice", a=100, b=100, c=100, steps=10),
        # an unstructured kNN mesh in random index order, resting on the ground
        dict(name="mesh_500k", kind="mesh", points=500_000, knn=8, steps=10),
        # the paper's swarm: 100 worms of 27 x 5 x 3 masses in one system, worm actuation, on the ground
        dict(name="worms_100", kind="worms", worms=100, a=27, b=5, c=3, steps=20),
        # a design sweep: many actuated robots of mixed sizes rolled out together, launch shapes tuned once
        dict(name="robots_1024", kind="robots", robots=1024, lo=3, hi=12, steps=200, tuned=True),
        # a screened search generation: 64 voxel robots, default launch shapes, their fitness read back
        dict(name="voxels_64", kind="voxels", robots=64, grid=8, steps=1000),
        # gradient-based design: displacement of each robot and its gradient in every amplitude and phase
        dict(name="adjoint_256", kind="adjoint", robots=256, lo=3, hi=12, steps=100, every=50),
        # the surrogate ranking one generation of 1024 mutants
        dict(name="mlp_predict_1024", kind="predict", batch=1024, n_in=1024, hidden=512),
        # the surrogate's training: a few optimiser steps, then the parameters are read
        dict(name="mlp_train_4096", kind="train", batch=4096, n_in=1024, hidden=512, steps=8),
        # the tensor-core product alone, large
        dict(name="gemm_8192", kind="gemm", m=8192, n=8192, k=8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["control", "frame", "lattice", "lattice", "mesh", "worms", "robots", "voxels", "adjoint",
                       "predict", "train", "gemm"])
    if kind == "control":
        return dict(kind=kind, a=_log_int(rng, 2, 40), b=_log_int(rng, 2, 40), c=_log_int(rng, 2, 40))
    if kind == "frame":
        return dict(kind=kind, a=rng.randint(2, 12), b=rng.randint(2, 12), c=rng.randint(2, 12),
                    steps=_log_int(rng, 1, 60))
    if kind == "lattice":
        return dict(kind=kind, a=_log_int(rng, 14, 100), b=_log_int(rng, 14, 100), c=_log_int(rng, 14, 100),
                    steps=rng.randint(2, 10))
    if kind == "mesh":
        return dict(kind=kind, points=_log_int(rng, 4_000, 500_000), knn=rng.randint(4, 10), steps=rng.randint(2, 10))
    if kind == "worms":
        return dict(kind=kind, worms=_log_int(rng, 12, 120), a=rng.randint(9, 27), b=rng.randint(3, 5),
                    c=rng.randint(2, 4), steps=rng.randint(2, 24))
    if kind == "robots":
        return dict(kind=kind, robots=_log_int(rng, 32, 1024), lo=3, hi=rng.randint(6, 12),
                    steps=_log_int(rng, 20, 200), tuned=rng.random() < 0.5)
    if kind == "voxels":
        return dict(kind=kind, robots=_log_int(rng, 16, 256), grid=rng.choice([5, 6, 7, 8]),
                    steps=_log_int(rng, 50, 1000))
    if kind == "adjoint":
        return dict(kind=kind, robots=_log_int(rng, 2, 256), lo=3, hi=rng.randint(5, 12), steps=rng.randint(10, 100),
                    every=rng.choice([7, 20, 50]))
    if kind == "predict":
        return dict(kind=kind, batch=128 * _log_int(rng, 1, 64), n_in=128 * rng.randint(2, 10),
                    hidden=128 * rng.randint(1, 8))
    if kind == "train":
        return dict(kind=kind, batch=128 * _log_int(rng, 1, 64), n_in=128 * rng.randint(2, 10),
                    hidden=128 * rng.randint(1, 8), steps=rng.randint(2, 8))
    return dict(kind=kind, m=128 * _log_int(rng, 1, 64), n=128 * _log_int(rng, 1, 64), k=64 * _log_int(rng, 2, 128))


# ------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=4)
def _box(a, b, c):
    """Sites and 26-neighbour springs of an a x b x c lattice (pitch 0.1 m)."""
    pos = inputs.lattice_points(a, b, c, 0.1)
    ends = inputs.lattice_springs(a, b, c)
    return pos, ends, _lengths(pos, ends)


@functools.lru_cache(maxsize=2)
def _mesh(points, knn):
    """Random points of the unit cube and the springs to their nearest neighbours, in random order."""
    rng = np.random.default_rng([points, knn])
    pos = rng.uniform(0.0, 1.0, (points, 3))
    ends = inputs.knn_pairs(pos, knn)
    ends = np.ascontiguousarray(ends[rng.permutation(len(ends))])
    return pos, ends, _lengths(pos, ends)


def _lengths(pos, ends):
    e = ends.astype(np.int64)
    return np.sqrt(((pos[e[:, 1]] - pos[e[:, 0]]) ** 2).sum(axis=1))


def _system(rng, pos, ends, rest, *, k, damping, mass, dt, ground, fixed=None, vel=None, spacing=0.1):
    n, s = len(pos), len(ends)
    return inputs.System(pos=pos, vel=np.zeros_like(pos) if vel is None else vel, mass=np.full(n, mass),
                         fixed=np.zeros(n, np.uint8) if fixed is None else fixed, ends=ends,
                         k=np.full(s, k) if np.isscalar(k) else k, rest=rest, damping=np.full(s, damping), dt=dt,
                         ground=ground, ground_k=GROUND_K, mu=MU, spacing=spacing)


def _cube(case, rng):
    """A cube tossed at the ground: it lands within the first steps."""
    pos, ends, length = _box(case["a"], case["b"], case["c"])
    vel = np.tile(rng.uniform(-1.0, 1.0, 3) - [0, 0, 1.5], (len(pos), 1)) + rng.normal(0.0, 0.05, pos.shape)
    return _system(rng, pos + [0, 0, 1e-3], ends, length * rng.uniform(0.98, 1.02, len(ends)), k=1e4, damping=1.0,
                   mass=0.1, dt=1e-4, ground=True, vel=vel)


def _lattice(case, rng):
    """The benchmark's lattice: perturbed rest lengths, lognormal stiffness, fixed base."""
    pos, ends, length = _box(case["a"], case["b"], case["c"])
    fixed = np.zeros(len(pos), np.uint8)
    fixed[: case["a"] * case["b"]] = 1
    return _system(rng, pos, ends, length * rng.uniform(0.95, 1.05, len(ends)),
                   k=1e4 * np.exp(0.5 * rng.standard_normal(len(ends))), damping=1.0, mass=0.1, dt=5e-5, ground=False,
                   fixed=fixed)


def _mesh_system(case, rng):
    pos, ends, length = _mesh(case["points"], case["knn"])
    spacing = float(np.cbrt(1.0 / len(pos)))
    vel = np.tile(rng.uniform(-0.2, 0.2, 3), (len(pos), 1)) + rng.normal(0.0, 0.02, pos.shape)
    return _system(rng, pos, ends, length * rng.uniform(0.95, 1.05, len(ends)), k=5e3, damping=0.5, mass=1e-3,
                   dt=2e-5, ground=True, vel=vel, spacing=spacing)


def _worms(case, rng):
    """The swarm side by side on one grid, each crawling; the wave of rest lengths runs along the body."""
    pos1, ends1, length1 = _box(case["a"], case["b"], case["c"])
    n1, s1, w = len(pos1), len(ends1), case["worms"]
    side = max(1, int(round(math.sqrt(w * case["b"] / case["a"]))))          # worms per row of the swarm
    at = np.array([[(i % side) * (case["a"] + 3) * 0.1, (i // side) * (case["b"] + 3) * 0.1, 0.0] for i in range(w)])
    pos = (pos1[None] + at[:, None]).reshape(-1, 3)
    ends = (ends1[None].astype(np.int64) + n1 * np.arange(w)[:, None, None]).reshape(-1, 2).astype(np.uint32)
    vel = np.repeat(np.concatenate([rng.uniform(-0.5, 0.5, (w, 2)), np.zeros((w, 1))], axis=1), n1, axis=0)
    vel = vel + rng.normal(0.0, 0.02, vel.shape)
    sy = _system(rng, pos, ends, np.tile(length1, w), k=1e4, damping=1.0, mass=0.1, dt=1e-4, ground=True, vel=vel)
    # offset by half a step: the jump of the rest length at each period never falls on a step boundary
    x = pos1[ends1[:, 0].astype(np.int64), 0] / (0.1 * case["a"])
    off = np.floor((x[None] + rng.uniform(0.0, 1.0, (w, 1))) % 1.0 / sy.dt) * sy.dt + 0.5 * sy.dt
    amp = np.where(rng.random((w, s1)) < 0.5, 0.1, 0.0)
    return sy, amp.reshape(-1).astype(np.float32), off.reshape(-1).astype(np.float32)


def _push(rng, sy, swing=0.05):
    """A robot met in mid-gait: moving along the ground, its masses swinging a little."""
    sy.vel = np.tile(np.append(rng.uniform(-0.5, 0.5, 2), -0.1), (sy.n_masses, 1)) + rng.normal(0.0, swing, sy.pos.shape)
    return sy


def _robots(case, rng, swing=0.05):
    """Mixed lattice robots resting on the ground, 30 % of their springs actuated."""
    dims = np.random.default_rng(case["robots"]).integers(case["lo"], case["hi"] + 1, (case["robots"], 3))
    out = []
    for a, b, c in dims:
        a, b, c = int(a), int(b), int(c)
        pos, ends, length = _robot_box(a, b, c)
        s = len(ends)
        act = rng.random(s) < 0.3
        sy = _system(rng, pos, ends, length, k=1e4, damping=1.0, mass=0.1, dt=1e-4, ground=True)
        sy.act_amp = np.where(act, rng.uniform(0.0, 0.2, s), 0.0)
        sy.act_phase = np.where(act, rng.uniform(0.0, 2.0 * np.pi, s), 0.0)
        sy.act_freq = 2.0
        out.append(_push(rng, sy, swing))
    return out


_robot_box = functools.lru_cache(maxsize=None)(_box.__wrapped__)     # at most 10^3 small boxes


@functools.lru_cache(maxsize=2)
def _shapes(robots, grid):
    """The voxel bodies of one generation."""
    rng = np.random.default_rng([robots, grid])
    return [inputs.voxel_morphology(rng, grid, 0.6) for _ in range(robots)]


def _voxels(case, rng):
    return [_push(rng, inputs.voxel_robot(occ, rng.uniform(0.0, 2.0 * np.pi, occ.shape)))
            for occ in _shapes(case["robots"], case["grid"])]


def _mlp_params(rng, n_in, hidden):
    """Weights as a trained network has them, flat: W1^T, b1, W2^T, b2, W3^T, b3, w4, b4."""
    parts = []
    for fan in (n_in, hidden, hidden):
        parts += [rng.standard_normal(hidden * fan) * math.sqrt(1.6 / fan), 0.1 * rng.standard_normal(hidden)]
    parts += [rng.standard_normal(hidden) / math.sqrt(hidden), 0.1 * rng.standard_normal(1)]
    return np.concatenate(parts).astype(np.float32)


def _features(seed, batch, n_in):
    """Occupancy bits, then phases in [-1, 1), zero where empty."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    occ = (torch.rand(batch, n_in // 2, device=DEV, generator=g) < 0.6).float()
    ph = torch.rand(batch, n_in // 2, device=DEV, generator=g) * 2 - 1
    x = torch.cat([occ, occ * ph], dim=1).bfloat16().contiguous()
    return x, torch.randn(batch, device=DEV, generator=g)


def _mlp_inputs(case, seed):
    p = _mlp_params(np.random.default_rng([seed, 1]), case["n_in"], case["hidden"])
    return (p, *_features(seed, case["batch"], case["n_in"]))


def _gemm_inputs(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    A = torch.randn(case["m"], case["k"], device=DEV, generator=g).bfloat16()
    B = torch.randn(case["n"], case["k"], device=DEV, generator=g).bfloat16()
    return A, B


def _control_inputs(case, seed):
    sy = _cube(case, np.random.default_rng(seed))
    f = lambda x: torch.tensor(x, dtype=torch.float32, device=DEV)  # noqa: E731
    return sy, dict(pos=f(sy.pos), vel=f(sy.vel), inv=f(1.0 / sy.mass), k=f(sy.k), rest=f(sy.rest),
                    ends=torch.tensor(sy.ends.astype(np.int32), device=DEV))


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    kind, rng, st = case["kind"], np.random.default_rng(seed), dict(case=case)
    if kind == "control":
        sy, st["dev"] = _control_inputs(case, seed)
        p = T.titan_default_params()
        p.dt, p.ground, p.ground_k, p.mu = sy.dt, 1, sy.ground_k, sy.mu
        st.update(params=p, n=sy.n_masses, s=sy.n_springs, pos=torch.empty_like(st["dev"]["pos"]),
                  vel=torch.empty_like(st["dev"]["vel"]))
    elif kind in ("frame", "lattice", "mesh", "worms"):
        if kind == "worms":
            sy, amp, off = _worms(case, rng)
        else:
            sy = {"frame": _cube, "lattice": _lattice, "mesh": _mesh_system}[kind](case, rng)
        st["sim"] = T.Sim(sy)
        if kind == "worms":
            T.titan_set_worm_actuation(st["sim"].handle, np.arange(sy.n_springs), amp, off, WORM_OMEGA, WORM_PERIOD)
        if kind != "frame":
            st.update(pos=torch.empty(sy.n_masses, 3, device=DEV), vel=torch.empty(sy.n_masses, 3, device=DEV))
    elif kind in ("robots", "voxels"):
        st["batch"] = T.Batch((_robots if kind == "robots" else _voxels)(case, rng))
        if case.get("tuned"):
            st["batch"].autotune()
    elif kind == "adjoint":
        f = T.CentroidRollout(_robots(case, rng, 0.0), case["steps"], every=case["every"])
        t = lambda x: torch.tensor(x, dtype=torch.float32, device=DEV, requires_grad=True)  # noqa: E731
        st.update(f=f, amp=t(f.system.act_amp), phase=t(f.system.act_phase),
                  w=torch.tensor(rng.uniform(0.5, 1.5, case["robots"]), dtype=torch.float32, device=DEV))
    elif kind in ("predict", "train"):
        p, x, t = _mlp_inputs(case, seed)
        net = T.MLP(case["n_in"], case["hidden"], seed=0)
        net.set_params(p)
        st.update(net=net, x=x, t=t, y=torch.empty(case["batch"], device=DEV), loss=torch.empty(1, device=DEV))
    else:
        A, B = _gemm_inputs(case, seed)
        st.update(A=A, B=B, C=torch.empty(case["m"], case["n"], device=DEV))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "control":
        d = st["dev"]
        T.titan_step_atomic_noalloc(st["n"], d["pos"], d["vel"], d["inv"], st["s"], d["ends"], d["k"], d["rest"], 1.0,
                                    st["params"], st["pos"], st["vel"])
        return dict(pos=st["pos"], vel=st["vel"])
    if kind == "frame":
        pos, vel, _ = st["sim"].step(case["steps"]).snapshot()
        return dict(pos=pos, vel=vel)
    if kind in ("lattice", "mesh", "worms"):
        st["sim"].step(case["steps"])
        T.titan_read_state_dev(st["sim"].handle, st["pos"], st["vel"])
        return dict(pos=st["pos"], vel=st["vel"])
    if kind in ("robots", "voxels"):
        b = st["batch"]
        b.reset()
        b.rollout(case["steps"])
        return dict(centroids=b.centroids())           # what decides each robot's fitness
    if kind == "adjoint":
        d = st["f"](st["amp"], st["phase"])
        ga, gp = torch.autograd.grad(d, (st["amp"], st["phase"]), st["w"])
        return dict(displacement=d.detach(), grad_amp=ga, grad_phase=gp)
    if kind == "predict":
        st["net"].forward(st["x"], st["y"])
        return dict(y=st["y"])
    if kind == "train":
        for _ in range(case["steps"]):
            st["net"].train_step(st["x"], st["t"], 1e-3, st["loss"])
        return dict(params=st["net"].get_params(), loss=st["loss"])
    T.titan_gemm_bf16_tn(st["A"], st["B"], st["C"])
    return dict(C=st["C"])


# ------------------------------------------------------------------ what a pass cannot do without

def _counts(case):
    """Masses and springs of a case's system (over all its bodies)."""
    kind = case["kind"]
    if kind == "mesh":
        return case["points"], len(_mesh(case["points"], case["knn"])[1])
    if kind in ("control", "frame", "lattice", "worms"):
        a, b, c = case["a"], case["b"], case["c"]
        w = case.get("worms", 1)
        return w * a * b * c, w * inputs.lattice_spring_count(a, b, c)
    if kind == "voxels":                                 # what Bernoulli(0.6) voxels come to
        g = case["grid"]
        return int(0.6 * g ** 3 * case["robots"]), int(0.36 * inputs.lattice_spring_count(g, g, g) * case["robots"])
    dims = np.random.default_rng(case["robots"]).integers(case["lo"], case["hi"] + 1, (case["robots"], 3))
    return (int(sum(a * b * c for a, b, c in dims.tolist())),
            int(sum(inputs.lattice_spring_count(a, b, c) for a, b, c in dims.tolist())))


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 2.0 * (m * k + n * k) + 4.0 * m * n, "flops": 2.0 * m * n * k}
    if kind in ("predict", "train"):
        b, i, h = case["batch"], case["n_in"], case["hidden"]
        params = h * i + 2 * h * h + 4 * h + 1
        fwd = 2.0 * b * (i * h + 2 * h * h)
        if kind == "predict":
            return {"bytes": 2.0 * b * i + 2.0 * params + 4.0 * b, "flops": fwd}
        # weights and both moments are read and written, the gradients formed, each step
        return {"bytes": case["steps"] * (2.0 * b * i + 4.0 * b + 24.0 * params),
                "flops": case["steps"] * (3 * fwd - 2.0 * b * i * h)}
    n, s = _counts(case)
    actuated = kind in ("worms", "robots", "voxels", "adjoint")
    spring = 16.0 + (8.0 if actuated else 0.0)           # both ends, k, rest length, actuation
    steps = case.get("steps", 1)
    flops = steps * (33.0 * s + 15.0 * n)
    if kind == "adjoint":                                # the rollout, then forward again and back
        return {"bytes": spring * s + 52.0 * n + 8.0 * s, "flops": 4.0 * flops}
    once = spring * s + 52.0 * n
    # springs and states that fit on the chip are read once a pass, larger ones once a step
    return {"bytes": once * (steps if once > L2_BYTES else 1), "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits

class _Body:
    """The springs and masses of one system as FP64 tensors, and one time step of it."""

    def __init__(self, systems, amp=None, phase=None, worm=None):
        cat = lambda f: torch.tensor(np.concatenate([np.asarray(getattr(s, f), np.float64) for s in systems]), device=DEV)  # noqa: E731
        first = np.cumsum([0] + [len(s.pos) for s in systems])
        ends = np.concatenate([s.ends.astype(np.int64) + o for s, o in zip(systems, first)])
        s0 = systems[0]
        self.first = first
        self.i, self.j = (torch.tensor(np.ascontiguousarray(ends[:, e]), device=DEV) for e in (0, 1))
        self.x, self.v, self.m, self.k, self.L0, self.c = (cat(f) for f in ("pos", "vel", "mass", "k", "rest", "damping"))
        self.free = (cat("fixed") == 0).double()[:, None]
        self.dt, self.ground = s0.dt, s0.ground
        self.worm, self.amp, self.phase = worm, amp, phase
        if amp is None and s0.act_amp is not None:
            self.amp, self.phase = cat("act_amp"), cat("act_phase")
        self.freq = s0.act_freq

    def length(self, n, amp, phase):
        if amp is None:
            return self.L0
        t = n * self.dt
        if self.worm:
            return self.L0 * (1 + amp * torch.sin(WORM_OMEGA * torch.remainder(t - phase, WORM_PERIOD)))
        return self.L0 * (1 + amp * torch.sin(2 * math.pi * self.freq * t + phase))

    def step(self, n, x, v, amp, phase):
        d = x[self.j] - x[self.i]
        l = d.square().sum(1).sqrt()
        u = d / l[:, None]
        f = self.k * (l - self.length(n, amp, phase)) + self.c * ((v[self.j] - v[self.i]) * u).sum(1)
        F = torch.zeros_like(x).index_add(0, self.i, f[:, None] * u).index_add(0, self.j, -f[:, None] * u)
        a = F / self.m[:, None] + torch.tensor([0.0, 0.0, GRAVITY], dtype=torch.float64, device=DEV)
        if self.ground:
            an = GROUND_K * (-x[:, 2]).clamp(min=0) / self.m
            vt2 = v[:, :2].square().sum(1)
            some = vt2 > 0
            vt = torch.where(some, vt2, torch.ones_like(vt2)).sqrt()
            fr = torch.where(some, torch.minimum(MU * an, vt / self.dt), torch.zeros_like(vt))
            a = a + torch.cat([-(fr / vt)[:, None] * v[:, :2], an[:, None]], dim=1)
        v1 = (v + a * self.dt) * self.free
        return x + v1 * self.dt, v1

    def rollout(self, steps, keep=None):
        x, v = self.x, self.v
        for n in range(steps):
            if keep is not None:
                keep.append((x, v))
            x, v = self.step(n, x, v, self.amp, self.phase)
        return x, v

    def centroids(self, x):
        x = x.cpu().numpy()
        return np.stack([x[a:b].mean(axis=0) for a, b in zip(self.first[:-1], self.first[1:])])


def _exact_adjoint(case, rng):
    robots = _robots(case, rng, 0.0)
    w = torch.tensor(rng.uniform(0.5, 1.5, case["robots"]), dtype=torch.float32, device=DEV).double()
    b = _Body(robots)
    amp, phase = b.amp.float().double(), b.phase.float().double()     # the tensors the pass is given
    b.amp, b.phase = amp, phase
    kept = []
    x, _ = b.rollout(case["steps"], kept)
    disp = torch.tensor((b.centroids(x) - b.centroids(b.x))[:, 0])
    size = torch.tensor(np.diff(b.first), device=DEV)
    gx = torch.zeros_like(x)
    gx[:, 0] = torch.repeat_interleave(w / size, size)
    gv, ga, gp = torch.zeros_like(x), torch.zeros_like(amp), torch.zeros_like(phase)
    for n in reversed(range(case["steps"])):
        args = [t.detach().requires_grad_() for t in (*kept.pop(), amp, phase)]
        with torch.enable_grad():
            out = b.step(n, *args)
        gx, gv, da, dp = torch.autograd.grad(out, args, (gx, gv))
        ga += da
        gp += dp
    return dict(displacement=disp, grad_amp=ga, grad_phase=gp)


def _unpack(p, n_in, hidden):
    out, o = [], 0
    for shape in [(hidden, n_in), (hidden,), (hidden, hidden), (hidden,), (hidden, hidden), (hidden,), (hidden,), (1,)]:
        size = math.prod(shape)
        out.append(p[o:o + size].view(shape))
        o += size
    return out


def _net(x, p, n_in, hidden):
    w1, b1, w2, b2, w3, b3, w4, b4 = _unpack(p, n_in, hidden)
    for w, b in ((w1, b1), (w2, b2), (w3, b3)):
        x = torch.nn.functional.gelu(x @ w.T + b)
    return x @ w4 + b4


def exact(case, seed):
    kind, rng = case["kind"], np.random.default_rng(seed)
    if kind == "control":
        sy, d = _control_inputs(case, seed)
        b = _Body([sy])
        b.x, b.v, b.k, b.L0 = (d[f].double() for f in ("pos", "vel", "k", "rest"))
        b.m = 1 / d["inv"].double()
        x, v = b.rollout(1)
        return dict(pos=x, vel=v)
    if kind in ("frame", "lattice", "mesh"):
        b = _Body([{"frame": _cube, "lattice": _lattice, "mesh": _mesh_system}[kind](case, rng)])
    elif kind == "worms":
        sy, amp, off = _worms(case, rng)
        b = _Body([sy], *(torch.tensor(t, dtype=torch.float64, device=DEV) for t in (amp, off)), worm=True)
    elif kind in ("robots", "voxels"):
        b = _Body((_robots if kind == "robots" else _voxels)(case, rng))
        x, _ = b.rollout(case["steps"])
        return dict(centroids=b.centroids(x))
    elif kind == "adjoint":
        return _exact_adjoint(case, rng)
    elif kind in ("predict", "train"):
        p, x, t = _mlp_inputs(case, seed)
        p, x, t = torch.tensor(p, device=DEV).double(), x.double(), t.double()
        if kind == "predict":
            return dict(y=_net(x, p, case["n_in"], case["hidden"]))
        m, v = torch.zeros_like(p), torch.zeros_like(p)
        for n in range(1, case["steps"] + 1):              # Adam, beta 0.9 and 0.999, eps 1e-8
            q = p.detach().requires_grad_()
            loss = (_net(x, q, case["n_in"], case["hidden"]) - t).square().mean()
            g, = torch.autograd.grad(loss, q)
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - 1e-3 * (m / (1 - 0.9 ** n)) / ((v / (1 - 0.999 ** n)).sqrt() + 1e-8)
        return dict(params=p, loss=loss.detach().view(1))
    else:
        A, B = _gemm_inputs(case, seed)
        return dict(C=A.double() @ B.double().T)
    x, v = b.rollout(case["steps"])
    return dict(pos=x, vel=v)
