"""The workloads the library's speed is measured on.

Each case is one pass of something a program linked against the library does
over and over: a force evaluation of new bodies, a run of leapfrog steps, a
fast multipole evaluation, a direct-sum check, a training run of the
correction network.  The bodies are synthetic (Plummer spheres, uniform
cubes, colliding spheres), drawn on the GPU from the seed alone; opening
angles, softenings and leaf thresholds are the ones the benchmark and the
tests use.  Everything goes through ``tc.Context``; results are read into the
caller's device buffers, as a simulation that keeps its state on the GPU
does.
"""
from __future__ import annotations

import ctypes
import math
import random

import numpy as np
import torch

from paper_1211_2293_gb300 import tc

_EXACT_PAIRS = 2.0e10  # body pairs an FP64 direct sum gets through in seconds


class _Program(tc.Context):
    """A context whose results and training data stay in device memory."""

    def state_into(self, pos: torch.Tensor, vel: torch.Tensor):
        self._c(self._lib.tc_get_state(self._h, ctypes.c_void_p(pos.data_ptr()), ctypes.c_void_p(vel.data_ptr())))

    def train(self, X, T, F, epochs, batch, lr, seed, band, losses):
        self._c(self._lib.tc_mlp_train(self._h, *(ctypes.c_void_p(t.data_ptr()) for t in (X, T, F)),
                                       tc.TC_MLP_FACTORS, X.shape[0], epochs, batch, lr, seed, band,
                                       ctypes.c_void_p(losses.ctypes.data)))

    def model_into(self, model: torch.Tensor):
        self._c(self._lib.tc_mlp_get(self._h, ctypes.c_void_p(model.data_ptr()), None))


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest calls: one force evaluation of a few thousand new
        # bodies (the library's reference configuration), where launches and
        # host round trips count
        dict(name="eval_plummer_4k", kind="eval", shape="plummer", n=4096, theta=0.5, eps=0.01, leaf=8,
             walk="monopole", pot=False, precise=True),
        # a small simulation at the smallest of the paper's sizes (10k
        # bodies): leapfrog steps replayed back to back, then the state
        dict(name="steps_plummer_10k", kind="steps", shape="plummer", n=10007, theta=0.5, eps=0.01, leaf=8,
             steps=4, dt=1e-3),
        # the paper's largest size (100k bodies) with the potential, as an
        # energy check needs
        dict(name="eval_pot_100k", kind="eval", shape="two_plummer", n=100003, theta=0.6, eps=0.01, leaf=16,
             walk="monopole", pot=True, precise=True),
        # the uniform cube of the benchmark, integrated
        dict(name="steps_uniform_1m", kind="steps", shape="uniform", n=1 << 20, theta=0.5, eps=1e-3, leaf=16,
             steps=2, dt=1e-4),
        # the benchmark's sphere at the opening angle of a 1e-3 error: the
        # plain walk from new positions to accelerations
        dict(name="eval_plummer_4m", kind="eval", shape="plummer", n=1 << 22, theta=0.62, eps=1e-3, leaf=16,
             walk="monopole", pot=False, precise=True),
        # the same sphere with the learned far-field correction at its own
        # 1e-3 opening angle
        dict(name="learned_plummer_4m", kind="eval", shape="plummer", n=1 << 22, theta=0.67, eps=1e-3, leaf=16,
             walk="learned", pot=False, precise=True, band=0.55),
        # the quadrupole walk at its 1e-3 opening angle
        dict(name="quadrupole_plummer_1m", kind="eval", shape="plummer", n=1000003, theta=0.68, eps=1e-3, leaf=16,
             walk="quadrupole", pot=False, precise=True),
        # the largest calls: two colliding spheres of 8M bodies each
        dict(name="eval_two_plummer_16m", kind="eval", shape="two_plummer", n=1 << 24, theta=0.75, eps=5e-4, leaf=16,
             walk="monopole", pot=False, precise=True),
        # a batch of uneven independent systems, one step of all of them
        dict(name="steps_batch_512", kind="steps", shape="batch", nsys=512, lo=1024, hi=65536, sizes=1, theta=0.6,
             eps=0.01, leaf=8, steps=1, dt=1e-3),
        # the fast multipole method on new bodies
        dict(name="fmm_plummer_1m", kind="fmm", shape="plummer", n=1000003, theta=0.55, eps=1e-3, leaf=16),
        # the accuracy check of every run: direct sums of sampled bodies
        dict(name="direct_4k_of_1m", kind="direct", shape="plummer", n=1 << 20, targets=4096, eps=1e-3),
        # training the correction network: one pass over the pairs
        dict(name="train_256k", kind="train", pairs=1 << 18, batch=1024, epochs=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["eval", "eval", "eval", "steps", "steps", "batch", "quadrupole", "learned", "fmm", "direct",
                       "train"])
    leaf = rng.choice([8, 16, 32])
    eps = rng.choice([1e-2, 1e-3, 5e-4])
    shape = rng.choice(["plummer", "uniform", "two_plummer"])
    if kind == "eval":
        n = _log_int(rng, 1000, 1 << 23)
        return dict(kind="eval", shape=shape, n=n, theta=round(rng.uniform(0.5, 0.8), 3), eps=eps, leaf=leaf,
                    walk="monopole", pot=rng.random() < 0.4, precise=rng.random() < 0.8)
    if kind == "quadrupole":
        return dict(kind="eval", shape=shape, n=_log_int(rng, 1000, 1 << 21), theta=round(rng.uniform(0.55, 0.9), 3),
                    eps=eps, leaf=leaf, walk="quadrupole", pot=rng.random() < 0.5, precise=True)
    if kind == "learned":
        return dict(kind="eval", shape="plummer", n=_log_int(rng, 4000, 1 << 22),
                    theta=round(rng.uniform(0.6, 0.9), 3), eps=1e-3, leaf=16, walk="learned", pot=False, precise=True,
                    band=rng.choice([0.5, 0.55, 0.6]))
    if kind == "steps":
        return dict(kind="steps", shape=shape, n=_log_int(rng, 1000, 1 << 21), theta=round(rng.uniform(0.5, 0.8), 3),
                    eps=eps, leaf=leaf, steps=rng.choice([1, 2, 4]), dt=1e-4)
    if kind == "batch":
        return dict(kind="steps", shape="batch", nsys=_log_int(rng, 2, 512), lo=rng.choice([1, 100, 1024]),
                    hi=rng.choice([4096, 65536]), sizes=rng.randrange(1 << 16), theta=round(rng.uniform(0.5, 0.8), 3),
                    eps=0.01, leaf=leaf, steps=rng.choice([1, 2]), dt=1e-4)
    if kind == "fmm":
        return dict(kind="fmm", shape=shape, n=_log_int(rng, 1000, 1 << 21), theta=round(rng.uniform(0.4, 0.7), 3),
                    eps=eps, leaf=leaf)
    if kind == "direct":
        return dict(kind="direct", shape=shape, n=_log_int(rng, 1000, 1 << 22), targets=_log_int(rng, 1, 8192),
                    eps=eps)
    return dict(kind="train", pairs=_log_int(rng, 2000, 1 << 19), batch=rng.choice([256, 1000, 1024, 4096]),
                epochs=1)


# ----------------------------------------------------------------- inputs
def _plummer(n, g, velocity=False):
    """A Plummer sphere of unit mass and scale, cut at radius 10."""
    f = dict(device="cuda", dtype=torch.float64, generator=g)
    edge = (100.0 / 101.0) ** 1.5  # enclosed mass at the cut
    m = torch.rand(n, **f).clamp_(min=1e-12) * edge
    r = (m.pow(-2.0 / 3.0) - 1.0).rsqrt()
    d = torch.randn(n, 3, **f)
    pos = d * (r / d.norm(dim=1)).unsqueeze(1)
    if not velocity:
        return pos, None
    # the speed over the local escape speed, squared, is Beta(3/2, 9/2)
    a = torch.randn(n, 3, **f).square_().sum(1)
    b = torch.zeros(n, device="cuda", dtype=torch.float64)
    for _ in range(3):
        b += torch.randn(n, 3, **f).square_().sum(1)
    speed = (a / (a + b)).sqrt() * math.sqrt(2.0) * (1.0 + r * r).pow(-0.25)
    d = torch.randn(n, 3, **f)
    return pos, d * (speed / d.norm(dim=1)).unsqueeze(1)


def _sizes(case):
    """Bodies of each system of a case."""
    if case["shape"] != "batch":
        return [case["n"]]
    rng = random.Random(case["sizes"])
    return [_log_int(rng, case["lo"], case["hi"]) for _ in range(case["nsys"])]


def _bodies(case, seed, velocity=False):
    """(pos, vel or None, mass) on the GPU, float32."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["shape"] == "batch":
        sizes = _sizes(case)
        pos, vel = _plummer(sum(sizes), g, velocity)
        mass = torch.cat([torch.full((k,), 1.0 / k, device="cuda") for k in sizes])
    else:
        n = case["n"]
        mass = torch.full((n,), 1.0 / n, device="cuda")
        if case["shape"] == "uniform":
            pos = torch.rand(n, 3, device="cuda", dtype=torch.float64, generator=g) * 2.0 - 1.0
            vel = torch.zeros_like(pos) if velocity else None
        else:
            pos, vel = _plummer(n, g, velocity)
            if case["shape"] == "two_plummer":
                # two spheres of half the mass each, approaching along x
                side = torch.ones(n, device="cuda", dtype=torch.float64)
                side[: n // 2] = -1.0
                pos[:, 0] += 3.0 * side
                if velocity:
                    vel *= math.sqrt(0.5)
                    vel[:, 0] -= 0.25 * side
    return pos.float().contiguous(), None if vel is None else vel.float().contiguous(), mass


def _model(seed):
    """A network in the library's packing: weights uniform in 1/sqrt(fan-in),
    feature maps of the order that walks at these opening angles meet."""
    rng = np.random.RandomState(seed & 0x7FFFFFFF)
    parts = []
    for i, o in ((13, 64), (64, 64), (64, 3)):
        parts += [rng.uniform(-1, 1, (i, o)) / math.sqrt(i), rng.uniform(-1, 1, o) / math.sqrt(i)]
    mean = np.array([0, 0, 0, 0.52, 0.01, 6.0, 1e-3, 0.06, 0, 0, 0.06, 0, 0.06])
    scale = 1.0 / np.array([1.2, 1.2, 1.2, 0.1, 0.02, 3.0, 5e-3, 0.03, 0.02, 0.02, 0.03, 0.02, 0.03])
    parts += [mean, scale, np.full(3, 0.2)]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


def _pairs(n, seed):
    """Training pairs as a walk emits them: features of a cell seen from a
    body, the quadrupole field of its second moments as the label, and the
    factor that turns a label into an acceleration."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    f = dict(device="cuda", dtype=torch.float64, generator=g)
    d = torch.randn(n, 3, **f)
    r = 1.45 + torch.rand(n, **f)  # distance over side
    d *= (r / d.norm(dim=1)).unsqueeze(1)
    count = torch.exp2(1.0 + 11.0 * torch.rand(n, **f)).floor()
    w = torch.randn(n, 3, 3, **f) * 0.12
    q = torch.bmm(w, w.transpose(1, 2)) + 0.04 * torch.eye(3, device="cuda", dtype=torch.float64)
    u = d / r.unsqueeze(1)
    qu = torch.bmm(q, u.unsqueeze(2)).squeeze(2)
    uqu = (qu * u).sum(1, keepdim=True)
    tr = q.diagonal(dim1=1, dim2=2).sum(1, keepdim=True)
    label = (7.5 * uqu - 1.5 * tr) * u - 3.0 * qu
    eps_s = 1e-3 * torch.exp2(6.0 * torch.rand(n, **f))
    six = torch.stack([q[:, 0, 0], q[:, 0, 1], q[:, 0, 2], q[:, 1, 1], q[:, 1, 2], q[:, 2, 2]], 1)
    mfrac = count / float(1 << 20)
    X = torch.cat([d, (1.0 / r).unsqueeze(1), eps_s.unsqueeze(1), count.log2().unsqueeze(1), mfrac.unsqueeze(1), six],
                  1)
    F = mfrac / (r * r).square() * (1e3 * eps_s).square()
    return X.float().contiguous(), label.float().contiguous(), F.float().contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        X, T, F = _pairs(case["pairs"], seed)
        return dict(case=case, ctx=_Program(), X=X, T=T, F=F, losses=np.zeros(case["epochs"], np.float32),
                    model=torch.empty(tc.MLP_NMODEL, device="cuda"))
    pos, vel, mass = _bodies(case, seed, velocity=kind == "steps")
    st = dict(case=case, pos=pos, mass=mass, acc=torch.empty_like(pos))
    if kind == "eval":
        walk = case["walk"]
        ctx = _Program(want_pot=case["pot"], precise=case["precise"], quad=walk != "monopole",
                       quadrupole=walk == "quadrupole")
        if case["pot"]:
            st["pot"] = torch.empty_like(mass)
        if walk == "learned":
            ctx.mlp_set(_model(seed), case["band"])
            ctx.set_config(learned=1)
    elif kind == "steps":
        ctx = _Program()
        if case["shape"] == "batch":
            ctx.build_batch(pos, mass, np.concatenate([[0], np.cumsum(_sizes(case))]), case["leaf"])
        else:
            ctx.build(pos, mass, case["leaf"])
        ctx.set_velocity(vel)
        ctx.forces(case["theta"], case["eps"])
        st.update(out_pos=torch.empty_like(pos), out_vel=torch.empty_like(pos))
    elif kind == "direct":
        ctx = _Program()
        ctx.build(pos, mass, 16)
        st["idx"] = _targets(case, seed)
    else:
        ctx = _Program()
    st["ctx"] = ctx
    return st


def _targets(case, seed):
    """Sampled bodies of a direct-sum check: distinct, in order."""
    k = min(case["targets"], case["n"])
    return np.sort(np.random.RandomState(seed & 0x7FFFFFFF).permutation(case["n"])[:k]).astype(np.int64)


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "eval":
        ctx.build(st["pos"], st["mass"], case["leaf"])
        ctx.forces(case["theta"], case["eps"])
        if case["pot"]:
            ctx.get_acc(acc=st["acc"], pot=st["pot"])
            return dict(acc=st["acc"], pot=st["pot"])
        ctx.get_acc(acc=st["acc"])
        return dict(acc=st["acc"])
    if kind == "steps":
        for _ in range(case["steps"]):
            ctx.step(case["dt"])
        ctx.state_into(st["out_pos"], st["out_vel"])
        ctx.get_acc(acc=st["acc"])
        return dict(pos=st["out_pos"], vel=st["out_vel"], acc=st["acc"])
    if kind == "fmm":
        ctx.build(st["pos"], st["mass"], case["leaf"])
        ctx.fmm(case["theta"], case["eps"])
        ctx.get_acc(acc=st["acc"])
        return dict(acc=st["acc"])
    if kind == "direct":
        acc, pot = ctx.direct(st["idx"], case["eps"])
        return dict(acc=acc, pot=pot)
    ctx.train(st["X"], st["T"], st["F"], case["epochs"], case["batch"], 2e-3, 3, 0.55, st["losses"])
    ctx.model_into(st["model"])
    return dict(model=st["model"], losses=st["losses"].copy())


# ------------------------------------------------------------------- work
def _interactions(n, theta):
    """Interactions per body of a walk, to within tens of per cent: each of
    the tree's levels adds a shell of cells whose number falls with theta;
    small systems run out of bodies."""
    a = 37.0 * max(1.0, math.log2(n) - 2.0) * theta ** -2.3 if n > 1 else 1.0
    return a / (1.0 + a / n)


def work(case):
    kind = case["kind"]
    if kind == "train":
        # 13-64-64-3 forward and backward (two products per weight back)
        n = case["pairs"] * case["epochs"]
        return dict(bytes=case["pairs"] * 4 * (13 + 3 + 1) + 4 * tc.MLP_NMODEL, flops=n * 6 * (13 * 64 + 64 * 64 + 64 * 3))
    if kind == "direct":
        k = min(case["targets"], case["n"])
        return dict(bytes=16 * case["n"] + 40 * k, flops=20.0 * k * case["n"])
    sizes = _sizes(case)
    n = sum(sizes)
    pairs = sum(k * _interactions(k, case["theta"]) for k in sizes)
    if kind == "fmm":
        # leaf-against-leaf sums and low-order expansions: some hundreds of
        # operations' worth of pairs per body at any size
        return dict(bytes=28 * n, flops=20.0 * n * min(n, 100.0 * case["theta"] ** -2))
    if kind == "steps":
        # state read and written, mass read, accelerations written
        return dict(bytes=case["steps"] * (48 + 4 + 12) * n, flops=20.0 * pairs * case["steps"])
    per = 20.0 if case["walk"] != "quadrupole" else 40.0
    return dict(bytes=(28 + 4 * case["pot"]) * n, flops=per * pairs)


# ------------------------------------------------------------------ exact
def _direct64(pos, mass, eps, targets=None, pot=False):
    """Softened direct sum in FP64 by plain torch (G = 1)."""
    x = pos if targets is None else pos[targets]
    me = mass if targets is None else mass[targets]
    acc = torch.empty_like(x)
    phi = torch.empty_like(me)
    block = max(1, (1 << 27) // pos.shape[0])
    for a in range(0, x.shape[0], block):
        d = pos.unsqueeze(0) - x[a:a + block].unsqueeze(1)
        ri = (d.square().sum(2) + eps * eps).rsqrt_()
        if pot:
            phi[a:a + block] = me[a:a + block] / eps - ri @ mass
        w = ri.pow_(3).mul_(mass)
        acc[a:a + block] = torch.bmm(w.unsqueeze(1), d).squeeze(1)
    return (acc, phi) if pot else acc


def exact(case, seed):
    """The sums that the walks and expansions approximate, in FP64: a walk's
    own error at its opening angle (about 1e-3) is part of what is said.
    The learned walk and training have no exact counterpart."""
    kind = case["kind"]
    if kind == "train" or case["shape"] == "batch" or case.get("walk") == "learned":
        return None
    n, eps = case["n"], float(np.float32(case["eps"]))
    if kind == "direct":
        if n * float(case["targets"]) > _EXACT_PAIRS:
            return None
        pos, _, mass = _bodies(case, seed)
        idx = torch.from_numpy(_targets(case, seed)).cuda()
        acc, pot = _direct64(pos.double(), mass.double(), eps, idx, pot=True)
        return dict(acc=acc.cpu().numpy(), pot=pot.cpu().numpy())
    if float(n) * n * (case.get("steps", 0) + 1) > _EXACT_PAIRS:
        return None
    pos, vel, mass = _bodies(case, seed, velocity=kind == "steps")
    pos, mass = pos.double(), mass.double()
    if kind == "steps":
        vel, dt = vel.double(), float(np.float32(case["dt"]))
        acc = _direct64(pos, mass, eps)
        for _ in range(case["steps"]):
            vel = vel + acc * (0.5 * dt)
            pos = pos + vel * dt
            acc = _direct64(pos, mass, eps)
            vel = vel + acc * (0.5 * dt)
        return dict(pos=pos, vel=vel, acc=acc)
    if case.get("pot"):
        acc, pot = _direct64(pos, mass, eps, pot=True)
        return dict(acc=acc, pot=pot)
    return dict(acc=_direct64(pos, mass, eps))
