"""The work that users of this framework have it do, as cases for measuring.

Every case goes through the public entry points of ``paper_2103_00331_gb300``
(the calls of the README): value iteration, policy iteration and single
backups of GridWorlds, batches of GridWorlds, dense CP models, and the learned
warm start (inference and training). ``listed`` gives the fixed ones, ``draw``
more of the same ranges:

* ``vi``     value iteration of one GridWorld (1 to 9 dimensions, FP32 / FP64)
* ``pi``     policy iteration of one GridWorld
* ``backup`` one Bellman backup of a GridWorld with policy and residual
* ``batch``  many uneven GridWorlds solved together, then certified
* ``dense``  one Bellman backup of a dense CP model (FP32, FP64, BF16x3)
* ``dvi``    value iteration of a dense CP model
* ``start``  warm start of a batch of 3-D GridWorlds (coarse value iteration,
             network, upsampling)
* ``train``  one training step of the warm-start network

Grid sizes, slip models, discounts and reward distributions are those of the
repository's configurations, tests and benchmark.
"""
from __future__ import annotations

import math
import os
from types import SimpleNamespace

import numpy as np
import torch

import paper_2103_00331_gb300 as cp
from paper_2103_00331_gb300 import warmstart as ws

FREE, OBSTACLE, TERMINAL = 0, 1, 2
TOL = 1e-6
CH = 64                                    # channels of the warm-start network
PREC = {"f32": cp.F32, "f64": cp.F64, "bf16x3": cp.BF16X3}
WEIGHTS = os.path.join(os.path.dirname(cp.__file__), "data", "warmstart_weights.npz")


# --------------------------------------------------------------------------
# the cases

def listed():
    return [
        # the smallest call: a 10 x 10 FP64 grid solved on its own, bound by latency
        {"name": "vi-10x10-f64", "kind": "vi", "shape": "10x10", "dtype": "f64", "gamma": 0.9, "world": "small"},
        # the benchmark's 64^3 grid, value iteration with the FP64 policy of its result
        {"name": "vi-64^3-f32", "kind": "vi", "shape": "64x64x64", "dtype": "f32", "gamma": 0.99, "world": "goals"},
        # the same grid by policy iteration
        {"name": "pi-64^3-f32", "kind": "pi", "shape": "64x64x64", "dtype": "f32", "gamma": 0.99, "world": "goals"},
        # the largest 2-D grid of the paper's tables, in its double precision
        {"name": "vi-1000x1000-f64", "kind": "vi", "shape": "1000x1000", "dtype": "f64", "gamma": 0.9,
         "world": "paper"},
        # sides as a user's map has them: rows of no multiple of four states
        {"name": "pi-101x97x103-f32", "kind": "pi", "shape": "101x97x103", "dtype": "f32", "gamma": 0.95,
         "world": "goals"},
        # one sweep of a grid that outgrows the cache: the caller's own loop, or a check of a value function
        {"name": "backup-384^3-f32", "kind": "backup", "shape": "384x384x384", "dtype": "f32", "gamma": 0.99,
         "world": "goals"},
        # many uneven instances at once, each with its certificate and policy
        {"name": "batch-1024", "kind": "batch", "count": 1024, "mix": 0},
        # the dense model of the benchmark on the tensor cores: one sweep
        {"name": "dense-64^4-bf16x3", "kind": "dense", "shape": "64x64x64x64", "actions": 8, "rank": 8,
         "dtype": "bf16x3"},
        # a dense model of uneven sides in plain FP32
        {"name": "dense-48x50x52x46-f32", "kind": "dense", "shape": "48x50x52x46", "actions": 4, "rank": 4,
         "dtype": "f32"},
        # a small dense model solved to the end in FP64
        {"name": "dvi-8^4-f64", "kind": "dvi", "shape": "8x8x8x8", "actions": 4, "rank": 3, "dtype": "f64",
         "gamma": 0.9},
        # inference of the warm start, before a batched solve
        {"name": "start-128x64^3", "kind": "start", "count": 128, "shape": "64x64x64"},
        # one minibatch of the warm start's training (its default size)
        {"name": "train-32x64^3", "kind": "train", "count": 32, "shape": "64x64x64"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, ndim, states):
    """Sides of about equal size with ``states`` in all, each off by up to a fifth."""
    side = states ** (1.0 / ndim)
    return "x".join(str(max(2, int(round(side * rng.uniform(0.8, 1.2))))) for _ in range(ndim))


def draw(rng):
    kind = rng.choice(["vi", "vi", "vi", "pi", "pi", "backup", "batch", "dense", "dense", "dvi", "start", "train"])
    gamma = round(rng.uniform(0.9, 0.99), 4)
    dtype = rng.choice(["f32", "f64"])
    if kind in ("vi", "pi"):
        ndim = rng.choice([1, 2, 2, 3, 3, 3, 4, 6, 9] if kind == "vi" else [1, 2, 3])
        states = _log_int(rng, 2 ** ndim * 4 if ndim > 6 else 40, 600_000 if dtype == "f32" else 200_000)
        return {"kind": kind, "shape": _shape(rng, ndim, states), "dtype": dtype, "gamma": min(gamma, 0.96),
                "world": rng.choice(["small", "goals"])}
    if kind == "backup":
        ndim = rng.choice([2, 3, 3, 3])
        states = _log_int(rng, 10_000, 40_000_000 if dtype == "f32" else 4_000_000)
        return {"kind": kind, "shape": _shape(rng, ndim, states), "dtype": dtype, "gamma": gamma, "world": "goals"}
    if kind == "batch":
        return {"kind": kind, "count": _log_int(rng, 16, 700), "mix": rng.randrange(1 << 20)}
    if kind == "dense":
        ndim = rng.choice([2, 3, 4])
        states = _log_int(rng, 5_000, 4_000_000 if ndim > 2 else 500_000)
        if dtype == "f64":
            states = min(states, 60_000 + states // 20)
        return {"kind": kind, "shape": _shape(rng, ndim, states), "actions": rng.randint(2, 8),
                "rank": rng.randint(1, 4), "dtype": dtype}
    if kind == "dvi":
        return {"kind": kind, "shape": _shape(rng, rng.choice([2, 3, 4]), _log_int(rng, 100, 8_000)),
                "actions": rng.randint(2, 6), "rank": rng.randint(1, 4), "dtype": dtype,
                "gamma": round(rng.uniform(0.8, 0.92), 4)}
    side = rng.randint(17, 64)
    shape = "x".join(str(max(9, side - rng.randint(0, 6))) for _ in range(3))
    return {"kind": kind, "count": _log_int(rng, 4, 120 if kind == "start" else 30), "shape": shape}


def _dims(case):
    return tuple(int(n) for n in case["shape"].split("x"))


# --------------------------------------------------------------------------
# inputs

def _gridworld(rng, shape, world, gamma, p=0.8):
    """A GridWorld as the repository's generators draw them: `small` one +1 and
    one -1 terminal, `goals` 8 goals U(0.5, 1) and 5 % obstacles, `paper` 22
    terminals of +-100, 800 obstacles in a million and a step reward of -3."""
    n = int(np.prod(shape))
    step, goals, rate = {"small": (-0.04, [1.0, -1.0], 0.0), "goals": (-0.01, rng.uniform(0.5, 1.0, 8), 0.05),
                         "paper": (-3.0, [100.0, -100.0] * 11, 800e-6), "batch": (-0.04, [1.0, -1.0], 0.05)}[world]
    cell = np.zeros(n, dtype=np.uint8)
    reward = np.full(n, step, dtype=np.float64)
    if rate:
        blocked = rng.random(n, dtype=np.float32) < rate
        cell[blocked] = OBSTACLE
        reward[blocked] = 0.0
    at = rng.choice(n, size=min(len(goals), n - 1), replace=False) if n < 1 << 20 else \
        np.unique(rng.integers(0, n, len(goals)))
    cell[at] = TERMINAL
    reward[at] = np.asarray(goals)[:len(at)]
    return SimpleNamespace(shape=tuple(shape), p=p, gamma=gamma, cell=cell.reshape(shape),
                           reward=reward.reshape(shape), nstates=n)


def _one(case, seed):
    return _gridworld(np.random.default_rng([seed, 1]), _dims(case), case["world"], case["gamma"])


def _many(case, seed):
    rng = np.random.default_rng([seed, 2])
    if case["kind"] == "batch":
        sizes = np.random.default_rng([case["mix"], 3])    # the batch's make-up belongs to the case
        out = []
        for _ in range(case["count"]):
            shape = sizes.integers(8, 129, 2) if sizes.random() < 0.5 else sizes.integers(8, 49, 3)
            p, gamma = sizes.uniform(0.6, 0.95), sizes.uniform(0.9, 0.995)
            out.append(_gridworld(rng, tuple(int(n) for n in shape), "batch", gamma, p))
        return out
    return [_gridworld(rng, _dims(case), "goals", g) for g in rng.uniform(0.9, 0.995, case["count"])]


def _dense(case, seed):
    """Dense CP model: U(0, 1) entries normalised by row, equal rank weights, N(0, 1) rewards."""
    rng = np.random.default_rng([seed, 4])
    shape, A, R = _dims(case), case["actions"], case["rank"]
    parts = []
    for _ in range(A * R):
        for n in shape:
            m = rng.random((n, n))
            parts.append((m / m.sum(axis=1, keepdims=True)).ravel())
    reward = rng.standard_normal(int(np.prod(shape)))
    packed = np.concatenate(parts)
    return SimpleNamespace(shape=shape, nactions=A, rank=R, lam=np.full((A, R), 1.0 / R), reward=reward,
                           gamma=case.get("gamma", 0.95), packed=packed, packed_factors=lambda: packed)


def _values(n, seed, dtype):
    g = torch.Generator(device="cuda").manual_seed(seed * 7919 + 5)
    return (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 6.0 - 3.0).to(dtype)


def _net(seed):
    """The shipped network, its weights moved a little as training moves them."""
    d = np.load(WEIGHTS)
    rng = np.random.default_rng([seed, 6])
    w, b = d["w"], d["b"]
    w = w + (w != 0) * rng.standard_normal(w.shape).astype(np.float32) * np.float32(1e-3)
    return w.astype(np.float32), b.astype(np.float32), tuple(int(x) for x in d["dilations"]), int(d["n_feat"])


STEP, LR, V2 = 200, 1e-4, 1e-3             # a step in the middle of training: Adam's second moment is V2 squared


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(case=case, kind=kind)
    if kind in ("vi", "pi", "backup"):
        gw = _one(case, seed)
        s.dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
        s.prec = PREC[case["dtype"]]
        s.factors = cp.build_factors(gw, device=0)
        s.policy = torch.zeros(gw.nstates, dtype=torch.uint8, device="cuda")
        s.V = torch.zeros(gw.nstates, dtype=s.dtype, device="cuda")
        s.opts = cp.default_opts(tol=TOL)
        if kind == "backup":
            s.V = _values(gw.nstates, seed, s.dtype)
            s.out = torch.empty_like(s.V)
            s.residual = torch.zeros(1, dtype=torch.float64, device="cuda")
    elif kind == "batch":
        s.batch = cp.batch_build(_many(case, seed), device=0)
        s.V = torch.zeros(int(s.batch.total_states), dtype=torch.float32, device="cuda")
        s.policy = torch.zeros(int(s.batch.total_states), dtype=torch.uint8, device="cuda")
        s.opts = cp.default_opts(tol=TOL, max_iter=5000)
    elif kind in ("dense", "dvi"):
        model = _dense(case, seed)
        n = model.reward.size
        s.dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
        s.prec = PREC[case["dtype"]]
        s.factors = cp.build_factors(model, device=0)
        s.V = torch.zeros(n, dtype=s.dtype, device="cuda") if kind == "dvi" else _values(n, seed, s.dtype)
        s.out = torch.empty_like(s.V)
        s.policy = torch.zeros(n, dtype=torch.uint8, device="cuda")
        s.residual = torch.zeros(1, dtype=torch.float64, device="cuda")
        s.opts = cp.default_opts(tol=TOL)
    else:
        shape = _dims(case)
        w, b, dil, nf = _net(seed)
        s.net = ws.WarmStartNet(device=0, init=(w, b), dilations=dil, n_feat=nf)
        s.batch = cp.batch_build(_many(case, seed), device=0)
        s.V = torch.zeros(int(s.batch.total_states), dtype=torch.float32, device="cuda")
        if kind == "train":
            cp.batch_value_iteration(s.batch, s.V, opts=cp.default_opts(tol=TOL, max_iter=5000))
            s.feat, s.base = ws.coarse_inputs(s.batch, case["count"], shape, s.V.device)
            s.dims = ws.coarse_dims(case["count"], shape)
            s.resid = torch.empty(case["count"] * int(np.prod(shape)), dtype=torch.float32, device="cuda")
            s.loss = torch.zeros(1, dtype=torch.float32, device="cuda")
            s.net.step = STEP
            s.net.vw.fill_(V2 * V2)
            s.net.vb.fill_(V2 * V2)
    return s


def run(s):
    c = s.case
    if s.kind == "vi":
        s.V.zero_()
        r = cp.value_iteration(s.factors, s.prec, s.V, s.policy, opts=s.opts, raise_on_noconv=False)
        return {"V": s.V, "policy": s.policy, "sweeps": r["iterations"]}
    if s.kind == "pi":
        s.V.zero_()
        r = cp.policy_iteration(s.factors, s.prec, s.V, s.policy, opts=s.opts, raise_on_noconv=False)
        return {"V": s.V, "policy": s.policy, "sweeps": r["iterations"]}
    if s.kind == "backup":
        cp.bellman_backup(s.factors, s.prec, s.V, s.out, s.policy, s.residual)
        return {"V": s.out, "policy": s.policy, "residual": s.residual}
    if s.kind == "batch":
        s.V.zero_()
        r, sweeps, _ = cp.batch_value_iteration(s.batch, s.V, opts=s.opts, raise_on_noconv=False)
        cp.batch_certify(s.batch, s.V, s.policy)
        return {"V": s.V, "policy": s.policy, "sweeps": sweeps}
    if s.kind == "dense":
        # the tensor-core sweep as value iteration runs it: values and residual
        pol = None if c["dtype"] == "bf16x3" else s.policy
        cp.bellman_backup(s.factors, s.prec, s.V, s.out, pol, s.residual)
        out = {"V": s.out, "residual": s.residual}
        return out if pol is None else dict(out, policy=pol)
    if s.kind == "dvi":
        s.V.zero_()
        r = cp.value_iteration(s.factors, s.prec, s.V, s.policy, opts=s.opts, raise_on_noconv=False)
        return {"V": s.V, "policy": s.policy, "sweeps": r["iterations"]}
    if s.kind == "start":
        pred, base = ws.warm_start_values(s.net, s.batch, c["count"], _dims(c), s.V)
        return {"V": s.V, "correction": pred, "coarse": base}
    s.loss.zero_()
    s.net.train_step(s.feat, None, None, s.dims, lr=LR, loss_acc=s.loss, fine=(s.batch, s.V, 0, s.base, s.resid))
    n = s.net
    return {"loss": s.loss, "dw": n.dw, "db": n.db, "w": n.w, "b": n.b, "mw": n.mw, "vw": n.vw}


def work(case):
    """Inputs read once and outputs written once; operations of one sweep (solves
    need at least one) or of the layers."""
    kind = case["kind"]
    if kind == "batch":
        n = sum(g.nstates * (10 * len(g.shape)) for g in _many(case, 0))
        states = sum(g.nstates for g in _many(case, 0))
        return {"bytes": states * (4 + 8 + 1 + 4 + 4 + 1), "flops": n}
    shape = _dims(case)
    n, d = int(np.prod(shape)), len(shape)
    if kind in ("vi", "pi", "backup"):
        e = 8 if case["dtype"] == "f64" else 4
        return {"bytes": n * (3 * e + 2), "flops": n * 10 * d}
    if kind in ("dense", "dvi"):
        e = 8 if case["dtype"] == "f64" else 4
        chains = case["actions"] * case["rank"]
        return {"bytes": n * 3 * e + chains * sum(x * x for x in shape) * e, "flops": 2 * chains * n * sum(shape)}
    vox = case["count"] * int(np.prod([(x + 3) // 4 for x in shape]))
    conv = 2 * 27 * CH * CH * vox
    if kind == "start":
        return {"bytes": case["count"] * n * (5 + 4) + 3 * 27 * CH * CH * 2, "flops": 3 * conv}
    # forward of three layers, data gradient of two, weight gradient of three
    return {"bytes": case["count"] * n * 5 + vox * CH * 2 + 3 * 27 * CH * CH * 4 * 7, "flops": 8 * conv}


# --------------------------------------------------------------------------
# the same results in 64 bits, plain torch

def _stencil(cell, shape, dev):
    """Per direction, where the move is possible: [(dim, sign, mask)], obstacles, terminals.
    ``cell`` may have leading instance dimensions."""
    lead = cell.dim() - len(shape)
    obst = cell == OBSTACLE
    moves = []
    for d in range(len(shape)):
        for sg in (-1, 1):
            ax = lead + d
            ok = torch.zeros_like(obst)
            n = shape[d]
            if n > 1:
                here, there = (ok.narrow(ax, 1, n - 1), obst.narrow(ax, 0, n - 1)) if sg < 0 else \
                    (ok.narrow(ax, 0, n - 1), obst.narrow(ax, 1, n - 1))
                here.copy_(~there)
            moves.append((ax, sg, ok))
    return moves, obst, cell == TERMINAL


def _sweep(V, R, moves, obst, term, p, gamma):
    """One Bellman backup: the values and the largest expectation's action."""
    D = len(moves) // 2
    nb = [torch.where(ok, torch.roll(V, -sg, ax), V) for ax, sg, ok in moves]
    pair = [nb[2 * d] + nb[2 * d + 1] for d in range(D)]
    total = pair[0].clone()
    for x in pair[1:]:
        total += x
    slip = (1.0 - p) / (2 * (D - 1)) if D > 1 else None
    best = None
    for j in range(2 * D):
        e = p * nb[j] + (slip * (total - pair[j // 2]) if D > 1 else (1.0 - p) * V)
        best = e if best is None else torch.maximum(best, e)
    out = R + gamma * best
    out = torch.where(term, R, out)
    return torch.where(obst, torch.zeros_like(out), out)


def _grid_tensors(gw):
    cell = torch.as_tensor(np.asarray(gw.cell)).cuda()
    return cell, torch.as_tensor(np.asarray(gw.reward)).cuda()


def _solve(gw, tol, max_iter):
    cell, R = _grid_tensors(gw)
    moves, obst, term = _stencil(cell, gw.shape, cell.device)
    V = torch.zeros_like(R)
    for _ in range(max_iter):
        W = _sweep(V, R, moves, obst, term, gw.p, gw.gamma)
        done = bool(((W - V).abs().max() < tol).item())
        V = W
        if done:
            break
    return V


def _solve_many(cell, R, shape, p, gamma, tol, max_iter, v0=None):
    """Value iteration of instances of one shape stacked along dimension 0, each to its own stop."""
    moves, obst, term = _stencil(cell, shape, cell.device)
    g = gamma.view(-1, *([1] * len(shape)))
    V = torch.zeros_like(R) if v0 is None else v0
    live = torch.ones(R.shape[0], dtype=torch.bool, device=R.device)
    for k in range(max_iter):
        W = _sweep(V, R, moves, obst, term, p, g)
        far = (W - V).abs().flatten(1).amax(1)
        V = torch.where(live.view(-1, *([1] * len(shape))), W, V)
        live = live & ~(far < tol)
        if k % 8 == 7 and not bool(live.any().item()):
            break
    return V


def _coarse(case, seed):
    """Cell features and coarse values of the instances (the warm start's inputs), in 64 bits."""
    shape = _dims(case)
    inst = _many(case, seed)
    cell = torch.as_tensor(np.stack([np.asarray(g.cell) for g in inst])).cuda()
    R = torch.as_tensor(np.stack([np.asarray(g.reward) for g in inst])).cuda()
    gamma = torch.tensor([g.gamma for g in inst], dtype=torch.float64, device="cuda")
    cd = [(n + 3) // 4 for n in shape]

    def cells(x, fill):
        pad = []
        for n, c in zip(reversed(shape), reversed(cd)):
            pad += [0, 4 * c - n]
        x = torch.nn.functional.pad(x, pad, value=fill)
        return x.view(-1, cd[0], 4, cd[1], 4, cd[2], 4).permute(0, 1, 3, 5, 2, 4, 6).reshape(-1, *cd, 64)

    c = cells(cell.to(torch.int32), -1)
    r = cells(R, 0.0)
    inside = c >= 0
    n = inside.sum(-1).double()
    nob = (c == OBSTACLE).sum(-1).double()
    free = c == FREE
    live = free | (c == TERMINAL)
    anyt = (c == TERMINAL).any(-1)
    tmax = torch.where(anyt, torch.where(c == TERMINAL, r, torch.full_like(r, -math.inf)).amax(-1),
                       torch.zeros_like(n))
    mean = torch.where(live.any(-1), (r * live).sum(-1) / live.sum(-1).clamp(min=1), torch.zeros_like(n))
    gg = gamma.view(-1, 1, 1, 1)
    steps = 1 + gg + gg * gg + gg ** 3
    nfree = free.sum(-1)
    rc = torch.where(nfree > 0, (r * free).sum(-1) / nfree.clamp(min=1) * steps, torch.zeros_like(n))
    kind = torch.where(2 * nob >= n, OBSTACLE, torch.where(anyt, TERMINAL, FREE))
    rc = torch.where(kind == TERMINAL, tmax, rc)
    rc = torch.where(kind == OBSTACLE, torch.zeros_like(rc), rc)
    v0 = torch.where(kind == TERMINAL, rc, torch.zeros_like(rc))
    cv = _solve_many(kind, rc, cd, 0.8, gamma ** 4, ws.COARSE_TOL, 4000, v0=v0)
    feat = torch.stack([mean, nob / n, tmax, (-torch.log(1 - gamma) / 5).view(-1, 1, 1, 1).expand_as(mean), cv], 1)
    return inst, cell, R, gamma, feat.to(torch.bfloat16).double(), cv


def _network(feat, w, b, dil, wgrad=False):
    """The three convolutions in 64 bits: channel 0 of the last one."""
    x = feat
    ws_, bs_ = [], []
    for layer in range(w.shape[0]):
        k = w[layer].double().view(3, 3, 3, CH, CH).permute(3, 4, 0, 1, 2).contiguous()
        bias = b[layer].double().contiguous()
        if wgrad:
            k.requires_grad_(True)
            bias.requires_grad_(True)
        ws_.append(k)
        bs_.append(bias)
        kk, d = (k[:, :x.shape[1]] if layer == 0 else k), dil[layer]
        # a sum of 27 shifted matrix products ("same" zero padding)
        pad = torch.nn.functional.pad(x, (d,) * 6)
        y = bias.view(1, -1, 1, 1, 1)
        sz = x.shape[2:]
        for t in range(27):
            o = [d * (t // 9), d * (t // 3 % 3), d * (t % 3)]
            part = pad[:, :, o[0]:o[0] + sz[0], o[1]:o[1] + sz[1], o[2]:o[2] + sz[2]]
            y = y + torch.einsum("oc,nczyx->nozyx", kk[:, :, t // 9, t // 3 % 3, t % 3], part)
        x = torch.relu(y) if layer < w.shape[0] - 1 else y
    return x[:, 0], ws_, bs_


def _upsample(c, shape):
    """Trilinear interpolation of cell values at the states, clamped to the outermost cell centres."""
    for d, n in enumerate(shape):
        nc = c.shape[1 + d]
        u = ((torch.arange(n, dtype=torch.float64, device=c.device) + 0.5) / 4 - 0.5).clamp(0, nc - 1)
        lo = u.floor().long()
        hi = (lo + 1).clamp(max=nc - 1)
        t = (u - lo).view(*([1] * (1 + d)), -1, *([1] * (2 - d)))
        c = c.index_select(1 + d, lo) * (1 - t) + c.index_select(1 + d, hi) * t
    return c


def _packed(x):
    """Instances back to back, each on a multiple of four values."""
    flat = x.flatten(1)
    pad = (-flat.shape[1]) % 4
    return torch.nn.functional.pad(flat, (0, pad)).flatten()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("vi", "pi"):
        V = _solve(_one(case, seed), TOL if kind == "vi" else 1e-11, 1000 if kind == "vi" else 20000)
        return {"V": V.flatten(), "policy": None, "sweeps": None}
    if kind == "backup":
        gw = _one(case, seed)
        cell, R = _grid_tensors(gw)
        V = _values(gw.nstates, seed, torch.float64 if case["dtype"] == "f64" else torch.float32).double()
        moves, obst, term = _stencil(cell, gw.shape, cell.device)
        W = _sweep(V.view(gw.shape), R, moves, obst, term, gw.p, gw.gamma).flatten()
        far = torch.where(obst.flatten(), torch.zeros_like(W), (W - V).abs()).max()
        return {"V": W, "policy": None, "residual": far.reshape(1)}
    if kind == "batch":
        if case["count"] > 48:             # one instance after the other takes too long
            return None
        out = []
        for g in _many(case, seed):
            V = _solve(g, TOL, 5000).flatten()
            out.append(torch.nn.functional.pad(V, (0, (-V.numel()) % 4)))
        return {"V": torch.cat(out), "policy": None, "sweeps": None}
    if kind in ("dense", "dvi"):
        m = _dense(case, seed)
        R = torch.as_tensor(m.reward).cuda()
        U, off = [], 0
        packed = torch.as_tensor(m.packed).cuda()
        for _ in range(m.nactions * m.rank):
            row = []
            for n in m.shape:
                row.append(packed[off:off + n * n].view(n, n))
                off += n * n
            U.append(row)

        def backup(V):
            best = None
            for a in range(m.nactions):
                e = 0
                for r in range(m.rank):
                    x = V.view(m.shape)
                    for d, u in enumerate(U[a * m.rank + r]):
                        x = torch.tensordot(u, x, dims=([1], [d])).movedim(0, d)
                    e = e + float(m.lam[a, r]) * x.reshape(-1)
                q = R + m.gamma * e
                best = q if best is None else torch.maximum(best, q)
            return best

        if kind == "dense":
            V = _values(R.numel(), seed, torch.float64 if case["dtype"] == "f64" else torch.float32).double()
            W = backup(V)
            res = (W - V).abs().max().reshape(1)
            out = {"V": W, "residual": res}
            return out if case["dtype"] == "bf16x3" else dict(out, policy=None)
        V = torch.zeros_like(R)
        for _ in range(1000):
            W = backup(V)
            done = bool(((W - V).abs().max() < TOL).item())
            V = W
            if done:
                break
        return {"V": V, "policy": None, "sweeps": None}
    shape = _dims(case)
    w, b, dil, _ = _net(seed)
    w, b = torch.as_tensor(w).cuda(), torch.as_tensor(b).cuda()
    inst, cell, R, gamma, feat, cv = _coarse(case, seed)
    obst, term = cell == OBSTACLE, cell == TERMINAL
    if kind == "start":
        pred, _, _ = _network(feat, w, b, dil)
        V = _upsample(pred + cv, shape)
        V = torch.where(term, R, V)
        V = torch.where(obst, torch.zeros_like(V), V)
        return {"V": _packed(V), "correction": pred.flatten(), "coarse": cv.flatten()}
    Vt = _solve_many(cell, R, shape, 0.8, gamma, TOL, 5000)
    pred, wl, bl = _network(feat, w, b, dil, wgrad=True)
    off = torch.where(obst | term, torch.zeros_like(Vt), _upsample(pred + cv, shape) - Vt)
    loss = off.square().sum() / off.numel()
    loss.backward()
    dw = torch.stack([k.grad.permute(2, 3, 4, 0, 1).reshape(27, CH, CH) for k in wl])
    db = torch.stack([x.grad for x in bl])
    moved = []
    for p, g in ((w.double(), dw), (b.double(), db)):
        mm, vv = 0.1 * g, 0.999 * V2 * V2 + 0.001 * g * g
        k = STEP + 1
        moved.append((p - LR * (mm / (1 - 0.9 ** k)) / ((vv / (1 - 0.999 ** k)).sqrt() + 1e-8), mm, vv))
    return {"loss": loss.detach().reshape(1), "dw": dw, "db": db, "w": moved[0][0], "b": moved[1][0],
            "mw": moved[0][1], "vw": moved[0][2]}
