"""The measured cases: what a program that uses this library has it do, through its public entry points.

A case names a ``kind`` (which calls are made) and its sizes.  ``listed()`` gives the standing
cases, ``draw(rng)`` more of the same ranges, ``prepare(case, seed)`` a program's inputs, handles and
output buffers, ``run(state)`` one pass, ``work(case)`` the least bytes and operations of a pass and
``exact(case, seed)`` the surrogate's outputs in 64 bits.

Kinds
  rollout     a staged batch: win counts and step totals, then probabilities and odds
  live        the same from host arrays each time: stage, roll out, probabilities, release
  places      finishing places to the K-th finisher and the probability of the first K
  orders      dense tallies of the ordered first K, with the places of the same pass
  histogram   the finishing orders of every race as (key, count) pairs in key order
  population  an actual race, and at every step of it all its bettors' dry-runs, odds and predictions
  infer       the surrogate's probabilities for a staged batch of queries
  mixed       the same with a share of queries outside the training ranges, answered by Monte Carlo
  grad        loss and gradient of the surrogate on one batch of states
  train       optimiser steps of the surrogate, then its parameters
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2108_02419_gb300 import bbe
from paper_2108_02419_gb300 import workloads as W

OPS_PER_STEP = 62  # the method's operations per competitor and step (generator, Eq. 1, advance, finish)


# ------------------------------------------------------------------ cases

def listed():
    return [
        # the paper's example race asked for its odds once more: the smallest call, all latency
        dict(name="single_start", kind="rollout", shape="start", races=1, n=5, length=2000.0, rollouts=1000),
        # a live exchange re-evaluates one snapshot: 1000 bettors with 50 dry-runs each, from host buffers
        dict(name="live_snapshot", kind="live", shape="bunched", races=1000, n=5, length=2000.0, rollouts=50),
        # the benchmark's uniform batch: large equal races
        dict(name="uniform_4096x20", kind="rollout", shape="spread", races=4096, n=20, length=5000.0, rollouts=10000),
        # the benchmark's uneven batch: 2..24 competitors, 10^3..10^5 rollouts, all remaining distances
        dict(name="uneven_10000", kind="rollout", shape="uneven", races=10000, n=24, length=5000.0, rollouts=0),
        # mid-race snapshots of races as they are run (everyone started together) under the time law
        dict(name="time_law_700x13", kind="rollout", shape="bunched", races=700, n=13, length=3000.0, rollouts=3000,
             law="time"),
        # place and each-way markets
        dict(name="places3_512x20", kind="places", shape="spread", races=512, n=20, length=5000.0, rollouts=10000, k=3),
        # the distribution of whole finishing orders
        dict(name="histogram_96x20", kind="histogram", shape="spread", races=96, n=20, length=5000.0, rollouts=10000,
             k=20),
        # Section 6: one race with 1000 bettors of 50 dry-runs at each of its steps
        dict(name="population_5x1000", kind="population", shape="start", races=1, n=5, length=2000.0, rollouts=50,
             bettors=1000),
        # many queries of the trained network, none outside its ranges
        dict(name="infer_200k", kind="infer", shape="uneven", races=200000, n=24, length=5000.0, rollouts=1000),
        # queries of which three in a hundred have more competitors than the network was trained on
        dict(name="mixed_20k", kind="mixed", shape="uneven", races=20000, n=24, length=5000.0, rollouts=20000,
             outside=0.03),
        # the gradient of one training batch
        dict(name="grad_4096", kind="grad", shape="uneven", races=4096, n=24, length=5000.0, rollouts=1000),
        # one call of the training loop: 16 steps of 4096 states
        dict(name="train_16x4096", kind="train", shape="uneven", races=65536, n=24, length=5000.0, rollouts=1000,
             batch=4096, steps=16),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["rollout"] * 6 + ["live"] * 2 + ["places"] * 2 + ["orders", "histogram", "population", "infer",
                                                                       "infer", "mixed", "grad", "train"])
    c = dict(kind=kind)
    if kind in ("infer", "mixed", "grad", "train"):
        c.update(shape="uneven", n=24, length=5000.0, rollouts=1000)
        if kind == "infer":
            c["races"] = int(_log(rng, 1, 250000))
        elif kind == "mixed":
            c.update(races=int(_log(rng, 200, 25000)), outside=round(rng.uniform(0.005, 0.05), 4),
                     rollouts=int(_log(rng, 3000, 30000)))
        elif kind == "grad":
            c["races"] = int(_log(rng, 50, 9000))
        else:
            c.update(races=int(_log(rng, 5000, 80000)), batch=int(_log(rng, 700, 5000)), steps=rng.randint(2, 20))
        return c
    if kind == "population":
        c.update(shape="start", races=1, n=rng.randint(2, 14), length=float(rng.randint(600, 2200)),
                 rollouts=rng.randint(20, 100), bettors=int(_log(rng, 20, 600)))
        return c
    c["shape"] = rng.choice(["spread", "spread", "bunched", "bunched", "start"] +
                            (["uneven", "uneven"] if kind != "histogram" else []))
    c["n"] = rng.randint(2, 20 if kind == "histogram" else 32)
    c["length"] = round(rng.uniform(800.0, 6000.0), 1)
    budget = {"rollout": 3e10, "live": 3e8, "places": 4e9, "orders": 4e9, "histogram": 3e9}[kind]
    c["rollouts"] = int(_log(rng, 40, 20000 if kind != "live" else 1000))
    per_rollout = c["n"] * (40 if c["shape"] in ("spread", "uneven") else c["length"] / 16.0)
    if kind in ("places", "orders", "histogram"):
        per_rollout = c["n"] * c["length"] / 16.0
    most = max(1.0, budget / (per_rollout * c["rollouts"]))
    c["races"] = max(1, int(_log(rng, 1, min(most, 9000.0))))
    if kind in ("places", "orders"):
        c["k"] = rng.randint(1, min(3 if kind == "orders" else 6, c["n"]))
    if kind == "histogram":
        c["k"] = rng.randint(1, c["n"])
    if rng.random() < 0.25:
        c["law"] = "time"
    if rng.random() < 0.2:
        c["dist"] = rng.choice(["uniform", "two_point"])
    if rng.random() < 0.3:
        c["theta"] = round(rng.uniform(0.2, 4.0), 2)
    if rng.random() < 0.25:
        c["preference"] = True  # preference coefficients below 1
    if rng.random() < 0.25:
        c["previous"] = True    # previous steps given, as a live snapshot has them
    return c


# ------------------------------------------------------------------ inputs

def _races(case, seed, outside=0):
    """The batch of a case: host arrays, from the seed alone.  outside: that many races of 26..30 at the end."""
    rng = np.random.default_rng([seed, 7])
    m, n, L, shape = case["races"], case["n"], case["length"], case["shape"]
    if shape == "uneven":
        # the competitor counts belong to the case, everything else to the seed
        by_case = np.random.default_rng([m, n, 3])
        sizes = np.concatenate([by_case.integers(2, n + 1, m - outside), by_case.integers(26, 31, outside)])
        nt = int(sizes.sum())
        R = case["rollouts"] or np.floor(10.0 ** rng.uniform(3.0, 5.0, m))
        rb = W.from_arrays(sizes, L, R, L - rng.uniform(100.0, L, nt), rng.uniform(15.0, 17.0, nt),
                           rng.uniform(0.5, 1.5, nt), rng.uniform(0.0, 1.0, nt))
    elif shape == "spread":
        rb = W.uniform_batch(seed=seed, n_races=m, n=n, L=L, rollouts=case["rollouts"])
    else:
        rb = W.uniform_batch(seed=seed, n_races=m, n=n, L=L, rollouts=case["rollouts"])
        # everyone at the start line, or t steps of their own pace after it
        t = 0.0 if shape == "start" else np.random.default_rng([m, n, 5]).uniform(0.1, 0.8) * L / 17.0
        d = t * rb.mu + math.sqrt(t) * rb.sigma * rng.standard_normal(rb.n_total)
        rb.d0 = np.clip(d, 0.0, 0.9 * L).astype(np.float32)
    rb.seed = seed
    rb.dist = {"uniform": W.DIST_UNIFORM, "two_point": W.DIST_TWO_POINT}.get(case.get("dist"), W.DIST_NORMAL)
    if "theta" in case:
        rb.theta = np.full(rb.n_total, case["theta"], np.float32)
    if case.get("preference"):
        rb.P = rng.uniform(0.85, 1.0, rb.n_total).astype(np.float32)
    if case.get("previous"):
        rb.prev0 = (rb.mu * rng.uniform(0.8, 1.2, rb.n_total)).astype(np.float32)
    if case.get("law") == "time":
        done = (rb.d0.reshape(-1)[rb.race_off[:-1]] / 16.0).astype(np.float32)
        rb.elapsed = np.floor(done)
        rb.horizon = np.full(rb.n_races, L / 16.0, np.float32)
    return rb


def _params(seed):
    """A network's float32 parameters: He-scaled layers, a head that separates the competitors."""
    rng = np.random.default_rng([seed, 11])
    u = lambda rows, cols, fan, gain: rng.uniform(-1.0, 1.0, (rows, cols)) * math.sqrt(gain / fan)
    w1 = u(128, 16, 14, 6.0)
    w1[:, 14:] = 0.0
    parts = [w1, u(1, 128, 128, 0.02), u(128, 128, 128, 6.0), u(1, 128, 128, 0.02), u(128, 128, 128, 6.0),
             u(1, 128, 128, 0.02), u(128, 256, 256, 6.0), u(1, 128, 128, 0.02), u(1, 128, 128, 12.0), np.zeros((1, 1))]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


def _targets(rb):
    """Win probabilities to train on: a softmax of how soon each competitor is expected home."""
    r = np.repeat(np.arange(rb.n_races), rb.sizes())
    t = -((rb.L[r] - rb.d0) / rb.mu).astype(np.float64)
    first = np.maximum.reduceat(t, rb.race_off[:-1])
    e = np.exp(t - first[r])
    return (e / np.add.reduceat(e, rb.race_off[:-1])[r]).astype(np.float32)


class _Network:
    """A surrogate whose parameters come from the seed and whose ranges cover the queries of `like`."""

    def __init__(self, case, seed, ranges):
        self.h = bbe.bbe_surrogate_create(seed)
        if ranges:
            lo = dict(case, races=2048, rollouts=1000)
            rb = _races(lo, seed + 5)
            # the extreme values that a training set of millions of states reaches
            e = W.from_arrays([2, 24], case["length"], 1000, np.tile([0.0, case["length"] - 100.0], 13),
                              np.tile([15.0, 17.0], 13), np.tile([0.5, 1.5], 13), np.tile([0.0, 1.0], 13))
            with bbe.Batch(W.concat([rb, e])) as b:
                t = torch.from_numpy(_targets(b.rb)).cuda()
                bbe.bbe_surrogate_train(self.h, b.handle, t, batch_states=b.rb.n_races, steps=1)
                bbe.bbe_surrogate_status(self.h)
        bbe.bbe_surrogate_set_params(self.h, _params(seed))

    def __del__(self):
        bbe.bbe_surrogate_destroy(self.h)


class _State:
    pass


def _empty(n, dtype):
    return torch.empty(n, dtype=dtype, device="cuda")


def prepare(case, seed):
    s = _State()
    s.kind, s.case = case["kind"], case
    outside = max(1, int(case["outside"] * case["races"])) if s.kind == "mixed" else 0
    rb = s.rb = _races(case, seed, outside)
    if s.kind == "live":
        s.counts, s.probs, s.odds = _empty(rb.n_total, torch.int32), _empty(rb.n_total, torch.float32), _empty(rb.n_total, torch.float32)
        return s
    s.batch = bbe.Batch(rb)
    if s.kind == "rollout":
        s.counts, s.steps = s.batch.new_outputs()
        s.probs, s.odds = _empty(rb.n_total, torch.float32), _empty(rb.n_total, torch.float32)
    elif s.kind == "places":
        s.counts, s.steps = _empty((rb.n_total, case["k"]), torch.int32), _empty(rb.n_races, torch.int64)
        s.probs = _empty(rb.n_total, torch.float32)
    elif s.kind == "population":
        s.cap = 1024
        s.pos = torch.zeros(rb.n_total * s.cap, dtype=torch.float32, device="cuda")
        s.stp = torch.zeros_like(s.pos)
        s.n_steps = _empty(1, torch.int32)
        s.snaps = int(case["length"] / 12.0) + 8  # room for more snapshots than such a race has steps
        m = s.snaps * case["bettors"]
        zeros = lambda k, dtype: torch.zeros(k, dtype=dtype, device="cuda")
        s.counts, s.steps = zeros(m * rb.n_total, torch.int32), zeros(m, torch.int64)
        s.probs, s.odds = zeros(m * rb.n_total, torch.float32), zeros(m * rb.n_total, torch.float32)
        s.pred = zeros(s.snaps * 4, torch.int32)
    elif s.kind in ("infer", "mixed"):
        s.net = _Network(case, seed, ranges=True)
        s.probs, s.used = _empty(rb.n_total, torch.float32), _empty(rb.n_races, torch.uint8)
        if s.kind == "mixed":
            bbe.bbe_surrogate_set_fallback(s.net.h, 2000, 0.01 / 4.5)
    elif s.kind in ("grad", "train"):
        s.net = _Network(case, seed, ranges=False)
        s.target = torch.from_numpy(_targets(rb)).cuda()
        s.grad, s.loss = _empty(bbe.bbe_surrogate_num_params(), torch.float32), _empty(case.get("steps", 1), torch.float32)
    return s


# ------------------------------------------------------------------ one pass

def run(s):
    c = s.case
    if s.kind == "rollout":
        s.batch.rollout(s.counts, s.steps)
        s.batch.win_probs(s.counts, s.probs, s.odds)
        return s.counts, s.steps, s.probs, s.odds
    if s.kind == "live":
        with bbe.Batch(s.rb) as b:
            b.rollout(s.counts)
            b.win_probs(s.counts, s.probs, s.odds)
        return s.counts, s.probs, s.odds
    if s.kind == "places":
        s.batch.places(c["k"], s.counts, s.steps)
        s.batch.place_probs(s.counts, c["k"], s.probs)
        return s.counts, s.steps, s.probs
    if s.kind == "orders":
        return s.batch.orders(c["k"], with_places=True)
    if s.kind == "histogram":
        keys, counts, off, places, steps = s.batch.order_histogram(c["k"], with_places=True)
        # equal races have tables of equal size: each race's orders by key (unused entries hold -1)
        m = s.rb.n_races
        keys, counts = keys.view(torch.int64).view(m, -1), counts.view(m, -1)
        keys, at = torch.sort(keys, dim=1)
        return keys, counts.gather(1, at), places, steps
    if s.kind == "population":
        h0 = s.batch.handle
        bbe.bbe_race_trajectory(h0, 1 << 30, s.cap, s.pos, s.stp, s.n_steps)
        h, snaps = bbe.bbe_snapshot_batch(h0, 0, s.pos, s.stp, s.n_steps, s.cap, 1, c["bettors"], c["rollouts"], 1 << 20)
        try:
            if snaps > s.snaps:
                raise RuntimeError("more snapshots than room")
            bbe.bbe_rollout_batch(h, s.counts, s.steps)
            bbe.bbe_win_probs(h, s.counts, s.probs, s.odds)
            bbe.bbe_bettor_predictions(h0, 0, s.pos, s.stp, s.n_steps, s.cap, 1, snaps, 10, 3.0, 77, s.pred)
        finally:
            bbe.bbe_destroy_batch(h)
        return s.pos, s.stp, s.n_steps, s.counts, s.steps, s.probs, s.odds, s.pred
    if s.kind in ("infer", "mixed"):
        bbe.bbe_surrogate_infer(s.net.h, s.batch.handle, s.probs, s.used if s.kind == "mixed" else None)
        return [s.probs, s.used] if s.kind == "mixed" else [s.probs]
    if s.kind == "grad":
        bbe.bbe_surrogate_grad(s.net.h, s.batch.handle, s.target, s.grad, s.loss)
        return s.grad, s.loss
    if s.kind == "train":
        bbe.bbe_surrogate_train(s.net.h, s.batch.handle, s.target, lr=1e-3, batch_states=c["batch"], steps=c["steps"],
                                shuffle_seed=3, loss_log=s.loss)
        return bbe.bbe_surrogate_get_params(s.net.h), s.loss
    raise ValueError(s.kind)


# ------------------------------------------------------------------ least work

def _mean_size(case):
    return (2 + case["n"]) / 2 if case["shape"] == "uneven" else case["n"]


def _steps_per_rollout(case, k=1):
    """Expected steps to the k-th finisher at 16 units a step."""
    n, L = _mean_size(case), case["length"]
    if case["shape"] == "spread":
        return (0.1 * L + 0.9 * L * k / (n + 1)) / 16.0
    if case["shape"] == "uneven":
        return (100.0 + (L - 100.0) * k / (n + 1)) / 16.0
    return L / 16.0 * (1.0 if case["shape"] == "start" else 0.55)


def work(case):
    """The inputs once, the outputs once, and the method's arithmetic."""
    kind, m, n = case["kind"], case["races"], _mean_size(case)
    rows = m * n
    net = 2.0 * (16 * 128 + 2 * 128 * 128 + 256 * 128 + 128)  # one forward evaluation per competitor
    if kind == "infer":
        return {"bytes": rows * (20 + 4) + m * 8, "flops": rows * net}
    if kind in ("grad", "train"):
        if kind == "train":
            rows = case["batch"] * case["steps"] * n
        return {"bytes": rows * 24 + 68225 * 8, "flops": 3 * rows * net}
    R = case["rollouts"] or (1e5 - 1e3) / math.log(100.0)  # mean of the log-uniform budgets
    if kind == "mixed":
        sims = m * case["outside"] * 28 * R * 0.5 * (100 + 4900 / 29) / 16.0
        return {"bytes": rows * 24 + m * 9, "flops": rows * net + sims * OPS_PER_STEP}
    if kind == "population":
        steps = case["length"] / 16.0
        sims = steps * case["bettors"] * n * R * steps / 2
        return {"bytes": steps * case["bettors"] * n * 12.0, "flops": sims * OPS_PER_STEP}
    k = case.get("k", 1)
    out = {"rollout": 12, "live": 12}.get(kind, 4 * k + 4)
    if kind == "orders":
        out += 4 * n ** (k - 1)
    if kind == "histogram":
        out += 12 * min(R, math.perm(int(n), k)) / n  # the distinct orders at most
    return {"bytes": rows * (28 + out) + m * 20, "flops": rows * R * _steps_per_rollout(case, k) * OPS_PER_STEP}


# ------------------------------------------------------------------ the surrogate in 64 bits

def _features64(rb, a, b):
    """Races a..b-1 as [races, 32, 16] features and a mask of their competitors (float64, on the GPU)."""
    rows = slice(int(rb.race_off[a]), int(rb.race_off[b]))
    sizes = torch.from_numpy(rb.sizes()[a:b]).cuda()
    m, N = b - a, int(sizes.max())
    mask = torch.arange(N, device="cuda")[None, :] < sizes[:, None]

    def pad(x):
        out = torch.zeros((m, N), dtype=torch.float64, device="cuda")
        out[mask] = torch.from_numpy(np.ascontiguousarray(x[rows])).cuda().double()
        return out

    d, mu, sigma, rho = pad(rb.d0), pad(rb.mu), pad(rb.sigma), pad(rb.rho)
    mu = torch.where(mask, mu, torch.ones_like(mu))
    L = torch.from_numpy(rb.L[a:b]).cuda().double()[:, None]
    inf = math.inf
    frac = d / L
    v = mu * (1 + 0.1 * (2 * rho - 1) * frac)
    T = (L - d) / v
    sd = sigma * T.sqrt() / v
    best = torch.where(mask, T, torch.full_like(T, inf)).argmin(1, keepdim=True)
    lag = T - T.gather(1, best)
    other = d[:, None, :] - d[:, :, None]  # [race, competitor, other]
    seen = mask[:, None, :]
    ahead = torch.where(seen & (other > 0), other, torch.full_like(other, inf))
    behind = torch.where(seen & (other < 0), -other, torch.full_like(other, inf))
    (ga, ia), (gb, ib) = ahead.min(2), behind.min(2)
    none_a, none_b = ga == inf, gb == inf
    ga, gb = ga.clamp(max=1e6), gb.clamp(max=1e6)
    va, vb, Tb = v.gather(1, ia), v.gather(1, ib), T.gather(1, ib)
    one = torch.ones_like(v)
    da = torch.where(v > va, v - va, one)
    db = torch.where(vb > v, vb - v, one)
    f = [frac, (L - d) / 5000.0, mu - 16, sigma - 1, 2 * rho - 1, T / 100, lag.clamp(max=100) / 10, sd,
         (lag / (sd ** 2 + sd.gather(1, best) ** 2 + 0.01).sqrt()).clamp(max=20) / 5, ga.clamp(max=100) / 10,
         (1.0 / sizes.double())[:, None].expand(m, N), gb.clamp(max=100) / 10,
         torch.where(~none_a & (v > va), (ga / da / T).clamp(max=2) / 2, one),
         torch.where(~none_b & (vb > v), (gb / db / Tb).clamp(max=2) / 2, one), 0 * v, 0 * v]
    return torch.stack(f, 2) * mask[:, :, None], mask, sizes


def _log_probs64(x, mask, sizes, flat):
    shapes = [(128, 16), (128,), (128, 128), (128,), (128, 128), (128,), (128, 256), (128,), (128,), (1,)]
    p, o = [], 0
    for s in shapes:
        k = math.prod(s)
        p.append(flat[o:o + k].view(s))
        o += k
    h = x
    for w, b in ((p[0], p[1]), (p[2], p[3]), (p[4], p[5])):
        h = torch.relu(h @ w.T + b)
    g = (h * mask[:, :, None]).sum(1, keepdim=True) / sizes.double()[:, None, None]
    u = torch.relu(torch.cat([h, g.expand_as(h)], 2) @ p[6].T + p[7])
    z = (u @ p[8] + p[9]).masked_fill(~mask, -math.inf)
    return torch.log_softmax(z, 1)


def exact(case, seed):
    if case["kind"] not in ("infer", "grad"):
        return None  # counts are whole numbers; a trained network's weights have no value of their own
    rb = _races(case, seed)
    flat = torch.from_numpy(_params(seed)).cuda().double()
    if case["kind"] == "infer":
        out = []
        for a in range(0, rb.n_races, 8192):
            x, mask, sizes = _features64(rb, a, min(a + 8192, rb.n_races))
            out.append(_log_probs64(x, mask, sizes, flat).exp()[mask])
        return [torch.cat(out)]
    x, mask, sizes = _features64(rb, 0, rb.n_races)
    t = torch.zeros(mask.shape, dtype=torch.float64, device="cuda")
    t[mask] = torch.from_numpy(_targets(rb)).cuda().double()
    flat.requires_grad_(True)
    logq = _log_probs64(x, mask, sizes, flat).masked_fill(~mask, 0.0)
    loss = -(t * logq).sum() / rb.n_races
    loss.backward()
    return flat.grad, loss.detach().reshape(1)
