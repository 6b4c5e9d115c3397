"""Runs the contender search on the checked build of the library, which counts what a pass came across (work
items run on contenders alone, rollouts listed to be run again, items with a rest to run with everybody) and
can be told to look for contenders whatever that costs; every result is compared with the oracle's whole
races.  Started by tests/test_gpu_contenders_reached.py with BBE_LIB naming the checked build."""
import ctypes
import os
import sys

import numpy as np
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import oracle  # noqa: E402
from paper_2108_02419_gb300 import bbe  # noqa: E402
from tests import test_gpu_contenders as C  # noqa: E402

assert bbe.LIB_PATH == os.environ["BBE_LIB"], bbe.LIB_PATH
lib = bbe.lib()
lib.bbe_checked_contenders.argtypes = [ctypes.c_void_p, ctypes.c_int32]
lib.bbe_checked_seen.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]


class Batch(bbe.Batch):
    def __init__(self, rb, always=True, **cfg):
        super().__init__(rb)
        if cfg:
            self.set_cfg(**cfg)
        assert lib.bbe_checked_contenders(self.handle, int(always)) == 0

    def seen(self):
        out = np.zeros(3, np.int32)
        assert lib.bbe_checked_seen(self.handle, out.ctypes.data, torch.cuda.current_stream().cuda_stream) == 0
        return out


def stage(name, races, rollouts):
    C.RACES, C.ROLLOUTS = races, rollouts
    return C.CASES[name]()


def same(got, want, what):
    got = got.cpu().numpy()
    assert np.array_equal(got.ravel(), np.ravel(want)), what


def limited(b):
    try:
        b.status()
    except bbe.BbeError as e:
        assert e.status == -5, e
        return True
    return False


# previous steps up to 200 units let anybody reach the line; the same with steps that a race can have
RULED_OUT_NOBODY = ("fast starts",)
C.CASES["previous steps"] = lambda: C._spread(12, 18, prev=(5.0, 30.0), theta=3.0)

# every geometry, law and distribution, to the first, second and fourth place
for name in C.CASES:
    rb = stage(name, 96, {"two": 4000, "five": 2000}.get(name, 1200))  # a normal launch in each
    with Batch(rb) as b:
        counts, steps = b.rollout()
        b.status()
        seen = b.seen()
        want, want_s, _ = oracle.batch_counts(rb)
        same(counts, want, name)
        same(steps, want_s, name)
        print(name, "win", seen)
        assert seen[0] > 0 or name in RULED_OUT_NOBODY, name
        assert name != "stuck behind the leader" or seen[1] > 0
        for places in (2, 4):
            pc, ps = b.places(places)
            b.status()
            seen = b.seen()
            want, want_s, _ = oracle.batch_places(rb, places)
            same(pc, want, (name, places))
            same(ps, want_s, (name, places))
            print(name, places, seen)
            assert seen[0] > 0 or places == 4 or name in RULED_OUT_NOBODY + ("two", "stuck behind the leader"), name

# order tables and histograms of the first places
for name in ("twenty", "full warp", "far blocking", "time law, late"):
    rb = stage(name, 96, 1200)
    with Batch(rb) as b:
        orders, pc, _ = b.orders(2, with_places=True)
        b.status()
        seen_o = b.seen()
        keys, hcounts, off, _, _ = b.order_histogram(2)
        b.status()
        seen_h = b.seen()
        keys, hcounts = keys.cpu().numpy(), hcounts.cpu().numpy()
    print(name, "orders", seen_o, seen_h)
    assert seen_o[0] > 0 and seen_h[0] > 0
    want = oracle.batch_orders(rb, 2)[0]
    same(orders, np.concatenate([np.ravel(t) for t in want]), name)
    want_h = oracle.batch_order_histograms(rb, 2)[0]
    for r in range(rb.n_races):
        n = int(rb.race_off[r + 1] - rb.race_off[r])
        k, c = keys[off[r]:off[r + 1]], hcounts[off[r]:off[r + 1]]
        used = k != np.uint64(2 ** 64 - 1)
        got = {tuple(int(x) for x in bbe.bbe_order_key_decode(n, 2, int(key))): int(v) for key, v in zip(k[used], c[used])}
        assert got == dict(want_h[r]), r

# the step limit below the contenders' horizon, and above it for rollouts that are run again with everybody
for name, limit in (("twenty", 27), ("stuck behind the leader", 27), ("stuck behind the leader", 150)):
    rb = stage(name, 96, 1200)
    want, want_s, _ = oracle.batch_counts(rb, max_steps=limit)
    with Batch(rb, max_steps=limit) as b:
        counts, steps = b.rollout()
        assert limited(b)
        seen = b.seen()
        print(name, "limit", limit, seen)
        assert seen[0] > 0
        same(counts, want, (name, limit))
        same(steps, want_s, (name, limit))

# every layout
for slots in (1, 2, 3, 4):
    rb = stage("twenty", 96, 1200)
    with Batch(rb, slots_per_lane=slots) as b:
        counts, steps = b.rollout()
        b.status()
        seen = b.seen()
        print("slots", slots, seen)
        assert seen[0] > 0
        want, want_s, _ = oracle.batch_counts(rb)
        same(counts, want, slots)
        same(steps, want_s, slots)
        pc, ps = b.places(3)
        b.status()
        want, want_s, _ = oracle.batch_places(rb, 3)
        same(pc, want, slots)
        same(ps, want_s, slots)

# batches that a program stages: the search by its own rule, a sample of races against the oracle; in the last
# one nearly every rollout is listed, so the lists fill and the rest runs with everybody
for name, races, rollouts, sample in (("two", 96, 48000, 2), ("five", 96, 18000, 3), ("twenty", 96, 6000, 4),
                                      ("uniform steps", 96, 6000, 3), ("time law, late", 96, 6500, 3),
                                      ("stuck behind the leader", 40, 40000, 1)):
    rb = stage(name, races, rollouts)
    head = rb.slice(0, sample)
    with Batch(rb, always=False) as b:
        counts, steps = b.rollout()
        b.status()
        seen = b.seen()
        print(name, "by the rule", seen)
        assert seen[0] > 0, name
        want, want_s, _ = oracle.batch_counts(head)
        same(counts[:head.n_total], want, name)
        same(steps[:sample], want_s, name)
        if name.startswith("stuck"):
            assert seen[1] > 64 and seen[2] > 0
        if name in ("twenty", "time law, late"):
            pc, ps = b.places(2)
            b.status()
            assert b.seen()[0] > 0
            want, want_s, _ = oracle.batch_places(head, 2)
            same(pc[:head.n_total], want, name)
            same(ps[:sample], want_s, name)

# the no-allocation entry point, by its rule
lib.bbe_checked_noalloc_seen.argtypes = [ctypes.c_void_p]
dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
for name, rollouts, sample in (("two", 200000, 2), ("twenty", 8000, 4), ("twenty", 1200, 8), ("previous steps", 16000, 3),
                               ("stuck behind the leader", 16000, 1)):
    rb = stage(name, 96, rollouts)
    counts = torch.empty(rb.n_total, dtype=torch.int32, device="cuda")
    steps = torch.empty(rb.n_races, dtype=torch.int64, device="cuda")
    bbe.bbe_rollout_noalloc(rb.n_races, rb.n_total, *(dev(a) for a in (rb.race_off, rb.L, rb.rollouts, rb.d0, rb.mu, rb.sigma,
                                                                     rb.rho, rb.P, rb.theta)),
                            None if rb.prev0 is None else dev(rb.prev0), rb.seed, rb.dist, rb.race_id0, counts, steps)
    seen = np.zeros(3, np.int32)
    assert lib.bbe_checked_noalloc_seen(seen.ctypes.data) == 0
    print(name, rollouts, "no allocation", seen)
    assert (seen[0] > 0) == (rollouts > 1200)  # 1200 each give every warp an item or less
    assert seen[2] > 0 or not name.startswith("stuck")
    head = rb.slice(0, sample)
    want, want_s, _ = oracle.batch_counts(head)
    same(counts[:head.n_total], want, name)
    same(steps[:sample], want_s, name)
print("contenders reached: ok")
