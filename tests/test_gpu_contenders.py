"""Win counts are run on a race's contenders only (the competitors near enough to the front to matter
to the first finish); counts and step totals must be those of the whole race, bit for bit, whatever
the geometry, the law, the distribution, the blocking distance and the previous steps given, and also
where the first finish comes later than the contenders were chosen for."""
import numpy as np
import pytest

import oracle
from paper_2108_02419_gb300 import workloads as W

pytestmark = pytest.mark.gpu

RACES, ROLLOUTS = 96, 1200  # enough rollouts for the batch's normal launch (a tiny batch advances everybody)


def _spread(n, seed, dist=W.DIST_NORMAL, sigma=(0.5, 1.5), theta=1.0, P=None, prev=None, lead=450.0, L=5000.0, ties=False):
    """Races of n: one competitor `lead` from the line, the others up to a tenfold of that behind it."""
    rng = np.random.default_rng(seed)
    nt = RACES * n
    rem = lead * rng.uniform(1.0, 10.0, (RACES, n))
    rem[np.arange(RACES), rng.integers(0, n, RACES)] = lead
    if ties:
        rem = np.round(rem / 200.0) * 200.0 + 200.0  # groups at equal positions
    P = None if P is None else rng.uniform(*P, nt)
    prev = None if prev is None else rng.uniform(*prev, nt)
    return W.from_arrays([n] * RACES, L, ROLLOUTS, (L - rem).ravel(), rng.uniform(15, 17, nt), rng.uniform(*sigma, nt),
                         rng.uniform(0, 1, nt), P=P, theta=np.full(nt, theta), prev0=prev, seed=seed, dist=dist)


def _stuck():
    """Chasers catch a slow leader early and stay blocked behind it: the first finish is far later than
    the least expected one.  A last competitor far behind is ruled out for a short race, and is not for the
    long one that it turns into."""
    rng = np.random.default_rng(5)
    d0 = np.tile([4800.0, 4600.0, 4550.0, 4300.0, 3600.0, 2000.0, 1000.0, 0.0], RACES)
    mu = np.tile([1.0, 16.0, 15.0, 17.0, 16.0, 16.0, 17.0, 15.0], RACES)
    sg = np.tile([0.1, 1.0, 0.5, 1.5, 1.0, 0.5, 1.5, 1.0], RACES)
    return W.from_arrays([8] * RACES, 5000.0, ROLLOUTS, d0, mu, sg, rng.uniform(0, 1, d0.size),
                         theta=np.full(d0.size, 60.0), seed=5)


CASES = {
    "two": lambda: _spread(2, 1),
    "five": lambda: _spread(5, 2),
    "twenty": lambda: _spread(20, 3),
    "full warp": lambda: _spread(32, 4),
    "alone in front": lambda: _spread(13, 5, lead=60.0),
    "wide noise": lambda: _spread(9, 6, sigma=(4.0, 9.0)),
    "uniform steps": lambda: _spread(17, 7, dist=W.DIST_UNIFORM),
    "two-point steps": lambda: _spread(11, 8, dist=W.DIST_TWO_POINT, sigma=(0.0, 3.0)),
    "far blocking": lambda: _spread(12, 9, theta=40.0),
    "no blocking": lambda: _spread(12, 10, theta=0.0),
    "preferences": lambda: _spread(10, 11, P=(0.3, 1.0)),
    "fast starts": lambda: _spread(10, 12, prev=(5.0, 200.0), theta=30.0),
    "level groups": lambda: _spread(16, 13, ties=True),
    "stuck behind the leader": _stuck,
    "time law, early": lambda: W.with_time_law(_spread(14, 14), 0.0, 300.0),
    "time law, late": lambda: W.with_time_law(_spread(14, 15), 250.0, 300.0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_contenders_alone_give_the_whole_race(name):
    import torch

    from paper_2108_02419_gb300 import bbe

    rb = CASES[name]()
    with bbe.Batch(rb) as b:
        counts, steps = b.rollout()
        b.status()
        torch.cuda.synchronize()
    want_counts, want_steps, st = oracle.batch_counts(rb)
    assert st == 0
    assert np.array_equal(counts.cpu().numpy(), want_counts)
    assert np.array_equal(steps.cpu().numpy(), want_steps)


def test_step_limit_among_contenders():
    # the limit cuts rollouts that the contenders' horizon does not
    import torch

    from paper_2108_02419_gb300 import bbe

    rb = _spread(12, 16)
    with bbe.Batch(rb) as b:
        b.set_cfg(max_steps=27)
        counts, steps = b.rollout()
        with pytest.raises(bbe.BbeError):
            b.status()
        torch.cuda.synchronize()
    want_counts, want_steps, _ = oracle.batch_counts(rb, max_steps=27)
    assert np.array_equal(counts.cpu().numpy(), want_counts)
    assert np.array_equal(steps.cpu().numpy(), want_steps)


@pytest.mark.parametrize("places", [2, 4])
@pytest.mark.parametrize("name", list(CASES))
def test_contenders_alone_give_the_first_places(name, places):
    import torch

    from paper_2108_02419_gb300 import bbe

    rb = CASES[name]()
    with bbe.Batch(rb) as b:
        counts, steps = b.places(places)
        b.status()
        torch.cuda.synchronize()
    want_counts, want_steps, st = oracle.batch_places(rb, places)
    assert st == 0
    assert np.array_equal(counts.cpu().numpy(), want_counts)
    assert np.array_equal(steps.cpu().numpy(), want_steps)


@pytest.mark.parametrize("name", ["twenty", "full warp", "far blocking", "stuck behind the leader", "time law, late"])
def test_contenders_alone_give_the_orders(name):
    # the tables are indexed by all the race's competitors, whoever is advanced
    import torch

    from paper_2108_02419_gb300 import bbe

    rb = CASES[name]()
    with bbe.Batch(rb) as b:
        orders = b.orders(2)[0]
        keys, hcounts, off, _, _ = b.order_histogram(3)
        b.status()
        torch.cuda.synchronize()
        orders, keys, hcounts = orders.cpu().numpy(), keys.cpu().numpy(), hcounts.cpu().numpy()
    want, want_h = oracle.batch_orders(rb, 2)[0], oracle.batch_order_histograms(rb, 3)[0]
    assert np.array_equal(orders, np.concatenate([np.ravel(t) for t in want]) if isinstance(want, list) else np.ravel(want))
    for r in range(rb.n_races):
        n = int(rb.race_off[r + 1] - rb.race_off[r])
        k, c = keys[off[r]:off[r + 1]], hcounts[off[r]:off[r + 1]]
        used = k != np.uint64(2 ** 64 - 1)
        got = {tuple(int(x) for x in bbe.bbe_order_key_decode(n, 3, int(key))): int(v) for key, v in zip(k[used], c[used])}
        assert got == dict(want_h[r]), r
