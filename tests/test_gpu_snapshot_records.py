"""A snapshot batch keeps one host record per snapshot for all its bettors' races and is laid out by the
device: whatever is asked of it (win counts, another launch, places, order tallies, the histogram's
layout, the batch's totals) equals the same races staged one by one."""
import numpy as np
import pytest

from paper_2108_02419_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, bettors, dry_runs, every, law", [
    (5, 1, 1, 1, "position"), (5, 37, 7, 9, "position"), (2, 400, 50, 11, "time"), (13, 3, 333, 20, "position"),
    (32, 5, 2100, 40, "time"), (20, 150, 129, 25, "position")])
def test_snapshot_batch_equals_its_races_staged_one_by_one(n, bettors, dry_runs, every, law):
    import torch

    from paper_2108_02419_gb300 import bbe

    L, cap, id0 = 900.0, 256, 4_000_000_000  # stream ids wrap around 2^32 in none of these, and are above 2^31
    rng = np.random.default_rng(n)
    src = W.single_race_start(seed=n, n=n, L=L)
    src.theta = rng.uniform(0.5, 6.0, n).astype(np.float32)
    src.P = rng.uniform(0.8, 1.0, n).astype(np.float32)
    if law == "time":
        src = W.with_time_law(src, 4.0, 60.0)
    with bbe.Batch(src) as b:
        pos = torch.zeros(n * cap, dtype=torch.float32, device="cuda")
        stp, ns = torch.zeros_like(pos), torch.zeros(1, dtype=torch.int32, device="cuda")
        bbe.bbe_race_trajectory(b.handle, 1 << 30, cap, pos, stp, ns)
        h, snaps = bbe.bbe_snapshot_batch(b.handle, 0, pos, stp, ns, cap, every, bettors, dry_runs, id0)
    P, S = pos.view(cap, n).cpu().numpy(), stp.view(cap, n).cpu().numpy()
    d0 = np.vstack([src.d0] + [P[s * every - 1] for s in range(1, snaps)])
    pv = np.vstack([src.mu * src.P] + [S[s * every - 1] for s in range(1, snaps)])
    m = snaps * bettors
    one = W.from_arrays([n] * m, L, dry_runs, np.repeat(d0, bettors, axis=0), np.tile(src.mu, m), np.tile(src.sigma, m),
                        np.tile(src.rho, m), P=np.tile(src.P, m), theta=np.tile(src.theta, m),
                        prev0=np.repeat(pv, bettors, axis=0), seed=src.seed)
    one.race_id0 = id0
    if law == "time":
        one = W.with_time_law(one, np.repeat(4.0 + every * np.arange(snaps), bettors), 60.0)

    def ask(handle, first):
        """Everything in turn: what needs one record per race comes after what does not."""
        out = [bbe.bbe_batch_info(handle)]
        counts = torch.empty(m * n, dtype=torch.int32, device="cuda")
        steps = torch.empty(m, dtype=torch.int64, device="cuda")

        def roll():
            bbe.bbe_rollout_batch(handle, counts, steps)
            bbe.bbe_batch_status(handle)
            out.extend([counts.cpu().numpy().copy(), steps.cpu().numpy().copy()])

        roll()
        if first == "shape":
            bbe.bbe_batch_set_cfg(handle, rollouts_per_lane=3, slots_per_lane=1)
            roll()
        k = min(n, 3)
        places = torch.empty((m * n, k), dtype=torch.int32, device="cuda")
        orders = torch.empty(bbe.bbe_order_table_size(handle, k), dtype=torch.int32, device="cuda")
        bbe.bbe_order_counts(handle, k, orders, places, steps)
        bbe.bbe_batch_status(handle)
        out.extend([orders.cpu().numpy(), places.cpu().numpy(), steps.cpu().numpy().copy(),
                    bbe.bbe_order_histogram_layout(handle, k, m)])
        bbe.bbe_batch_set_layout(handle, np.full(33, 2, np.int32))
        roll()
        out.append(bbe.bbe_batch_info(handle))
        return out

    for first in ("shape", "records"):
        if first == "records":
            with bbe.Batch(src) as b:
                h, snaps2 = bbe.bbe_snapshot_batch(b.handle, 0, pos, stp, ns, cap, every, bettors, dry_runs, id0)
                assert snaps2 == snaps
        try:
            got = ask(h, first)
        finally:
            bbe.bbe_destroy_batch(h)
        with bbe.Batch(one) as b:
            want = ask(b.handle, first)
        assert len(got) == len(want)
        for g, w in zip(got, want):
            assert g == w if isinstance(g, dict) else np.array_equal(g, w)
