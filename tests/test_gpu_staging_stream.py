"""Staging (bbe_race_init, bbe_snapshot_batch) is finished when the call returns, whatever stream it was given,
the default stream (handle 0) included: the batch may then be used on any stream, or destroyed."""
import numpy as np
import pytest

import oracle
from paper_2108_02419_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def busy():
    """Some ten milliseconds of ordinary work on the current stream."""
    a = torch.ones(4096, 4096, device="cuda")
    for _ in range(20):
        a = a @ a
    return a


def small(seed, n_races):
    # 40 races go up in one copy, 20000 (more than 4 MB) array by array
    return W.uneven_batch(seed=seed, n_races=n_races, n_lo=1, n_hi=24, rollouts=20, rem_lo=100.0, rem_hi=900.0)


def rolled(h, rb, stream):
    with torch.cuda.stream(stream):
        counts = torch.empty(rb.n_total, dtype=torch.int32, device="cuda")
        steps = torch.empty(rb.n_races, dtype=torch.int64, device="cuda")
    from paper_2108_02419_gb300 import bbe

    bbe.bbe_rollout_batch(h, counts, steps, stream)
    bbe.bbe_batch_status(h, stream)
    stream.synchronize()
    return counts.cpu().numpy(), steps.cpu().numpy()


@pytest.mark.parametrize("own", [False, True])
@pytest.mark.parametrize("n_races", [1, 40, 20000])
def test_a_batch_is_in_place_when_staging_returns(n_races, own):
    from paper_2108_02419_gb300 import bbe

    rb = small(n_races, n_races)
    staged_on = torch.cuda.Stream() if own else torch.cuda.default_stream()
    side = torch.cuda.Stream()
    rolled_first = None
    for attempt in range(2):
        with torch.cuda.stream(staged_on):
            busy()
            with bbe.Batch(rb, staged_on) as b:
                assert staged_on.query()  # nothing of the staging is left to do
                if attempt == 0:
                    continue  # destroyed without a pass
                rolled_first = rolled(b.handle, rb, side)
    m = min(n_races, 200)
    head = rb.slice(0, m)
    want_c, want_s, _ = oracle.batch_counts(head)
    assert np.array_equal(rolled_first[0][:head.n_total], want_c)
    assert np.array_equal(rolled_first[1][:m], want_s)


def test_a_snapshot_batch_is_in_place_when_the_call_returns():
    from paper_2108_02419_gb300 import bbe

    n, cap, bettors, dry = 5, 256, 60, 30
    src = W.single_race_start(seed=3, n=n, L=900.0)
    side = torch.cuda.Stream()
    with bbe.Batch(src) as b:
        pos = torch.zeros(n * cap, dtype=torch.float32, device="cuda")
        stp, ns = torch.zeros_like(pos), torch.zeros(1, dtype=torch.int32, device="cuda")
        bbe.bbe_race_trajectory(b.handle, 1 << 30, cap, pos, stp, ns)
        busy()
        h, snaps = bbe.bbe_snapshot_batch(b.handle, 0, pos, stp, ns, cap, 10, bettors, dry, 100)
        assert torch.cuda.default_stream().query()
        m = snaps * bettors
        P, S = pos.view(cap, n).cpu().numpy(), stp.view(cap, n).cpu().numpy()
        d0 = np.vstack([src.d0] + [P[s * 10 - 1] for s in range(1, snaps)])
        pv = np.vstack([src.mu * src.P] + [S[s * 10 - 1] for s in range(1, snaps)])
        one = W.from_arrays([n] * m, 900.0, dry, np.repeat(d0, bettors, axis=0), np.tile(src.mu, m),
                            np.tile(src.sigma, m), np.tile(src.rho, m), prev0=np.repeat(pv, bettors, axis=0), seed=src.seed)
        one.race_id0 = 100
        try:
            got_c, got_s = rolled(h, one, side)
        finally:
            bbe.bbe_destroy_batch(h)
    want_c, want_s, _ = oracle.batch_counts(one)
    assert np.array_equal(got_c, want_c)
    assert np.array_equal(got_s, want_s)


def test_host_arrays_are_read_when_the_stream_has_written_them():
    # every array in pinned memory, filled by copies that are still queued when the call is made
    from paper_2108_02419_gb300 import bbe

    rb = small(7, 40)
    rb.prev0 = (rb.mu * rb.P).astype(np.float32)
    s = torch.cuda.Stream()
    host = [np.ascontiguousarray(a) for a in (rb.race_off, rb.L, rb.rollouts, rb.d0, rb.mu, rb.sigma, rb.rho, rb.P, rb.theta,
                                             rb.prev0)]
    there = [torch.from_numpy(a).cuda() for a in host]
    here = [torch.from_numpy(np.zeros_like(a)).pin_memory() for a in host]
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        busy()
        for h, t in zip(here, there):
            h.copy_(t, non_blocking=True)
    h = bbe.bbe_race_init(rb.n_races, *here[:7], here[7], here[8], here[9], rb.seed, rb.dist, rb.race_id0, s)
    try:
        got_c, got_s = rolled(h, rb, s)
    finally:
        bbe.bbe_destroy_batch(h)
    want_c, want_s, _ = oracle.batch_counts(rb)
    assert np.array_equal(got_c, want_c)
    assert np.array_equal(got_s, want_s)
