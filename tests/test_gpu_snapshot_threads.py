"""A snapshot batch keeps one host record per snapshot until a call needs one per race.  Calls that only ask
for something may be made from several threads at once, before, while and after that happens."""
import threading

import numpy as np
import pytest

from paper_2108_02419_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_totals_while_another_thread_asks_for_a_layout():
    torch = pytest.importorskip("torch")
    from paper_2108_02419_gb300 import bbe

    n, cap, bettors, dry = 5, 256, 2000, 50
    src = W.single_race_start(seed=8, n=n, L=1500.0)
    with bbe.Batch(src) as b:
        pos = torch.zeros(n * cap, dtype=torch.float32, device="cuda")
        stp, ns = torch.zeros_like(pos), torch.zeros(1, dtype=torch.int32, device="cuda")
        bbe.bbe_race_trajectory(b.handle, 1 << 30, cap, pos, stp, ns)
        for _ in range(40):
            h, snaps = bbe.bbe_snapshot_batch(b.handle, 0, pos, stp, ns, cap, 1, bettors, dry, 100)
            m = snaps * bettors
            go, done = threading.Barrier(3), threading.Event()
            infos, sizes = [], []

            def ask():
                go.wait()
                while not done.is_set():
                    infos.append(bbe.bbe_batch_info(h))
                infos.append(bbe.bbe_batch_info(h))

            def relist():
                go.wait()
                bbe.bbe_batch_set_cfg(h, rollouts_per_lane=16)

            threads = [threading.Thread(target=ask), threading.Thread(target=relist)]
            for t in threads:
                t.start()
            go.wait()
            try:
                sizes.append(bbe.bbe_order_table_size(h, 2))
                sizes.append(bbe.bbe_order_table_size(h, 3))
            finally:
                done.set()
                for t in threads:
                    t.join()
            counts = torch.empty(m * n, dtype=torch.int32, device="cuda")
            bbe.bbe_rollout_batch(h, counts)
            bbe.bbe_batch_status(h)
            wins = counts.view(m, n).sum(dim=1).cpu().numpy()
            bbe.bbe_destroy_batch(h)
            assert sizes == [m * n ** 2, m * n ** 3]
            for i in infos:
                assert i == dict(n_races=m, n_competitors=m * n, total_rollouts=m * dry, max_competitors=n)
            assert np.all(wins == dry)
