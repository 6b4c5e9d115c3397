"""The contender search of the rollout kernel is reached and gives the whole race: the checked build of the
library counts the work items run on contenders alone (tests/checked_contenders_run.py)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_contenders_are_reached_and_give_the_whole_race():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_02419_gb300 import build

    so = build.build(checked=True)
    res = subprocess.run([sys.executable, os.path.join(HERE, "checked_contenders_run.py")],
                         env=dict(os.environ, BBE_LIB=so), capture_output=True, text=True, timeout=900)
    assert res.returncode == 0, res.stdout[-3000:] + res.stderr[-4000:]
    assert "contenders reached: ok" in res.stdout


@pytest.mark.parametrize("law", ["position", "time"])
def test_captured_passes_search_anew(law):
    # a caller's graph holds the search and the rollouts of a win and of a place pass
    torch = pytest.importorskip("torch")
    from paper_2108_02419_gb300 import bbe
    from paper_2108_02419_gb300 import workloads as W

    rb = W.uniform_batch(seed=1, n_races=256, n=20, rollouts=4000)
    if law == "time":
        rb = W.with_time_law(rb, 3.0, 300.0)
    with bbe.Batch(rb) as b:
        counts, steps = b.new_outputs()
        pc = torch.empty((rb.n_total, 3), dtype=torch.int32, device="cuda")
        ps = torch.empty_like(steps)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            b.rollout(counts, steps)
            b.places(3, pc, ps)
        for _ in range(2):
            for t in (counts, steps, pc, ps):
                t.fill_(-1)
            g.replay()
            torch.cuda.synchronize()
            want, want_s = b.rollout()
            places, places_s = b.places(3)
            b.status()
            assert torch.equal(counts, want) and torch.equal(steps, want_s)
            assert torch.equal(pc, places) and torch.equal(ps, places_s)
            assert torch.equal(counts.view(-1), pc[:, 0])
