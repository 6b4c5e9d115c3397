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
