"""A launch change whose work list cannot be made leaves the batch as it was (tests/checked_rebuild_run.py, on the
checked build of the library)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_a_failed_rebuild_leaves_the_batch_as_it_was():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_02419_gb300 import build

    so = build.build(checked=True)
    res = subprocess.run([sys.executable, os.path.join(HERE, "checked_rebuild_run.py")],
                         env=dict(os.environ, BBE_LIB=so), capture_output=True, text=True, timeout=600)
    assert res.returncode == 0, res.stdout[-3000:] + res.stderr[-4000:]
    assert "rebuild failures: ok" in res.stdout
