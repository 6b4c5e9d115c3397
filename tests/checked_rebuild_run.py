"""A work list that cannot be made (the checked build says so on request, as if memory had run out) leaves the
batch as it was: its launch, its layout and its results.  Started by tests/test_gpu_rebuild_failure.py with BBE_LIB
naming the checked build."""
import ctypes
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import oracle  # noqa: E402
from paper_2108_02419_gb300 import bbe  # noqa: E402
from paper_2108_02419_gb300 import workloads as W  # noqa: E402

assert bbe.LIB_PATH == os.environ["BBE_LIB"], bbe.LIB_PATH
lib = bbe.lib()
lib.bbe_checked_fail_list.argtypes = [ctypes.c_void_p, ctypes.c_int32]


def fails(call):
    try:
        call()
    except bbe.BbeError as e:
        assert e.status == -4, e
        return True
    return False


# 100 races of 8: enough items for tickets with two slots per lane, not with four
rb = W.uniform_batch(seed=17, n_races=100, n=8, L=1500.0, rollouts=1000)
want, want_s, _ = oracle.batch_counts(rb)
with bbe.Batch(rb) as b:

    def check():
        counts, steps = b.rollout()
        b.status()
        assert np.array_equal(counts.cpu().numpy(), want) and np.array_equal(steps.cpu().numpy(), want_s)

    check()
    cfg, layout = b.cfg(), b.layout()
    for change in (lambda: b.set_cfg(slots_per_lane=4), lambda: b.set_cfg(rollouts_per_lane=1, warps_per_block=8),
                   lambda: b.set_layout(np.full(33, 1, np.int32)), lambda: b.set_layout(np.full(33, 4, np.int32))):
        lib.bbe_checked_fail_list(b.handle, 1)
        assert fails(change)
        assert b.cfg() == cfg and np.array_equal(b.layout(), layout)
        lib.bbe_checked_fail_list(b.handle, 0)
        check()
    b.set_cfg(slots_per_lane=4)
    check()
    four, layout = b.cfg(), b.layout()
    lib.bbe_checked_fail_list(b.handle, 1)
    assert fails(lambda: b.set_cfg())
    assert b.cfg() == four and np.array_equal(b.layout(), layout)
    lib.bbe_checked_fail_list(b.handle, 0)
    check()
    b.set_cfg()
    check()
print("rebuild failures: ok")
