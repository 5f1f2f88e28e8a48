"""GPU: the host half of a batch -- its threads serve all systems' vectors and
temperatures together."""
import os
import threading
import time

import numpy as np
import pytest

import ftlm_workloads as W
import paper_2607_25585_gb300 as F

pytestmark = pytest.mark.gpu


@pytest.mark.skipif(len(os.sched_getaffinity(0)) < 8, reason="needs eight hardware threads")
def test_two_long_runs_use_more_than_two_threads():
    """Two systems of 64 vectors and 200 steps: 100 ms of eigenproblems on one thread,
    of which a thread a system would leave 50."""
    T = np.geomspace(1, 50, 40)
    systems = [F.System.from_dict(W.ring(N=6, two_s=2, Bdir=d)) for d in ((1, 1, 1), (0, 1, 2))]
    kw = dict(R=64, M=200, T=T, seed=3, dtype="c128")
    ref = F.run_batch(systems, **kw)
    most, done = [0], threading.Event()

    def watch():
        while not done.is_set():
            most[0] = max(most[0], len(os.listdir("/proc/self/task")))
            time.sleep(2e-4)

    w = threading.Thread(target=watch)
    w.start()
    time.sleep(0.05)
    before, most[0] = most[0], 0
    out = F.run_batch(systems, **kw)
    done.set()
    w.join()
    assert most[0] >= before + 4, (before, most[0])
    for k, (a, b) in enumerate(zip(out, ref)):       # any number of threads: the same bits
        one = F.sums(a["alpha"], a["beta"], a["p"], a["M_eff"], systems[k].dim, 2.0, T)
        for key in ("lnZ", "E", "C", "M_B"):
            assert np.array_equal(a[key], b[key]) and np.array_equal(a[key], one[key])
    for s in systems:
        s.close()


def test_a_batch_tells_the_first_system_that_failed():
    """A start vector of zero norm cannot be solved; the message is that system's."""
    T = np.array([1.0])
    systems = [F.System.from_dict(W.ring(N=n, two_s=2)) for n in (4, 5)]
    out = F.run_batch(systems, R=3, M=6, T=T, seed=1, dtype="c128")
    assert all(np.isfinite(o["lnZ"]).all() for o in out)
    bad = [F.System([1, 1], J=np.array([[0, 1e308], [0, 0]]), B=(0, 0, 1)), systems[0]]
    with pytest.raises(F.FtlmError):
        F.run_batch(bad, R=2, M=3, T=T, seed=1, dtype="c128")
    for s in systems + bad[:1]:
        s.close()
