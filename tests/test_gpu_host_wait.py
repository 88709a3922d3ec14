"""A host wait of the library beside another thread of the caller on one core."""
import os
import threading
import time

import pytest

from paper_1302_7104_gb300 import inputs as I
from paper_1302_7104_gb300 import pclb as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _share(work, seconds=0.4):
    """CPU share of this thread while `work` is repeated by another thread on the same core."""
    stop = threading.Event()

    def loop():
        while not stop.is_set():
            work()

    th = threading.Thread(target=loop)
    th.start()
    time.sleep(0.05)
    t0, c0 = time.perf_counter(), time.thread_time()
    while time.perf_counter() - t0 < seconds:
        pass
    share = (time.thread_time() - c0) / (time.perf_counter() - t0)
    stop.set()
    th.join()
    return share


def test_short_waits_leave_the_core_to_other_threads():
    """Waits of up to ~2 ms poll instead of sleeping; every now and then they offer
    the core, so a thread that computes there keeps nearly all of it (0.69, if
    the wait held on).  The best of three runs, as the machine may be busy."""
    if not hasattr(os, "sched_setaffinity"):
        pytest.skip("no affinity calls")
    w = I.kh(n_r=2048, n_theta=2048)
    cores = os.sched_getaffinity(0)
    with P.PCLB(w, precision="fp32") as g:
        g.set_state()
        g.sync()
        try:
            os.sched_setaffinity(0, {max(cores)})

            def work():
                g.step(5)          # about 1.5 ms
                g.sync()

            shares = [_share(work) for _ in range(3)]
        finally:
            os.sched_setaffinity(0, cores)
        assert g.status_flags() == 0
    assert max(shares) > 0.75, shares
