"""An operator whose requests come close together keeps its basis: another one that needs the room
waits until it has been idle for KEEP_IDLE_S, but no longer than KEEP_WAIT_S in all (no GPU)."""
import threading
import time

import pytest

from paper_0707_0131_gb300 import serving
from test_host_serving import _FakeWorker, _server


@pytest.mark.parametrize("steady", [False, True])
def test_recently_used_operator_is_kept(steady):
    a, b = _FakeWorker("a", 20, 60, time.perf_counter()), _FakeWorker("b", 30, 40, 0.0)
    srv = _server(80, [a, b])
    srv._admit(a)
    a.last_used = t0 = time.perf_counter()
    done = threading.Event()

    def requests():  # a is used again and again, each time for a moment
        while not done.is_set():
            a.last_used = time.perf_counter()
            done.wait(0.01)

    t = threading.Thread(target=requests)
    if steady:
        t.start()
    srv._admit(b)  # a's workspace is not enough: its basis has to go
    waited = time.perf_counter() - t0
    done.set()
    if steady:
        t.join()
    assert b.active and not a.resident and srv.closes == 1
    assert waited >= (serving.KEEP_WAIT_S if steady else serving.KEEP_IDLE_S) - 0.02
