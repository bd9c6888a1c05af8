"""How long a request waits before another operator is closed for it: not at all unless that one's requests
come closer together than the work its basis took, and no longer than that work (no GPU)."""
import threading
import time

import pytest

from paper_0707_0131_gb300 import serving
from test_host_serving import _FakeWorker, _server


@pytest.mark.parametrize("basis_s,gap_s,steady,least,most", [
    (0.0, 0.0, True, 0.0, 0.2),      # nothing to lose
    (0.01, 0.005, False, 0.005, 0.045),  # idle for as long as the basis took
    (0.1, 0.01, True, 0.08, 0.4),    # in use all the time: the work of the basis and no longer
    (0.03, 0.5, True, 0.0, 0.2),     # its next request comes too late to be worth the wait
    (20.0, 0.01, True, 0.48, 2.0),   # a costly basis: the limits stay
])
def test_wait_is_bounded_by_the_work_of_the_basis(basis_s, gap_s, steady, least, most):
    a, b = _FakeWorker("a", 20, 60, time.perf_counter()), _FakeWorker("b", 30, 40, 0.0)
    srv = _server(80, [a, b])
    srv._admit(a)
    a.basis_s, a.gap_s = basis_s, gap_s
    a.last_used = t0 = time.perf_counter()
    done = threading.Event()

    def requests():
        while not done.is_set():
            a.last_used = time.perf_counter()
            done.wait(0.002)

    t = threading.Thread(target=requests)
    if steady:
        t.start()
    srv._admit(b)
    waited = time.perf_counter() - t0
    done.set()
    if steady:
        t.join()
    assert b.active and not a.resident
    assert least <= waited <= most, waited


def test_gaps_between_requests_are_followed():
    w = _FakeWorker("a", 20, 60, 0.0)
    w.gap_s, w.last_asked = float("inf"), -float("inf")
    srv = _server(80, [w])
    import numpy as np

    b = np.zeros(4, dtype=np.complex128)
    srv.submit("a", b)
    assert w.gap_s == float("inf")
    time.sleep(0.02)
    srv.submit("a", b)
    assert 0.02 <= w.gap_s < 0.1
    for _ in range(10):
        srv.submit("a", b)
    assert w.gap_s < 0.01
