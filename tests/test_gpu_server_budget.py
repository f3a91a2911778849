"""What the server counts against its memory budget."""
import time

import pytest

from paper_2205_13399_gb300 import inputs

pytestmark = pytest.mark.gpu


def _until(cond, seconds=30.0):
    t0 = time.time()
    while not cond():
        assert time.time() - t0 < seconds, "server did not get there"
        time.sleep(0.001)


def test_requests_that_fit_by_their_buffers_run_together():
    """Two default requests of n = 75 (0.13 GB of buffers each; no field cache
    is allocated for them) under a budget of 1 GB."""
    from paper_2205_13399_gb300 import moda
    qi = inputs.euclid_instance(75, 0.0, False, index=1, workload="BATCH")
    inst = moda.Instance(qi.F1, qi.F2, qi.D)
    kw = dict(replicas=32, I_max=3_000_000)  # about 0.1 s
    srv = moda.Server(hbm_budget=10 ** 9)
    seen = []
    tickets = [srv.submit(inst, seed=k, **kw) for k in range(2)]
    runs = {}
    t0 = time.time()
    while len(runs) < 2:
        seen.append(srv.info())
        for t in tickets:
            if t not in runs:
                r = srv.poll(t)
                if r is not None:
                    runs[t] = r
        assert time.time() - t0 < 60
    assert max(i["running"] for i in seen) == 2
    assert all(i["bytes_in_use"] <= 10 ** 9 for i in seen)
    srv.close()


def test_the_budget_covers_every_buffer():
    """n = 40: archives beyond the slots on chip keep least penalties in device
    memory too.  A budget one byte below two requests holds one at a time."""
    from paper_2205_13399_gb300 import moda
    qi = inputs.euclid_instance(40, 0.0, False, index=1, workload="BATCH")
    inst = moda.Instance(qi.F1, qi.F2, qi.D)
    kw = dict(replicas=16, I_max=60_000, escape="offset", beta=1000)  # (no optional memory)
    srv = moda.Server()
    srv.submit(inst, seed=0, **kw)
    _until(lambda: srv.info()["running"] == 1)
    one = srv.info()["bytes_in_use"]
    srv.close()
    assert one > 0
    srv = moda.Server(hbm_budget=2 * one - 1)
    tickets = [srv.submit(inst, seed=k, **kw) for k in range(2)]
    done, most = 0, 0
    t0 = time.time()
    while done < 2:
        most = max(most, srv.info()["bytes_in_use"])
        for t in list(tickets):
            r = srv.poll(t)
            if r is not None:
                r.close()
                tickets.remove(t)
                done += 1
        assert time.time() - t0 < 60
    assert most <= 2 * one - 1
    srv.close()


def test_running_falls_without_a_poll():
    """A program that watches the server's counters until it is idle."""
    from paper_2205_13399_gb300 import moda
    qi = inputs.uniform_instance(8, index=1, workload="P8")
    inst = moda.Instance(qi.F1, qi.F2, qi.D)
    srv = moda.Server()
    t = srv.submit(inst, replicas=2, I_max=2000, seed=1)
    _until(lambda: srv.info()["pending"] == 0)
    _until(lambda: srv.info()["running"] == 0, seconds=5.0)
    assert srv.poll(t) is not None
    srv.close()
