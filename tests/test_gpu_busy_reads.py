"""Reading a finished run and creating an instance while another run fills the
device: neither waits for that run's blocks."""
import time

import pytest

from paper_2205_13399_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,replicas,I_max", [
    (40, 1500, 300_000),  # two blocks an SM, which leave no registers
    (75, 600, 300_000),   # one, four rounds of them
])
def test_fronts_are_read_beside_a_run_that_fills_the_device(n, replicas, I_max):
    import torch
    from paper_2205_13399_gb300 import moda
    small, big = (inputs.euclid_instance(k, 0.0, False, index=0, workload="BATCH") for k in (25, n))
    g, h = (moda.Instance(q.F1, q.F2, q.D) for q in (small, big))
    run = moda.anneal(g, replicas=64, I_max=20_000, snapshot_every=10_000).wait()
    want = run.read_archive(-1), run.read_archive(-1, snapshot=0)
    stream = torch.cuda.Stream()
    moda.anneal(h, replicas=replicas, I_max=100, stream=stream).wait()
    busy = moda.anneal(h, replicas=replicas, I_max=I_max, stream=stream)
    time.sleep(0.01)
    t0 = time.perf_counter()
    got = run.read_archive(-1), run.read_archive(-1, snapshot=0)
    other = moda.Instance(small.F1, small.F2, small.D)
    t1 = time.perf_counter()
    busy.wait()
    t2 = time.perf_counter()
    assert got == want and other.n == 25
    assert t1 - t0 < 0.25 * (t2 - t0)  # (about 10 ms of 150 to 400)
