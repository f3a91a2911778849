"""Delta E beyond int32: the counters of a run, the profiling ones among them,
are the same in every run."""
import numpy as np
import pytest

from test_gpu_reg import _Inst

pytestmark = pytest.mark.gpu


def test_counters_of_wide_runs_repeat():
    """300 replicas at a temperature at which states keep crossing the 32-bit
    range.  (When trials read a bound that another warp was writing, about one
    run in thirty of this one counted a few landings more or less.)"""
    from paper_2205_13399_gb300 import moda
    rng = np.random.default_rng(41)
    F1, F2 = (rng.integers(300, 900, (41, 41)) for _ in range(2))
    inst = _Inst(F1, F2, rng.integers(50, 120, (41, 41)))
    g = moda.Instance(inst.F1, inst.F2, inst.D)
    kw = dict(replicas=300, I_max=20_000, seed=1, delta0=1e10, deltaf=3e7, xi=2e-3)
    first = moda.anneal(g, **kw).wait().read()
    assert first.stats[:, 1].sum() > 0
    for _ in range(60):
        assert np.array_equal(moda.anneal(g, **kw).wait().read().stats, first.stats)
