"""Tuning requests of the options beyond the default algorithm: with the engine
left open the untuned request (the register annealer) is a candidate."""
import numpy as np
import pytest

from paper_2205_13399_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(escape="offset", beta=40_000), dict(normalize=True),
                                dict(snapshot_every=1000)])
def test_tuning_an_open_request_keeps_the_fastest_engine(kw):
    from paper_2205_13399_gb300 import moda
    qi = inputs.uniform_instance(30, index=8, workload="P8")
    g = moda.Instance(qi.F1, qi.F2, qi.D)
    kw = dict(replicas=100, I_max=4000, seed=3, **kw)
    best, ms = moda.autotune(g, trial_iters=3000, **kw)
    # the register annealer is two to thirteen times as fast as any block shape
    assert best.block_threads == 0 and best.prefetch == 0 and ms > 0
    assert best.replicas == 100 and best.I_max == 4000 and best.engine == 0
    assert best.snapshot_every == kw.get("snapshot_every", 0)
    a, b = (moda.anneal(g, **k).wait().read() for k in (dict(params=best), kw))
    for key in ("count", "E", "bits", "x", "E_final", "stats"):
        assert np.array_equal(getattr(a, key), getattr(b, key)), key


def test_prescribed_shapes_are_tuned_as_before():
    from paper_2205_13399_gb300 import moda
    qi = inputs.uniform_instance(12, index=8, workload="P8")
    g = moda.Instance(qi.F1, qi.F2, qi.D)
    best, ms = moda.autotune(g, trial_iters=300, engine="block", escape="offset", beta=40_000,
                             replicas=4, I_max=1000)
    assert best.block_threads >= 32 and ms > 0
