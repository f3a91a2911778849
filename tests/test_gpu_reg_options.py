"""The register annealer's options where its other shapes run them: four and
eight words a worker (larger instances, or small ones on a crowded device) and
archives beyond the slots on chip; and the team annealer at a prescribed layout
at full size."""
import numpy as np
import pytest

import oracle
from paper_2205_13399_gb300 import inputs
from parity import compare, gpu_run, oracle_run
from test_gpu_reg import FAST, _Inst

pytestmark = pytest.mark.gpu


def _anti(n):
    """Objectives whose flows add up to a constant: most states of a descent are
    not dominated by one another, so archives grow with the run."""
    rng = np.random.default_rng(0)
    F1 = rng.integers(0, 100, (n, n))
    return _Inst(F1, 99 - F1, rng.integers(1, 100, (n, n)))


@pytest.mark.parametrize("norm", [False, True])
def test_raises_on_a_crowded_device(norm):
    """400 replicas of n = 25: four words a worker, draws for chunks that may
    accept only."""
    inst = inputs.uniform_instance(25, index=85, workload="P8")
    kw = dict(I_max=1500, seed=25, escape="offset", beta=30_000, normalize=norm)
    kw.update(dict(delta0=3e8, deltaf=1e6, xi=0.02) if norm else FAST)
    _, _, res, tr = gpu_run(inst, trace=True, replicas=400, **kw)
    rows = [0, 151, 399]
    _, orc = oracle_run(inst, trace=True, replicas=rows, **kw)
    assert all(r[3] > 0 for r in orc["stats"])
    compare(res, rows, orc, 625, gpu_trace=tr)


def _snapshots(inst, R, I_max, every, **kw):
    from paper_2205_13399_gb300 import moda
    g = moda.Instance(inst.F1, inst.F2, inst.D)
    run = moda.anneal(g, replicas=R, I_max=I_max, snapshot_every=every, **kw).wait()
    _, orc = oracle_run(inst, replicas=R, I_max=I_max, snapshot_every=every, **kw)
    snap = orc["snapshots"]
    for r in range(R):
        for j in range(I_max // every):
            pts = [(int(a), int(b)) for a, b in snap["E"][r, j, :int(snap["count"][r, j])]]
            want = sorted(pts[i] for i in oracle.nondominated(pts))
            got = run.read_archive(replica=r, snapshot=j)
            assert [(p["E1"], p["E2"]) for p in got] == want, (r, j)
            for p in got:
                assert pts[p["slot"]] == (p["E1"], p["E2"])
                if p["perm"] is not None:
                    assert p["perm"] == oracle.decode_permutation(snap["bits"][r, j, p["slot"]])
    compare(run.read(), range(R), orc, inst.n * inst.n)
    return orc


@pytest.mark.parametrize("n,esc", [(40, "archive"), (56, "archive"), (56, "offset")])
def test_snapshots_of_larger_instances(n, esc):
    inst = inputs.uniform_instance(n, index=n, workload="P8")
    _snapshots(inst, 2, 900, 300, seed=n, escape=esc, beta=30_000, **FAST)


def test_snapshots_beyond_the_slots_on_chip():
    inst = _anti(36)
    orc = _snapshots(inst, 2, 9000, 3000, seed=36, accept="lenient", delta0=2e6, deltaf=3e5,
                     xi=0.01)
    assert (orc["count"] > 768).all() and (orc["stats"][:, 1] > 0).all()


def test_archives_beyond_the_slots_on_chip():
    inst = _anti(36)
    kw = dict(replicas=2, I_max=9000, seed=36, accept="lenient", delta0=2e6, deltaf=3e5, xi=0.01)
    _, _, res, tr = gpu_run(inst, trace=True, **kw)
    _, orc = oracle_run(inst, trace=True, **kw)
    assert (orc["count"] > 768).all() and (orc["stats"][:, 1] > 0).all()
    compare(res, range(2), orc, 36 * 36, gpu_trace=tr)


@pytest.mark.parametrize("layout", [dict(field_cache="on"), dict(prefetch=7)])
def test_team_annealer_at_a_prescribed_layout(layout):
    """The n = 25 workload at its full 10^5 iterations on the team annealer, which
    requests without a layout no longer reach."""
    inst = inputs.workload_instance("P25")
    kw = dict(I_max=100_000, seed=3)
    _, _, res, _ = gpu_run(inst, replicas=16, engine="warp", **layout, **kw)
    _, _, reg, _ = gpu_run(inst, replicas=16, **kw)
    for key in ("count", "E_final", "x"):
        assert np.array_equal(getattr(res, key), getattr(reg, key)), key
    rows = [0, 15]
    _, orc = oracle_run(inst, replicas=rows, **kw)
    compare(res, rows, orc, 625)
