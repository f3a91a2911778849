"""GPU parity of the register annealer, the warp engine's form without a
prescribed layout: per-iteration traces against the CPU oracle where its
tilings change (one word and several per worker, draw warps and inline
draws, the last word full and ragged, rebuilds by matrix products and
without, Delta E beyond int32 with a later return to it), and its
acceptance test over every draw."""
import numpy as np
import pytest

import oracle
from paper_2205_13399_gb300 import inputs
from parity import compare, gpu_run, oracle_run

pytestmark = pytest.mark.gpu

FAST = dict(delta0=2e6, deltaf=3e3, xi=0.02)


class _Inst:
    def __init__(self, F1, F2, D):
        for F in (F1, F2):
            np.fill_diagonal(F, 0)
        D = np.triu(D, 1)
        self.F1, self.F2 = F1.astype(np.int16), F2.astype(np.int16)
        self.D, self.n = (D + D.T).astype(np.int16), len(D)


# state words and words per worker change at n = 26 (W 22: two words), 36 (41:
# four), 54 (92: eight); 16, 32 and 48 have a full last word, 2 a single group
@pytest.mark.parametrize("n", [2, 3, 4, 8, 15, 16, 25, 26, 32, 35, 36, 48, 53, 54])
@pytest.mark.parametrize("acc,arc", [("strict", "explore"), ("lenient", "exploit")])
def test_traces_at_the_edges_of_the_tilings(n, acc, arc):
    inst = inputs.euclid_instance(n, 0.3, n % 2 == 1, index=n, workload="BATCH") if n > 3 else \
        inputs.uniform_instance(n, index=n, workload="P8")
    kw = dict(replicas=2, I_max=900, seed=n, accept=acc, archive=arc, **FAST)
    _, _, res, tr = gpu_run(inst, trace=True, **kw)
    _, orc = oracle_run(inst, trace=True, **kw)
    compare(res, range(2), orc, n * n, gpu_trace=tr)


@pytest.mark.parametrize("n,fmax,dmax", [
    (20, 120, 250),     # byte flows and distances: one plane of each
    (20, 120, 900),     # distances over two planes
    (21, 9000, 40),     # flows over two planes
    (18, 400, 20000),   # both (M up to 40,000)
    (14, 400, 32767),   # 2 max d = 65,534: the largest that fits 16 bits
])
@pytest.mark.parametrize("replicas", [3, 400])
def test_rebuilds_over_the_value_ranges(n, fmax, dmax, replicas):
    """Jumps to members that accept again rebuild Delta E; the same run with
    many replicas takes the tiling of a crowded device."""
    rng = np.random.default_rng(n + fmax + dmax)
    F1, F2 = (rng.integers(0, fmax + 1, (n, n)) * (rng.random((n, n)) < 0.3) for _ in range(2))
    D = rng.integers(dmax // 2, dmax + 1, (n, n))
    inst = _Inst(F1, F2, D)
    w = int((inst.F1.astype(int) + inst.F1.T).sum(1).max()) * int(inst.D.astype(int).sum(1).max())
    kw = dict(I_max=1500, seed=5, delta0=2.0 * w, deltaf=w / 500.0, xi=0.01)
    _, _, res, tr = gpu_run(inst, trace=True, replicas=replicas, **kw)
    rows = [0, replicas - 1]
    _, orc = oracle_run(inst, trace=True, replicas=rows, **kw)
    compare(res, rows, orc, n * n, gpu_trace=tr)
    assert res.stats[:, 7].sum() > 0  # some jumps rebuilt


# products from n = 29 up; a last block of 16 rows that is full, ragged or one
# row (n = 50, where a warp takes both halves of a strip, runs whole in
# test_gpu_warp.py)
@pytest.mark.parametrize("n,fmax,dmax", [
    (28, 99, 120), (29, 99, 120), (32, 99, 1023),   # whole entries of both
    (33, 400, 119),                                 # flows beyond a byte, whole
    (33, 900, 119), (33, 9000, 40),                 # flows in two bytes
    (33, 99, 1024),                                 # M in two bytes
    (29, 200, 32767), (32, 2000, 1500),             # 2 max d = 65,534; both in bytes
])
@pytest.mark.parametrize("replicas", [3, 320])
def test_matrix_products_over_the_value_ranges(n, fmax, dmax, replicas):
    rng = np.random.default_rng(n + fmax + dmax)
    F1, F2 = (rng.integers(0, fmax + 1, (n, n)) * (rng.random((n, n)) < 0.3) for _ in range(2))
    inst = _Inst(F1, F2, rng.integers(dmax // 2, dmax + 1, (n, n)))
    w = int((inst.F1.astype(int) + inst.F1.T).sum(1).max()) * int(inst.D.astype(int).sum(1).max())
    kw = dict(I_max=1500, seed=5, delta0=2.0 * w, deltaf=w / 500.0, xi=0.01)
    _, _, res, tr = gpu_run(inst, trace=True, replicas=replicas, **kw)
    rows = [0, replicas - 1]
    _, orc = oracle_run(inst, trace=True, replicas=rows, **kw)
    compare(res, rows, orc, n * n, gpu_trace=tr)
    # three replicas may have no jump to a member that accepts
    assert replicas == 3 or res.stats[:, 7].sum() > 0


# the widest tiling ends at 18 workers of 24 words: 432 words, n = 117
@pytest.mark.parametrize("n", [115, 116, 117, 118, 128])
@pytest.mark.parametrize("replicas", [2, 160])
def test_the_largest_sizes(n, replicas):
    inst = inputs.euclid_instance(n, 0.0, False, index=n, workload="BATCH")
    kw = dict(I_max=150, seed=n, delta0=2e7, deltaf=3e4, xi=0.05)
    _, _, res, tr = gpu_run(inst, trace=True, replicas=replicas, **kw)
    rows = [0, replicas - 1]
    _, orc = oracle_run(inst, trace=True, replicas=rows, **kw)
    compare(res, rows, orc, n * n, gpu_trace=tr)


@pytest.mark.parametrize("acc", ["strict", "lenient"])
@pytest.mark.parametrize("n,weights", [(41, None), (57, None), (9, (10 ** 12, 3))])
def test_delta_e_beyond_int32(n, weights, acc):
    """|Delta E_k| passes 2^31 while the state is dense and returns below it
    as the schedule cools (automatic weights); penalty weights far beyond
    32 bits keep the 64-bit form throughout."""
    rng = np.random.default_rng(n)
    F1, F2 = (rng.integers(300, 900, (n, n)) for _ in range(2))
    inst = _Inst(F1, F2, rng.integers(50, 120, (n, n)))
    kw = dict(replicas=2, I_max=2500, seed=3, accept=acc, w=weights, delta0=1e10, deltaf=1e6,
              xi=5e-3)
    _, _, res, tr = gpu_run(inst, trace=True, **kw)
    _, orc = oracle_run(inst, trace=True, **kw)
    compare(res, range(2), orc, n * n, gpu_trace=tr)


@pytest.mark.parametrize("name,n", [("dense", 100), ("sparse", 110)])
def test_large_instances(name, n):
    inst = inputs.euclid_instance(n, 0.0, name == "sparse", index=2, workload="P25")
    kw = dict(replicas=1, I_max=400, seed=1, **FAST)
    _, _, res, tr = gpu_run(inst, trace=True, **kw)
    _, orc = oracle_run(inst, trace=True, **kw)
    compare(res, range(1), orc, n * n, gpu_trace=tr)


def test_accept_every_draw():
    """Every table index, penalties inside and just outside the band that is
    left to the double test (2e-5 delta), and at the product itself."""
    from paper_2205_13399_gb300 import moda
    T = oracle.neglog_table()
    idx = np.arange(65536, dtype=np.uint32)
    for k, delta in enumerate((1.0e4, 3.7e6, 1.0e9)):
        prod = delta * T[idx]
        for off in (-1e-4, -2.1e-5, -1.9e-5, 0.0, 1.9e-5, 2.1e-5, 1e-4):
            a = np.maximum(np.floor(prod + off * delta), 0).astype(np.int64)
            acc, path = moda.check_accept(a, np.full(idx.size, delta), idx)
            assert np.array_equal(acc, a.astype(np.float64) <= prod), (k, off)
            if abs(off) < 2e-5 and delta > 1e6:
                assert (path == -1).all()


# the extensions: 12 one word a worker, 30 two, 40 four, 56 eight
@pytest.mark.parametrize("n", [3, 12, 30, 40, 56])
@pytest.mark.parametrize("esc", ["archive", "offset"])
@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("acc,arc", [("strict", "explore"), ("lenient", "exploit")])
def test_extensions_traced(n, esc, norm, acc, arc):
    if esc == "archive" and not norm:
        pytest.skip("the default algorithm")
    inst = inputs.uniform_instance(n, index=60 + n, workload="P8")
    kw = dict(replicas=2, I_max=900, seed=n, accept=acc, archive=arc, escape=esc, beta=30_000)
    # Sec. 4.2's units are larger: a schedule that reaches the frozen phase in both
    kw.update(dict(delta0=3e8, deltaf=1e6, xi=0.02) if norm else FAST)
    _, _, res, tr = gpu_run(inst, trace=True, normalize=norm, **kw)
    _, orc = oracle_run(inst, trace=True, normalize=norm, **kw)
    compare(res, range(2), orc, n * n, gpu_trace=tr)
    if esc == "offset" and n <= 30:  # (larger ones are still descending after 900 flips)
        assert res.stats[:, 3].sum() > 0


@pytest.mark.parametrize("esc", ["archive", "offset"])
@pytest.mark.parametrize("norm", [False, True])
def test_extensions_beyond_int32(esc, norm):
    if esc == "archive" and not norm:
        pytest.skip("the default algorithm")
    n = 41
    rng = np.random.default_rng(n)
    F1, F2 = (rng.integers(300, 900, (n, n)) for _ in range(2))
    inst = _Inst(F1, F2, rng.integers(50, 120, (n, n)))
    kw = dict(replicas=2, I_max=2500, seed=3, escape=esc, beta=4_000_000, delta0=1e10, deltaf=1e6,
              xi=5e-3)
    _, _, res, tr = gpu_run(inst, trace=True, normalize=norm, **kw)
    _, orc = oracle_run(inst, trace=True, normalize=norm, **kw)
    compare(res, range(2), orc, n * n, gpu_trace=tr)


@pytest.mark.parametrize("K", [1, 7, 250, 600])
@pytest.mark.parametrize("esc", ["archive", "offset"])
def test_snapshots(K, esc):
    """Snapshots at every spacing: after flips, inside runs of jumps, at the
    last iteration."""
    from paper_2205_13399_gb300 import moda
    n, R, I_max = 9, 2, 600
    inst = inputs.uniform_instance(n, index=5, workload="P8")
    kw = dict(replicas=R, I_max=I_max, seed=2, escape=esc, beta=2000, **FAST)
    g = moda.Instance(inst.F1, inst.F2, inst.D)
    run = moda.anneal(g, snapshot_every=K, **kw).wait()
    _, orc = oracle_run(inst, snapshot_every=K, **kw)
    snap = orc["snapshots"]
    for r in range(R):
        for j in range(0, I_max // K, max(1, I_max // K // 40)):
            c = int(snap["count"][r, j])
            E = snap["E"][r, j, :c]
            pts = [(int(a), int(b)) for a, b in E]
            want = sorted(pts[i] for i in oracle.nondominated(pts))
            got = run.read_archive(replica=r, snapshot=j)
            assert [(p["E1"], p["E2"]) for p in got] == want, (r, j)
            for p in got:
                slot = p["slot"]
                assert pts[slot] == (p["E1"], p["E2"])
                if p["perm"] is not None:
                    assert p["perm"] == oracle.decode_permutation(snap["bits"][r, j, slot])
    compare(run.read(), range(R), orc, n * n)
