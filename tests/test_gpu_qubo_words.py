"""Explicit QUBOs at the edges of the kernel's tilings: one and several
words, four and eight words a worker, ragged last words, int32 and int64
Delta E, records and rebuilds -- traces against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,m,mag", [
    (1, 1, 60), (2, 31, 60), (3, 33, 60), (3, 128, 60), (1, 129, 60), (2, 300, 60),
    (2, 64, 2 ** 30), (3, 130, 2 ** 28),  # |Delta E| beyond 2^30
])
@pytest.mark.parametrize("acc,arc,esc", [("strict", "explore", "archive"),
                                         ("lenient", "exploit", "archive"),
                                         ("lenient", "explore", "offset")])
@pytest.mark.parametrize("cache", ["auto", "off"])
def test_tilings(K, m, mag, acc, arc, esc, cache):
    from paper_2205_13399_gb300 import moda
    rng = np.random.default_rng(m + K)
    Q = rng.integers(-mag, mag, (K, m, m)).astype(np.int32)
    Q = np.triu(Q)
    kw = dict(replicas=2, I_max=700, seed=m, accept=acc, archive=arc, escape=esc,
              beta=max(1, mag // 3), delta0=50.0 * mag, deltaf=mag / 12.0, xi=0.02)
    res = moda.Qubo(Q).anneal(trace=True, field_cache=cache, **kw).wait().read(trace=True)
    orc = oracle.kqubo_run(oracle.KQubo(Q), trace=True, **kw)
    assert np.array_equal(res["trace"], orc["trace"])
    assert np.array_equal(res["count"], orc["count"])
    for r in range(2):
        c = int(res["count"][r])
        assert np.array_equal(res["E"][r, :c], orc["E"][r, :c])
        assert np.array_equal(moda.unpack_bits(res["bits"][r, :c], m), orc["bits"][r, :c])
    assert np.array_equal(moda.unpack_bits(res["x"], m), orc["x"])
    assert np.array_equal(res["stats"], orc["stats"])


def test_eight_words_a_worker():
    """m = 2,850: 90 state words, eight a worker; two objectives against the
    oracle over a short run."""
    from paper_2205_13399_gb300 import moda
    rng = np.random.default_rng(8)
    Q = np.triu(rng.integers(-20, 20, (2, 2850, 2850)).astype(np.int32))
    kw = dict(replicas=1, I_max=150, seed=4, delta0=2e4, deltaf=50.0, xi=0.05)
    res = moda.Qubo(Q).anneal(trace=True, **kw).wait().read(trace=True)
    orc = oracle.kqubo_run(oracle.KQubo(Q), trace=True, **kw)
    assert np.array_equal(res["trace"], orc["trace"])
    assert np.array_equal(res["stats"], orc["stats"])


@pytest.mark.parametrize("m", [140, 300, 530])
@pytest.mark.parametrize("arc", ["explore", "exploit"])
def test_shared_archive_scan(m, arc):
    """Archives of more than 128 slots: one to three helpers share the scan."""
    from paper_2205_13399_gb300 import moda
    rng = np.random.default_rng(m)
    Q = np.triu(rng.integers(-60, 60, (3, m, m)).astype(np.int32))
    kw = dict(replicas=2, I_max=1200, seed=m, archive=arc, delta0=2e4, deltaf=20.0, xi=0.01)
    res = moda.Qubo(Q).anneal(trace=True, **kw).wait().read(trace=True)
    orc = oracle.kqubo_run(oracle.KQubo(Q), trace=True, **kw)
    assert np.array_equal(res["trace"], orc["trace"])
    assert np.array_equal(res["count"], orc["count"])
    for r in range(2):
        c = int(res["count"][r])
        assert np.array_equal(res["E"][r, :c], orc["E"][r, :c])
        assert np.array_equal(moda.unpack_bits(res["bits"][r, :c], m), orc["bits"][r, :c])


@pytest.mark.parametrize("K,m,mag", [(1, 96, 50), (2, 200, 50), (3, 130, 50), (1, 257, 2 ** 29),
                                     (3, 70, 2 ** 29), (2, 2850, 8)])
def test_rebuilds_of_landings(K, m, mag):
    """Records off at a temperature at which most jumps land on members that may
    accept: Delta E from the rows of the set bits, one to four at a time, words
    with a ragged number of them."""
    from paper_2205_13399_gb300 import moda
    rng = np.random.default_rng(7 * m + K)
    Q = np.triu(rng.integers(-mag, mag, (K, m, m)).astype(np.int32))
    kw = dict(replicas=2, I_max=400 if m < 1000 else 120, seed=m, delta0=100.0 * mag * K,
              deltaf=mag * 1.5, xi=0.03 if m < 1000 else 0.1)
    res = moda.Qubo(Q).anneal(trace=True, field_cache="off", **kw).wait().read(trace=True)
    orc = oracle.kqubo_run(oracle.KQubo(Q), trace=True, **kw)
    assert np.array_equal(res["trace"], orc["trace"])
    assert np.array_equal(moda.unpack_bits(res["x"], m), orc["x"])
    assert np.array_equal(res["stats"], orc["stats"])
