"""Fronts read by their several ways (few members in all, one archive, many)
against the raw archives of the same run."""
import numpy as np
import pytest

import oracle
from paper_2205_13399_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,replicas,archive_size", [
    (3, 2, 0), (8, 4, 0), (8, 32, 0),          # up to 512 members, and beyond
    (20, 2, 1), (20, 512, 1), (20, 513, 1),    # the edge of it
    (45, 1, 0), (25, 40, 0)])
def test_fronts_equal_the_filter_of_the_archives(n, replicas, archive_size):
    from paper_2205_13399_gb300 import moda
    qi = inputs.uniform_instance(n, index=n, workload="P8")
    g = moda.Instance(qi.F1, qi.F2, qi.D)
    run = moda.anneal(g, replicas=replicas, I_max=3000, seed=5, delta0=2e6, deltaf=3e3, xi=0.01,
                      archive_size=archive_size).wait()
    res = run.read()
    for rows, which in ((range(replicas), -1), ([replicas - 1], replicas - 1)):
        where = [(r, k) for r in rows for k in range(int(res.count[r]))]
        pts = [tuple(int(v) for v in res.E[r, k]) for r, k in where]
        want = sorted((pts[i],) + where[i] for i in oracle.nondominated(pts))
        got = run.read_archive(which)
        assert [((p["E1"], p["E2"]), p["replica"], p["slot"]) for p in got] == want
        for p in got:
            bits = moda.unpack_bits(res.bits[p["replica"], p["slot"]], n * n).reshape(n, n)
            ok = (bits.sum(0) == 1).all() and (bits.sum(1) == 1).all()
            assert p["feasible"] == ok
            assert p["perm"] == (bits.argmax(1).tolist() if ok else None)
            assert p["g"] == int(((1 - bits.astype(np.int64).sum(1)) ** 2).sum()
                                 + ((1 - bits.astype(np.int64).sum(0)) ** 2).sum())
