"""The offset escape where E_off is far above the temperature: Delta E - E_off
then loses as much as the whole range of the draws to float rounding, and the
kernels with inline draws (four and more words a worker: n = 40, and n = 12 on
a crowded device) must still hand such bits to the double test.  Two objectives
whose costs are zero or a single pair, so that every bit of a permutation costs
the penalty weight, and weights, beta and delta such that the offset reached
lies within the draws' range below that weight, on the other side of a rounding
boundary of float."""
import numpy as np
import pytest

from parity import compare, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


class _Inst:
    def __init__(self, n, cmax):
        F = np.zeros((n, n), np.int16)
        self.F1, self.F2, self.D, self.n = F.copy(), F.copy(), F.copy(), n
        if cmax:  # largest cost coefficient, the unit of the normalisation
            self.F1[0, 1] = cmax
            self.D[0, 1] = self.D[1, 0] = 1


@pytest.mark.parametrize("n,replicas", [(40, 2), (12, 2000)])
@pytest.mark.parametrize("w,beta,delta,cmax", [
    # E_off = 4 beta = 2^30 + 60 (float 2^30), Delta E = 2^30 + 68 (2^30 + 128),
    # delta T_max = 94
    (2 ** 30 + 68, 268435471, 8.0, 0),
    # 2 beta = 2^26 + 2 (2^26), 2^26 + 5 (2^26 + 8), 7.1
    (2 ** 26 + 5, 33554433, 0.6, 0),
    # normalised: s = 2^23 / 3, s Delta E = 111,848,106.67 (111,848,110 with s in
    # float), 2 beta = 111,848,106 (111,848,104), 4.7
    (40, 55924053, 0.4, 3),
])
def test_offsets_far_above_the_temperature(n, replicas, w, beta, delta, cmax):
    inst = _Inst(n, cmax)
    kw = dict(I_max=4000, seed=n, escape="offset", beta=beta, delta0=delta, deltaf=delta, xi=0.5,
              w=(w, 0), normalize=cmax > 0, archive_size=4)
    _, _, res, tr = gpu_run(inst, trace=True, replicas=replicas, **kw)
    rows = [0, replicas - 1]
    _, orc = oracle_run(inst, trace=True, replicas=rows, **kw)
    assert all(r[3] > 20 for r in orc["stats"])  # raises
    compare(res, rows, orc, n * n, gpu_trace=tr)
