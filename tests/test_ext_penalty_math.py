"""The float form of the acceptance penalty s Delta E - E_off (normalisation and
the offset escape) against its definition in IEEE double, evaluated on the host
in float32 as the device does: a penalty within delta T_max, which some draw
accepts, never passes (1 + 2e-6) delta T_max + 1e-6 E_off, the bound above which
a chunk of bits is left out of a trial.  Without the second term it does."""
import numpy as np

import oracle

F = np.float32


def _both(s, dE, off):
    """(double, float): the product of two floats is exact in double, and one
    rounding to float follows the difference, as in a fused operation."""
    exact = np.maximum(s * dE - off, 0.0)
    fl = F(F(s).astype(np.float64) * F(dE).astype(np.float64) - F(off).astype(np.float64))
    return exact, np.maximum(fl, F(0))


def _bounds(delta, off):
    top = delta * oracle.neglog_table()[0]
    hi = F(F(top) * F(1 + 2e-6))
    return top, hi, F(hi + F(1e-6) * F(off))


def test_penalties_at_the_cooled_end_of_the_schedule():
    """Two of a sweep over largest coefficients, at the first delta <= 10^4 of
    the default schedule, E_off a multiple of beta = 40,960."""
    delta = 1e9
    while delta > 1e4:
        delta *= 1.0 - 1e-3
    for cmax, off, dE in ((8059, 37724160, 36355), (8033, 68730880, 65930)):
        exact, fl = _both(np.float64(2.0 ** 23 / cmax), np.float64(dE), np.float64(off))
        top, hi, lim = _bounds(delta, off)
        assert exact <= top and fl > hi and fl <= lim


def test_no_accepted_penalty_passes_the_bound():
    rng = np.random.default_rng(3)
    n = 400_000
    delta = 10.0 ** rng.uniform(-1, 9, n)
    off = np.floor(10.0 ** rng.uniform(0, 13, n))
    s = np.where(rng.random(n) < 0.5, 1.0, 2.0 ** 23 / rng.integers(1, 2 ** 31, n))
    top, hi, lim = _bounds(delta, off)
    # integers Delta E whose penalty is at or just below delta T_max
    dE = np.floor((off + top * rng.choice([0.0, 0.5, 0.999, 1.0], n)) / s)
    keep = np.abs(dE) < 2.0 ** 40
    exact, fl = _both(s, dE, off)
    some = keep & (exact <= top)
    assert some.sum() > n // 4
    assert np.all(fl[some] <= lim[some])
    assert np.any(fl[some] > hi[some])
