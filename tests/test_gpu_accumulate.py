"""The sum of a batch's final angles at every gap site against 64 bits.

Angles spread over 30 powers of two take the sum's slow branch at some sites
(two floats don't hold it), angles of similar size the fast one. The prediction
is the mean angle's value of the field's range: it may differ from the 64-bit
mean of the stored angles by the rounding of a float of the range's size, 2^-24
of it, and by the float scaling's, the same again.
"""
import numpy as np
import pytest

from paper_2212_01317_gb300 import synth
from paper_2212_01317_gb300.mpr import GapFiller

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("R", [1, 2, 5, 33])
@pytest.mark.parametrize("powers", [1, 30])
def test_mean_angle(storage, R, powers):
    z, m = synth.small_problem(37, 51, 0.6, seed=R)
    v = np.where(m != 0, np.nan, z).astype(np.float32)
    rng = np.random.default_rng(storage + 10 * powers)
    gf = GapFiller(v, m, 8, seed=3, storage=storage)
    gf.set_temperatures(np.full(gf.nblk, 0.1, np.float32))
    mean, n = np.zeros(v.shape), 0
    for _ in range(2):                  # an odd R starts the second batch in a pair's middle
        gf.sim_begin(R)
        for r in range(R):
            a = 2 * np.pi * rng.random(v.shape) * 2.0 ** -rng.integers(0, powers, v.shape)
            gf.set_state(r, a.astype(np.float32))
        mean += sum(gf.get_state(r).astype(np.float64) for r in range(R))
        n += R
        gf.sim_end()
    out = gf.predict()[0]
    gf.close()
    lo, hi = float(np.nanmin(v)), float(np.nanmax(v))
    want = lo + (hi - lo) * mean / n / (2 * np.pi)
    gap = m != 0
    tol = 2 * 2.0 ** -24 * (abs(lo) + abs(hi) + (hi - lo))
    np.testing.assert_allclose(out[gap], want[gap], rtol=0, atol=tol)
