"""3-D half-step: how the list is cut into runs of chunks, and how many pairs
share a launch, must not show in the results.

A launch of many pairs gives each warp several 32-entry chunks and sums block
changes in FP64; few pairs mean one chunk per warp. The random numbers belong to
the realization, so the same realizations in batches of different sizes are the
same chains: predictions may differ by the order of FP64 sums only (1e-12 of the
range for at most ten terms), far below the float32 step of 6e-8 relative that a
prediction is rounded to; 1e-6 of the range allows for that rounding.
"""
import numpy as np
import pytest

from paper_2212_01317_gb300.mpr import GapFiller3

pytestmark = pytest.mark.gpu


def _cube(shape, p, seed):
    rng = np.random.default_rng(seed)
    z = rng.standard_normal(shape).astype(np.float32)
    for axis in range(3):
        z = (z + np.roll(z, 1, axis) + np.roll(z, -1, axis)) / 3.0
    m = (rng.random(shape) < p).astype(np.uint8)
    m[0, 0, :2] = 0
    return z.astype(np.float32), m


# 64^3 at half the sites missing: 4096 chunks per colour, two chunks per warp
# from five pairs on; odd sides leave blocks, rows and the last chunk partial.
@pytest.mark.parametrize("shape,lb,p,batches", [
    ((64, 64, 64), 16, 0.5, (4, 6)),
    ((67, 61, 59), 16, 0.6, (4, 6)),
    ((67, 61, 59), 7, 0.9, (4, 8)),
    ((1, 9, 5), 3, 0.4, (4, 4)),
])
def test_batch_sizes_agree(shape, lb, p, batches):
    z, m = _cube(shape, p, 5)
    preds = []
    for split in (batches, (sum(batches),)):
        f = GapFiller3(np.where(m != 0, np.nan, z), m, lb, seed=77, n_max=30)
        T = np.random.default_rng(1).uniform(0.02, 0.3, f.nblk).astype(np.float32)
        f.set_temperatures(T)
        for n in split:
            f.simulate(n)
        preds.append((f.predict()[0], f.refresh().gap_updates))
        f.close()
    span = float(np.ptp(z[m == 0]))
    assert preds[0][1] == preds[1][1]
    assert np.abs(preds[0][0] - preds[1][0]).max() <= 1e-6 * span
