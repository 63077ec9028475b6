"""Calibration of small fields, one cluster per realization pair against the
launch-per-half-step form on the same chains.

cal_sweep = 1 forces the launch per half-step; the automatic choice takes the
cluster form up to 8192 gap sites per colour. Both run the same moves on the
same random numbers; the block energies differ only in how changes are summed
(FP32 warp sums against error-free sums). A bracket step compares a mean energy
with e_s, and a bracket decides differently only if the two lie within that
rounding, about 1e-8 of a unit against spreads of 1e-2: less than 1e-6 per
decision, so over the few thousand decisions below the temperatures are equal.
"""
import numpy as np
import pytest

from paper_2212_01317_gb300 import synth
from paper_2212_01317_gb300.mpr import BatchFiller, GapFiller

pytestmark = pytest.mark.gpu


def _temperatures(z, m, lb, **opts):
    v = np.where(m != 0, np.nan, z).astype(np.float32)
    out = []
    for form in (0, 1):
        gf = GapFiller(v, m, lb, seed=31, n_bisect=6, n_eq=5, n_meas=4, cal_sweep=form, **opts)
        out.append(gf.calibrate())
        gf.close()
    return out


# one site per thread: fields at the limit (8192 gap sites of a colour: 128 x 128
# all but one pair missing), just past it, tiny, odd and one row high
@pytest.mark.parametrize("h,w,lb,p", [(128, 128, 8, 0.999), (130, 130, 16, 0.999),
                                      (7, 5, 2, 0.5), (61, 45, 7, 0.6), (1, 40, 8, 0.4),
                                      (90, 33, 64, 0.3)])
@pytest.mark.parametrize("opts", [{}, {"cal_points": 2}, {"cal_points": 4, "cal_chains": 3},
                                  {"cal_chains": 3, "init": 1}, {"cal_points": 2, "q": 0.37}])
def test_cluster_form_equals_launch_form(h, w, lb, p, opts):
    z, _ = synth.small_problem(h, w, 0.5, seed=h * w)
    m = (np.random.default_rng(h + w).random((h, w)) < p).astype(np.uint8)
    m[0, :2] = 0
    a, b = _temperatures(z, m, lb, **opts)
    np.testing.assert_array_equal(a, b)


def test_cluster_form_of_a_batch():
    zs, ms = zip(*(synth.small_problem(h, w, 0.5, seed=h) for h, w in ((31, 20), (24, 24), (9, 40))))
    vs = [np.where(m != 0, np.nan, z).astype(np.float32) for z, m in zip(zs, ms)]
    got = []
    for form in (0, 1):
        bf = BatchFiller(vs, list(ms), 8, seed=5, n_bisect=5, n_eq=4, n_meas=3, cal_points=2,
                         cal_sweep=form)
        got.append(bf.calibrate())
        bf.close()
    np.testing.assert_array_equal(got[0], got[1])
