"""Box means of the site temperatures in runs of outputs against plain sums in
64 bits: radii at which the form changes (3 | 4, 7 | 8, beyond 1024), windows
wider than the field, widths and heights that are no multiple of a run, and
fields side by side whose boundary falls inside a run. Sums in FP64 of at most
a few thousand positive terms, rounded to float once: 2^-24 relative, and 1e-12
for the sums.
"""
import numpy as np
import pytest

from paper_2212_01317_gb300 import mpr, synth
from paper_2212_01317_gb300.mpr import BatchFiller, GapFiller

pytestmark = pytest.mark.gpu


def _smooth(T, h, w, lb, r, n):
    e = np.repeat(np.repeat(T.astype(np.float64).reshape(-(-h // lb), -(-w // lb)), lb, 0), lb, 1)[:h, :w]
    for _ in range(n):
        for ax, size in ((1, w), (0, h)):
            at = np.clip(np.arange(size)[:, None] + np.arange(-r, r + 1)[None], 0, size - 1)
            e = np.take(e, at, axis=ax).mean(axis=ax + 1)
    return e


@pytest.mark.parametrize("h,w,lb", [(75, 1043, 8), (16, 16, 8), (130, 7, 4), (33, 70, 16)])
@pytest.mark.parametrize("r", [1, 3, 4, 7, 8, 16, 40, 1025])
def test_box_means(h, w, lb, r):
    if r > 100 and h * w > 20000:
        pytest.skip("the reference's window table would be large")
    z, m = synth.small_problem(h, w, 0.4, seed=r)
    gf = GapFiller(np.where(m != 0, np.nan, z).astype(np.float32), m, lb, seed=1)
    T = np.random.default_rng(r).uniform(0.01, 1.0, gf.nblk).astype(np.float32)
    gf.set_temperatures(T)
    got = gf.smooth_temperatures(r, 2)
    gf.close()
    np.testing.assert_allclose(got, _smooth(T, h, w, lb, r, 2), rtol=2.0 ** -24 + 1e-12)


@pytest.mark.parametrize("r", [3, 6, 16])
def test_box_means_of_a_batch(r):
    shapes = [(31, 21), (24, 50), (9, 40)]
    zs, ms = zip(*(synth.small_problem(h, w, 0.5, seed=h) for h, w in shapes))
    vs = [np.where(m != 0, np.nan, z).astype(np.float32) for z, m in zip(zs, ms)]
    bf = BatchFiller(vs, list(ms), 8, seed=5)
    H, W, nby, nbx = bf.info.height, bf.info.width, bf.info.nby, bf.info.nbx
    T = np.random.default_rng(r).uniform(0.01, 1.0, (nby, nbx)).astype(np.float32)
    bf.set_temperatures(T.ravel())
    got = np.zeros((H, W), np.float32)
    mpr.mpr_smooth_temperatures(bf.ctx, r, 2, got)
    layout = bf.layout
    bf.close()
    for y, x, h, w in layout:
        t = T[y // 8:y // 8 - (-h // 8), x // 8:x // 8 - (-w // 8)]
        np.testing.assert_allclose(got[y:y + h, x:x + w], _smooth(t.ravel(), h, w, 8, r, 2),
                                   rtol=2.0 ** -24 + 1e-12)
