"""Setting a field up: the sample angles against the FP64 transform, and the
statistics of inputs that the wide loads cannot take.

Sample angles (Sec. 2.1) are 2 pi (z - zmin) / (zmax - zmin) in FP64, rounded to
FP32, exactly: the library multiplies by a precomputed scale and divides only
where the product lies too close to the middle of two floats to tell.
"""
import numpy as np
import pytest

import oracle
from paper_2212_01317_gb300 import mpr
from paper_2212_01317_gb300.mpr import BatchFiller, GapFiller

pytestmark = pytest.mark.gpu


def _angles(z, m):
    s = z[m == 0].astype(np.float64)
    lo, hi = s.min(), s.max()
    if not hi > lo:
        return np.zeros(z.shape, np.float32)
    return (2.0 * np.pi * (z.astype(np.float64) - lo) / (hi - lo)).astype(np.float32)


# values whose scaled offsets fall on float midpoints as often as possible:
# halves, thirds and tiny steps of the range, large offsets, a constant field
@pytest.mark.parametrize("values", ["normal", "grid", "offset", "tiny", "constant"])
@pytest.mark.parametrize("h,w,lb", [(301, 299, 16), (64, 64, 8), (5, 3, 4), (40, 700, 64)])
def test_sample_angles_are_the_fp64_transform(values, h, w, lb):
    rng = np.random.default_rng(h * w)
    z = {"normal": rng.standard_normal((h, w)),
         "grid": rng.integers(0, 3 * 2**10, (h, w)) / 3.0,
         "offset": 1e6 + rng.standard_normal((h, w)),
         "tiny": 1e-38 * rng.random((h, w)),
         "constant": np.full((h, w), 2.5)}[values].astype(np.float32)
    m = (rng.random((h, w)) < 0.5).astype(np.uint8)
    m[0, :2] = 0
    gf = GapFiller(np.where(m != 0, np.nan, z), m, lb, seed=1)
    gf.set_temperatures(np.full(gf.nblk, 0.1, np.float32))
    gf.sim_begin(1)
    got = gf.get_state(0)
    gf.close()
    np.testing.assert_array_equal(got[m == 0].view(np.uint32), _angles(z, m)[m == 0].view(np.uint32))


def _check_stats(got, z, m, lb):
    o = oracle.Oracle(z.shape[0], z.shape[1], lb)
    phi, *_ = o.transform(z, m)
    st = o.block_stats(phi, m)
    Es, Nsp, Nb, ng = got
    np.testing.assert_array_equal(Nsp, st.Nsp)
    np.testing.assert_array_equal(Nb, st.Nb)
    np.testing.assert_array_equal(ng, st.n_gap)
    np.testing.assert_allclose(Es, st.Es, rtol=1e-12, atol=1e-12)


# base addresses off the 16-byte grid, sizes off the 16-site grid, few and many
# blocks (256 and 128 threads per block), blocks of one site and of a whole field
@pytest.mark.parametrize("h,w,lb,shift", [(33, 31, 8, 1), (64, 64, 64, 3), (257, 130, 3, 0),
                                          (16, 16, 1, 2), (1, 37, 5, 1)])
def test_statistics_of_unaligned_inputs(h, w, lb, shift):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(h + w)
    z = rng.standard_normal((h, w)).astype(np.float32)
    m = (rng.random((h, w)) < 0.4).astype(np.uint8)
    m[0, :2] = 0
    v = torch.zeros(h * w + shift, device="cuda")
    k = torch.zeros(h * w + shift, dtype=torch.uint8, device="cuda")
    v[shift:] = torch.from_numpy(z).reshape(-1).cuda()
    k[shift:] = torch.from_numpy(m * 7).reshape(-1).cuda()
    n = -(-h // lb) * -(-w // lb)
    Es, zr = (torch.zeros(x, dtype=torch.float64, device="cuda") for x in (n, 2))
    Nsp, Nb, ng = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(3))
    mean = torch.zeros(n, device="cuda")
    assert mpr.mpr_block_stats_noalloc(h, w, lb, k[shift:], v[shift:], Es, Nsp, Nb, mean, ng, zr) == 0
    _check_stats([x.cpu().numpy() for x in (Es, Nsp, Nb, ng)], z, m, lb)
    assert zr.cpu().numpy().tolist() == [float(z[m == 0].min()), float(z[m == 0].max())]


def test_batch_fields_keep_their_own_ranges():
    rng = np.random.default_rng(4)
    shapes = [(37, 19), (8, 8), (50, 61)]
    zs = [(10.0 ** k * rng.standard_normal(s)).astype(np.float32) for k, s in enumerate(shapes)]
    ms = [(rng.random(s) < 0.5).astype(np.uint8) for s in shapes]
    for m in ms:
        m[0, :2] = 0
    bf = BatchFiller([np.where(m != 0, np.nan, z) for z, m in zip(zs, ms)], ms, 8, seed=2)
    n = bf.info.nblk
    Es, Nsp, Nb, ng = np.zeros(n), *(np.zeros(n, np.int32) for _ in range(3))
    mpr.mpr_get_block_stats(bf.ctx, Es, Nsp, Nb, None, ng)
    for k, (z, m) in enumerate(zip(zs, ms)):
        _check_stats([bf.block_slice(k, x) for x in (Es, Nsp, Nb, ng)], z, m, 8)
    bf.close()
