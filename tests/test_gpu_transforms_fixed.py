"""The fixed-point transforms against the DFT in extended precision: every azimuthal size, ragged
columns, columns of very different magnitude, zeros, infinities and NaN."""
import numpy as np
import pytest
import torch

from paper_2609_07172_gb300 import Plan, workloads as W

pytestmark = pytest.mark.gpu
L = np.longdouble


def _dft(x):
    nt = x.shape[1]
    nm = nt // 2 + 1
    th = 2 * np.arccos(L(-1)) * ((np.arange(nt)[:, None] * np.arange(nm)[None, :]) % nt) / nt
    c, s = np.cos(th), np.sin(th)
    re, im = np.einsum("kji,jm->kim", x.astype(L), c) / nt, -np.einsum("kji,jm->kim", x.astype(L), s) / nt
    im[..., 0] = im[..., -1] = 0
    return re, im, c, s


@pytest.mark.parametrize("nt", [2, 4, 8, 16, 32, 64, 128, 256])
@pytest.mark.parametrize("nr,nz", [(1, 3), (31, 2), (33, 2), (64, 1)])
def test_transforms_match_extended_precision(nt, nr, nz):
    p = W.annulus(nr, nt, nz)
    rng = np.random.default_rng(nt + nr)
    x = rng.standard_normal(p.shape) * 10.0 ** rng.uniform(-12, 12, (nz, 1, nr))   # columns apart by 24 decades
    x[:, rng.integers(nt), :] *= 1e3
    x[0, :, 0] = 0.0
    re, im, c, s = _dft(x)
    with Plan(p) as plan:
        u = plan.analyze(torch.from_numpy(x).cuda()).cpu().numpy()
        col = np.sqrt((re ** 2 + im ** 2).sum(-1))
        err = np.sqrt((u[..., 0] - re) ** 2 + (u[..., 1] - im) ** 2)
        # a unit is at most 2^-61 of the column's sum of magnitudes (<= sqrt(nt) times its norm sqrt(nt) col),
        # log2(nt) + 2 cuts of one unit per path, and one binary64 rounding of the result
        tol = (2.0 ** -53 + (np.log2(nt) + 2) * nt * 2.0 ** -61)
        assert np.all(err <= 2 * tol * col[..., None])
        assert np.all(u[0, 0] == 0.0)
        v = np.stack([re.astype(float), im.astype(float)], -1)
        v[..., 0, 1] = v[..., -1, 1] = np.nan                                     # not read
        phi = plan.inverse(torch.from_numpy(v).cuda()).cpu().numpy()
    w = np.full(nt // 2 + 1, L(2))
    w[0] = w[-1] = 1
    v[..., 0, 1] = v[..., -1, 1] = 0.0
    ref = np.einsum("kim,jm->kji", v[..., 0] * w, c) - np.einsum("kim,jm->kji", v[..., 1] * w, s)
    # column by column no further from the sum than binary64 rounding of its input and result plus
    # a binary64 transform are (the root mean square of log2(nt) + 1 rounded additions per value)
    err, norm = [np.sqrt((t.astype(L) ** 2).sum(1)) for t in (phi - ref, ref)]
    assert np.all(err <= 2.0 ** -53 * np.sqrt(np.log2(nt) + 1) * norm + (norm == 0))


def test_non_finite_columns_come_out_as_nan_and_leave_the_others_alone():
    p = W.annulus(40, 16, 3)
    x = np.random.default_rng(1).standard_normal(p.shape)
    y = x.copy()
    y[1, 3, 7], y[2, 0, 33] = np.inf, np.nan
    with Plan(p) as plan:
        a, b = [plan.analyze(torch.from_numpy(t).cuda()).cpu().numpy() for t in (x, y)]
        fa, fb = [plan.inverse(torch.from_numpy(np.where(bad, np.nan, a)).cuda()).cpu().numpy()
                  for bad in (False, np.arange(40)[None, :, None, None] == 5)]
    hit = np.zeros((3, 40), dtype=bool)
    hit[1, 7] = hit[2, 33] = True
    assert np.isnan(b[hit][:, :, 0]).all() and np.array_equal(a[~hit], b[~hit])
    assert np.isnan(fb[:, :, 5]).all() and np.array_equal(np.delete(fa, 5, 2), np.delete(fb, 5, 2))


def test_scales_at_the_ends_of_the_range():
    p = W.annulus(8, 32, 2)
    x = np.random.default_rng(2).standard_normal(p.shape)
    with Plan(p) as plan:
        ref = plan.analyze(torch.from_numpy(x).cuda()).cpu().numpy()
        for e in (-960, -500, 500, 960):
            got = plan.analyze(torch.from_numpy(np.ldexp(x, e)).cuda()).cpu().numpy()
            assert np.array_equal(got, np.ldexp(ref, e))
