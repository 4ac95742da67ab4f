"""Precision of the CMBWS_FP64 transforms where one scale per block could lose bits: values far
below the largest one of their block still count with the accuracy that FP64 gives them."""
import math

import numpy as np
import pytest

import paper_1710_00621_gb300 as cw
from oracle import grids as og
from oracle import sht as osht
from tests._gpu import rel_err, to_dev, to_host

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("nside,lmax", [(16, 63), (64, 255), (64, 767), (256, 767)])
def test_low_multipoles_under_a_high_band_limit(nside, lmax):
    """The rescaled Legendre values of m = 0 grow with l, so a high band-limit leaves those of low l
    the fewest bits.  A monopole and a dipole in closed form, on the rings of 4 nside pixels (the
    shorter ones go through chirps): one rounding each, at most half a unit of the largest pixel, of
    the scaled coefficients, the dipole's Legendre value, the ring spectra of both parities, their
    sum, its fixed-point form and the pixel, with exact products between them: 4 units cover it.
    The adjoint of a constant map adds whole numbers."""
    g = cw.cmbws_plan_grid(cw.CMBWS_GRID_HEALPIX, nside, lmax)
    maps = 8
    alm = np.zeros((maps, (lmax + 1) ** 2))
    alm[:, :2] = np.random.default_rng(lmax).uniform(0.5, 2.0, (maps, 2))
    out = to_dev(np.zeros((maps, g.npix)))
    cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(alm), out, maps)
    full = np.repeat(g.nphi == 4 * nside, g.nphi)
    x = np.cos(g.theta.astype(np.longdouble))
    c = np.sqrt(1 / (4 * np.arccos(np.longdouble(-1))))
    for k in range(maps):
        want = c * (alm[k, 0] + alm[k, 1] * np.sqrt(np.longdouble(3)) * x)
        err = np.abs(to_host(out)[k] - np.repeat(want, g.nphi))[full] / np.abs(want).max()
        assert err.max() <= 4 * U, float(err.max() / U)
    back = to_dev(np.zeros((lmax + 1) ** 2))
    cw.cmbws_sht_analysis(g, cw.CMBWS_FP64, to_dev(np.ones(g.npix)), back, 1, 0)
    want = g.npix / math.sqrt(4.0 * math.pi)
    assert abs(to_host(back)[0] - want) <= 4 * U * want


@pytest.mark.parametrize("nside,lmax", [(16, 255), (16, 767), (1, 3000)])
def test_monopole_on_short_rings(nside, lmax):
    """Rings of far fewer pixels than the band-limit leave room for the sum of all aliases of a
    frequency, but the ring spectra keep their bits all the same: the bound above on every ring of a
    power-of-two length."""
    g = cw.cmbws_plan_grid(cw.CMBWS_GRID_HEALPIX, nside, lmax)
    maps = 8
    a = np.random.default_rng(lmax).uniform(0.5, 2.0, maps)
    alm = np.zeros((maps, (lmax + 1) ** 2))
    alm[:, 0] = a
    out = to_dev(np.zeros((maps, g.npix)))
    cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(alm), out, maps)
    pow2 = np.repeat(g.nphi & (g.nphi - 1) == 0, g.nphi)
    want = a / math.sqrt(4.0 * math.pi)
    err = np.abs(to_host(out)[:, pow2] - want[:, None]) / want[:, None]
    assert err.max() <= 4 * U, err.max() / U


@pytest.mark.parametrize("nside,lmax", [(1, 31), (1, 33), (1, 200), (3, 150)])
def test_aliases_on_short_rings(nside, lmax):
    """Full spectra on rings of 4 to 12 pixels, around the number of aliases from which the sums are
    formed twice: the FP64 parity bound 40 (L+1) u of the largest pixel."""
    g = cw.cmbws_plan_grid(cw.CMBWS_GRID_HEALPIX, nside, lmax)
    alm = np.random.default_rng(lmax).standard_normal((lmax + 1) ** 2)
    out = to_dev(np.zeros(g.npix))
    cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(alm), out, 1)
    want = osht.synthesis(og.healpix(nside), lmax, alm)
    assert rel_err(to_host(out), want) < 40 * (lmax + 1) * U


def _grid(kind, n, lmax):
    if kind == "healpix":
        return cw.cmbws_plan_grid(cw.CMBWS_GRID_HEALPIX, n, lmax), og.healpix(n)
    g = cw.cmbws_plan_grid(cw.CMBWS_GRID_GL, n, lmax)
    nphi = np.full(n, 2 * lmax + 1)
    return g, og.RingGrid("gl", n, g.theta, np.zeros(n), nphi, g.weight,
                          np.concatenate([[0], np.cumsum(nphi)]))


@pytest.mark.parametrize("kind,n,lmax", [("gl", 64, 63), ("gl", 131, 129), ("healpix", 16, 47)])
@pytest.mark.parametrize("amp", [1e3, 1e6, 1e10])
def test_bright_polar_pixel_per_order(kind, n, lmax, amp):
    """One pixel of the first ring far above unit noise aliases into every m, but its Legendre values
    at high m are tiny: the coefficients of each order are as accurate, relative to the largest of the
    order, as the FP64 parity bound 40 (L+1) u asks."""
    g, o = _grid(kind, n, lmax)
    f = np.random.default_rng(n).standard_normal(g.npix)
    f[0] = amp
    back = to_dev(np.zeros((lmax + 1) ** 2))
    cw.cmbws_sht_analysis(g, cw.CMBWS_FP64, to_dev(f), back, 1, 0)
    got, want = to_host(back), osht.adjoint(o, lmax, f)
    for m in range(lmax + 1):
        a, b = (np.concatenate(osht.packed_m(v, lmax, m)) for v in (got, want))
        assert rel_err(a, b) < 40 * (lmax + 1) * U, m


@pytest.mark.parametrize("kind,n,lmax,m", [("gl", 64, 63, 16), ("gl", 131, 129, 60), ("gl", 131, 129, 129),
                                           ("healpix", 16, 47, 20)])
def test_dark_rings_of_one_order(kind, n, lmax, m):
    """Coefficients of a single high order leave rings near the poles dark: each ring is as accurate,
    relative to its own largest pixel, as the FP64 parity bound asks.  Walks start where the Legendre
    values pass 1e-30, so L + 1 terms of coefficients up to 3 below that are left out on every path; on
    rings brighter than 3e-30 / (40 u) = 7e-16 they are within the bound."""
    g, o = _grid(kind, n, lmax)
    alm = np.zeros((lmax + 1) ** 2)
    i = (lmax + 1) + (m - 1) * (2 * lmax + 2 - m)
    k = lmax - m + 1
    alm[i:i + 2 * k] = np.random.default_rng(m).standard_normal(2 * k)
    out = to_dev(np.zeros(g.npix))
    cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(alm), out, 1)
    got, want = to_host(out), osht.synthesis(o, lmax, alm)
    for r in range(g.nring):
        s = slice(int(o.offset[r]), int(o.offset[r + 1]))
        if np.abs(want[s]).max() > 7e-16:
            assert rel_err(got[s], want[s]) < 40 * (lmax + 1) * U, r


@pytest.mark.parametrize("kind,n,lmax,m", [("gl", 64, 63, 16), ("gl", 131, 129, 60), ("gl", 300, 280, 100),
                                           ("healpix", 16, 47, 20)])
@pytest.mark.parametrize("shape", ["step", "power"])
def test_steep_orders(kind, n, lmax, m, shape):
    """A spectrum of one order that falls by 1e10 within a few l, or as l^-40: rings near the poles only
    see the small coefficients, and keep the FP64 parity bound relative to their own largest pixel.
    The terms below the 1e-30 at which walks start are at most 8 (step) or L + 1 (power) of 3e10: 3e-20 (L + 1)
    in all, within the bound on rings brighter than 7e-6.  Maps of the same call that are not
    steep come out as in a call of their own."""
    g, o = _grid(kind, n, lmax)
    rng = np.random.default_rng(m)
    i, k = (lmax + 1) + (m - 1) * (2 * lmax + 2 - m), lmax - m + 1
    l = np.arange(m, lmax + 1)
    fall = np.where(l < m + 8, 1e10, 1.0) if shape == "step" else 1e10 * (l / m) ** -40.0
    alm = rng.standard_normal((3, (lmax + 1) ** 2))
    alm[1] = 0.0
    alm[1, i:i + 2 * k] = rng.standard_normal(2 * k) * np.concatenate([fall, fall])
    out = to_dev(np.zeros((3, g.npix)))
    cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(alm), out, 3)
    got, want = to_host(out), osht.synthesis(o, lmax, alm[1])
    for r in range(g.nring):
        s = slice(int(o.offset[r]), int(o.offset[r + 1]))
        if np.abs(want[s]).max() > 7e-6:
            assert rel_err(got[1][s], want[s]) < 40 * (lmax + 1) * U, r
    for j in range(3):
        one = to_dev(np.zeros((1, g.npix)))
        cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(alm[j:j + 1]), one, 1)
        assert np.array_equal(to_host(one)[0], got[j])
