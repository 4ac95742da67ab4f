"""The fixed-point tensor-core Legendre stage of CMBWS_FP64 at the edges of its tiles: ring pairs
around 32 and 128, band-limits around the stages and chunks of 8, 16 and 128 values of l, one to
five maps, powers of two far from one, and coefficients that are not finite.

Tolerance: the FP64 parity bound of test_gpu_sht.py, 40 (L+1) eps64 of the largest output (floor
1e-14); the fixed-point stage's own error is below 2^-47 of it at these sizes."""
import numpy as np
import pytest

import paper_1710_00621_gb300 as cw
from oracle import grids as og
from oracle import sht as osht
from tests._gpu import rel_err, to_dev, to_host

pytestmark = pytest.mark.gpu


def _tol(lmax):
    return max(1e-14, 40 * (lmax + 1) * 2.0 ** -53)


# (rings, lmax, maps)
CASES = [(1, 0, 1), (2, 1, 2), (17, 15, 1), (64, 16, 3), (65, 17, 4), (66, 31, 5), (255, 32, 2),
         (256, 33, 1), (257, 47, 3), (259, 64, 4), (130, 127, 3), (129, 128, 2), (131, 129, 1)]


@pytest.mark.parametrize("n,lmax,maps,scale", [(*c, 1.0) for c in CASES]
                         + [(66, 31, 5, 2.0 ** -600), (131, 129, 1, 2.0 ** 600)])
def test_tile_edges(n, lmax, maps, scale):
    g = cw.cmbws_plan_grid(cw.CMBWS_GRID_GL, n, lmax)
    nphi = np.full(n, 2 * lmax + 1)
    o = og.RingGrid("gl", n, g.theta, np.zeros(n), nphi, g.weight,
                    np.concatenate([[0], np.cumsum(nphi)]))
    rng = np.random.default_rng(n + 1000 * lmax)
    alm = scale * rng.standard_normal((maps, (lmax + 1) ** 2)) * 10.0 ** rng.uniform(-3, 3, (maps, 1))
    out = to_dev(np.zeros((maps, g.npix)))
    cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(alm), out, maps)
    f = scale * rng.standard_normal((maps, g.npix))
    back = to_dev(np.zeros((maps, (lmax + 1) ** 2)))
    cw.cmbws_sht_analysis(g, cw.CMBWS_FP64, to_dev(f), back, maps, 0)
    m, a = to_host(out), to_host(back)
    for k in range(maps):
        assert rel_err(m[k] / scale, osht.synthesis(o, lmax, alm[k] / scale)) < _tol(lmax)
        assert rel_err(a[k] / scale, osht.adjoint(o, lmax, f[k] / scale)) < _tol(lmax)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite_stays_in_its_map(bad):
    n, lmax, maps = 40, 39, 3
    g = cw.cmbws_plan_grid(cw.CMBWS_GRID_GL, n, lmax)
    rng = np.random.default_rng(3)
    alm = rng.standard_normal((maps, (lmax + 1) ** 2))
    ref = to_dev(np.zeros((maps, g.npix)))
    cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(alm), ref, maps)
    alm[1, 5] = bad   # m = 0, l = 5
    out = to_dev(np.zeros((maps, g.npix)))
    cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(alm), out, maps)
    r, o = to_host(ref), to_host(out)
    assert not np.isfinite(o[1]).any()
    assert np.array_equal(o[[0, 2]], r[[0, 2]])
    f = rng.standard_normal((maps, g.npix))
    ra = to_dev(np.zeros((maps, (lmax + 1) ** 2)))
    cw.cmbws_sht_analysis(g, cw.CMBWS_FP64, to_dev(f), ra, maps, 1)
    f[2, 100] = bad
    oa = to_dev(np.zeros((maps, (lmax + 1) ** 2)))
    cw.cmbws_sht_analysis(g, cw.CMBWS_FP64, to_dev(f), oa, maps, 1)
    r, o = to_host(ra), to_host(oa)
    assert not np.isfinite(o[2]).any()
    assert np.array_equal(o[:2], r[:2])


# rings of 4..4 nside pixels: one to four thousand points, powers of two and Bluestein plans
@pytest.mark.parametrize("nside,lmax,maps", [(1, 3, 1), (2, 12, 2), (24, 71, 1), (96, 100, 1)])
def test_ring_lengths(nside, lmax, maps):
    g = cw.cmbws_plan_grid(cw.CMBWS_GRID_HEALPIX, nside, lmax)
    o = og.healpix(nside)
    rng = np.random.default_rng(nside)
    ell = np.concatenate([np.arange(lmax + 1)] + [np.arange(m, lmax + 1) for m in range(1, lmax + 1)
                                                  for _ in range(2)])
    # a steep spectrum: the ring spectra's first entries dominate the others
    alm = rng.standard_normal((maps, (lmax + 1) ** 2)) * (1.0 + ell) ** -3.0
    out = to_dev(np.zeros((maps, g.npix)))
    cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(alm), out, maps)
    f = rng.standard_normal((maps, g.npix))
    back = to_dev(np.zeros((maps, (lmax + 1) ** 2)))
    cw.cmbws_sht_analysis(g, cw.CMBWS_FP64, to_dev(f), back, maps, 1)
    m, a = to_host(out), to_host(back)
    for k in range(maps):
        assert rel_err(m[k], osht.synthesis(o, lmax, alm[k])) < _tol(lmax)
        assert rel_err(a[k], osht.adjoint(o, lmax, f[k], weighted=True)) < _tol(lmax)


def test_zero_input():
    g = cw.cmbws_plan_grid(cw.CMBWS_GRID_HEALPIX, 8, 23)
    out = to_dev(np.ones(g.npix))
    cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(np.zeros(24 ** 2)), out, 1)
    back = to_dev(np.ones(24 ** 2))
    cw.cmbws_sht_analysis(g, cw.CMBWS_FP64, to_dev(np.zeros(g.npix)), back, 1, 1)
    assert not to_host(out).any() and not to_host(back).any()


# the last three change the ring FFT's registers between one map and the batch (128 and 256 threads)
@pytest.mark.parametrize("n,lmax,maps", [(n, lmax, k) for n, lmax in ((66, 31), (130, 127), (259, 129))
                                         for k in (5, 6, 7, 8, 9)]
                         + [(512, 511, 3), (512, 511, 5), (600, 599, 5)])
def test_maps_of_a_batch_are_those_of_single_calls(n, lmax, maps):
    """Integer sums do not depend on how the maps are grouped: equal bit for bit."""
    g = cw.cmbws_plan_grid(cw.CMBWS_GRID_GL, n, lmax)
    rng = np.random.default_rng(n + 1000 * lmax + maps)
    alm = rng.standard_normal((maps, (lmax + 1) ** 2)) * 10.0 ** rng.uniform(-3, 3, (maps, 1))
    f = rng.standard_normal((maps, g.npix))
    out, back = to_dev(np.zeros((maps, g.npix))), to_dev(np.zeros_like(alm))
    cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(alm), out, maps)
    cw.cmbws_sht_analysis(g, cw.CMBWS_FP64, to_dev(f), back, maps, 0)
    m, a = to_host(out), to_host(back)
    for k in range(maps):
        one, bone = to_dev(np.zeros((1, g.npix))), to_dev(np.zeros((1, (lmax + 1) ** 2)))
        cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(alm[k:k + 1]), one, 1)
        cw.cmbws_sht_analysis(g, cw.CMBWS_FP64, to_dev(f[k:k + 1]), bone, 1, 0)
        assert np.array_equal(m[k], to_host(one)[0])
        assert np.array_equal(a[k], to_host(bone)[0])
