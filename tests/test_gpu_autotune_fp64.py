"""The tuner's records of the CMBWS_FP64 synthesis: one per kernel instance (1 to 4 maps each, 5 and 6,
7 and 8), each with tiles of its own."""
import numpy as np
import pytest

import paper_1710_00621_gb300 as cw
from paper_1710_00621_gb300.binding import FP64_TILES
from tests._gpu import to_dev, to_host

pytestmark = pytest.mark.gpu


def test_every_instance_is_measured_and_reported_by_itself():
    n, lmax = 128, 127
    rng = np.random.default_rng(5)
    alm = to_dev(rng.standard_normal((12, (lmax + 1) ** 2)))
    assert len(set(FP64_TILES)) == len(FP64_TILES)
    try:
        cw.cmbws_set_autotune(cw.CMBWS_TUNE_MEASURED)
        g = cw.cmbws_plan_grid(cw.CMBWS_GRID_GL, n, lmax)
        out = to_dev(np.zeros((12, g.npix)))
        known = lambda: {k for k in range(1, 13) if cw.cmbws_grid_tuning(g, cw.CMBWS_FP64, k)}
        for maps, want in ((4, {4}), (5, {4, 5, 6}), (12, {4, 5, 6, 7, 8, 9, 10, 11, 12})):
            cw.cmbws_sht_synth(g, cw.CMBWS_FP64, alm, out, maps)  # 12 maps run as 8 and 4
            assert known() == want
        got = to_host(out).copy()
        t = cw.cmbws_grid_tuning(g, cw.CMBWS_FP64, 8)
        assert t["tile"] == FP64_TILES[t["variant"]] and len(t["ms"]) == len(FP64_TILES)
        cw.cmbws_set_autotune(cw.CMBWS_TUNE_DEFAULT)
        cw.cmbws_sht_synth(g, cw.CMBWS_FP64, alm, out, 12)
        assert np.array_equal(to_host(out), got)
    finally:
        cw.cmbws_set_autotune(cw.CMBWS_TUNE_DEFAULT)
